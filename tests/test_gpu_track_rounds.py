"""Track encoder and decoder against the oracle, byte for byte, for track
lengths around their rounds of 16 clusters and for every alignment of the
input arrays (the staging copies 16-byte windows)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import synth

import gpu_helpers as G
from test_gpu_unatt_encode import dec  # noqa: F401

pytestmark = pytest.mark.gpu

LENGTHS = [1, 2, 15, 16, 17, 31, 32, 33, 48, 64, 65, 152]
FIELDS = (("qpt", np.uint8), ("row", np.uint8), ("slice", np.uint8), ("pad", np.uint16),
          ("time", np.uint32), ("ncl", np.uint16), ("row_diff", np.uint8),
          ("slice_leg_diff", np.uint8), ("pad_res", np.uint16), ("time_res", np.uint32))


def _truth(seed):
    """Tracks cut to the lengths above (shorter ones as they are)."""
    u = synth.make_truth(n_tracks=500, n_unatt=0, seed=seed, looper_frac=0.3, max_legs=4)
    ncl = u["ncl"].astype(np.int64)
    cut = np.minimum(ncl, np.array(LENGTHS)[np.arange(len(ncl)) % len(LENGTHS)])
    place = np.arange(ncl.sum()) - np.repeat(np.cumsum(ncl) - ncl, ncl)
    keep = place < np.repeat(cut, ncl)
    for k, _, kind in O.TRUTH_FIELDS:
        if kind == "att":
            u[k] = u[k][keep]
    u["ncl"] = cut.astype(np.uint16)
    return u


def _shift(d, offset):
    """The arrays at `offset` elements past an aligned address."""
    import torch
    out = {}
    for k, v in d.items():
        buf = torch.empty(v.numel() + 16, dtype=v.dtype, device=v.device)
        out[k] = buf[offset:offset + v.numel()].copy_(v)
    return out


@pytest.mark.parametrize("offset", [0, 1, 2, 3, 7, 15])
def test_rounds(dec, offset):  # noqa: F811
    import torch
    from paper_2411_02206_gb300 import frames
    u = _truth(50 + offset)
    dev = frames.to_torch(u, "cuda:0")
    attached = [k for k, _, kind in O.TRUTH_FIELDS if kind in ("track", "att")]
    enc = dec.encode(_shift({k: dev[k] for k in attached}, offset))
    torch.cuda.synchronize()
    of = G.oracle_frame(u)
    assert int(enc["status"].item()) == 0
    for k, dt in FIELDS:
        assert np.array_equal(frames.to_numpy(enc[k], dt), of[k]), f"encoder field {k} differs"
    frame = frames.assemble(dev, enc)
    residuals = ("row_diff", "slice_leg_diff", "pad_res", "time_res")
    frame.update(_shift({k: frame[k] for k in residuals}, offset))
    ora = O.decode(of)
    for variant in (0, 1):
        dec.tmd_tune_set("decode_variant", variant)
        native, row_start, att, status = dec.decode(frame)
        torch.cuda.synchronize()
        G.assert_same_decode((native.cpu().numpy(), frames.to_numpy(row_start, np.uint32),
                              frames.to_numpy(att, np.uint32), int(status.item())), ora,
                             f"variant {variant}")
    dec.tmd_tune_set("decode_variant", 0)
