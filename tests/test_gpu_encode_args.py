"""tmd_encode_tracks refuses arrays that are not aligned to their element size
before anything is launched on them."""
import numpy as np
import pytest

from paper_2411_02206_gb300 import synth
from test_gpu_unatt_encode import dec  # noqa: F401

pytestmark = pytest.mark.gpu

TRUTH = {"ncl": 2, "pad": 2, "time": 4}
OUT = {"pad": 2, "time": 4, "ncl": 2, "pad_res": 2, "time_res": 4, "status": 4}


def _call(dec, truth, shift=None, by=1):  # noqa: F811
    """Encodes with one pointer shifted by some bytes; every array has room
    for a shift, and the outputs are returned."""
    import torch
    from paper_2411_02206_gb300 import frames, tmd
    dev = frames.to_torch(truth, "cuda:0")
    room = {k: torch.cat([v.view(torch.uint8), v.new_zeros(16).view(torch.uint8)])
            for k, v in dev.items() if k in tmd.TRUTH_FIELDS}
    nt, na = len(truth["ncl"]), len(truth["row"])
    out = {k: torch.full((4 * na + 16,), 0xAB, dtype=torch.uint8, device="cuda:0")
           for k in tmd.TRACK_OUT_FIELDS}
    pin = [room[k].data_ptr() + by * (shift == ("in", k)) for k in tmd.TRUTH_FIELDS]
    pout = [out[k].data_ptr() + by * (shift == ("out", k)) for k in tmd.TRACK_OUT_FIELDS]
    try:
        dec.tmd_encode_tracks(tmd.tmd_truth_in(nt, na, *pin), tmd.tmd_track_out(*pout))
        torch.cuda.synchronize()
    except tmd.TmdError as e:
        assert e.code == tmd.TMD_ERR_ARG
        torch.cuda.synchronize()
        assert all(bool((v == 0xAB).all()) for v in out.values()), "outputs were touched"
        return None
    return out


@pytest.mark.parametrize("shift, by", [((w, k), b) for w, ks in (("in", TRUTH), ("out", OUT))
                                       for k, size in ks.items() for b in {1, size // 2}])
def test_misaligned_arrays_are_refused(dec, shift, by):  # noqa: F811
    truth = synth.make_truth(n_tracks=50, n_unatt=0, seed=3)
    assert _call(dec, truth, shift, by) is None


def test_empty_and_aligned_arrays_are_accepted(dec):  # noqa: F811
    """Tracks of one cluster each have no residuals: their pointers may be any."""
    truth = synth.make_truth(n_tracks=50, n_unatt=0, seed=3)
    first = np.cumsum(truth["ncl"].astype(np.int64)) - truth["ncl"]
    for k in ("row", "sector", "leg", "pad", "time"):
        truth[k] = truth[k][first]
    truth["ncl"] = np.ones(50, np.uint16)
    for shift in (None, ("out", "pad_res"), ("out", "time_res")):
        out = _call(dec, truth, shift)
        assert out is not None
        assert int(out["status"][0]) == 0
        assert bytes(out["pad"][:100].cpu().numpy()) == truth["pad"].tobytes()
