"""The sorting paths of the GPU unattached encoder against the oracle encoder,
byte for byte, at the sizes where one path hands over to the next: bins of a
warp, of a block, of several time slices, and the general sort (bins too large
for a block, crowded times, times of 2^24 and more)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import synth
from test_gpu_unatt_encode import UNATT_OUT, _oracle, dec  # noqa: F401

pytestmark = pytest.mark.gpu

MIXED = [1, 2, 31, 32, 33, 127, 128, 129, 511, 513, 1000, 4095, 4096, 4097, 12288, 12289, 16384,
         40000]


def _truth(counts, seed, hi=None, shift=None):
    """Clusters of bins 300 k + 7 with the given counts, in random order."""
    rng = np.random.default_rng(seed)
    binid = np.repeat(300 * np.arange(len(counts)) + 7, counts)
    rng.shuffle(binid)
    n = len(binid)
    u = synth.make_unattached_truth(rng, n)
    u["row_u"] = (binid % synth.NROW).astype(np.uint8)
    u["sector_u"] = (binid // synth.NROW).astype(np.uint8)
    u["pad_u"] = rng.integers(0, 8000, n).astype(np.uint16)
    if hi:
        u["time_u"] = rng.integers(0, hi, n).astype(np.uint32)
    if shift:
        u["time_u"][: n // 2] += np.uint32(shift)
    dup = rng.integers(0, n, n // 50)  # exact repeats: ties in input order
    for k in ("row_u", "sector_u", "pad_u", "time_u"):
        u[k][dup] = u[k][np.roll(dup, 1)]
    return u


@pytest.mark.parametrize("what, counts, kw", [
    ("mixed", MIXED, {}),
    ("few times", MIXED, dict(hi=40)),              # buckets of equal times, then crowded bins
    ("one time", [100, 3000, 20000], dict(hi=1)),
    ("two groups of times", [120, 4000, 9000, 30000], dict(hi=500, shift=1 << 23)),
    ("wide times", [5, 200, 5000, 20000], dict(shift=1 << 25)),
    ("one bin beyond a block", [(1 << 18) + 5, 70, 3], {}),
])
@pytest.mark.parametrize("offset", [0, 1])
def test_paths(dec, what, counts, kw, offset):  # noqa: F811
    import torch
    from paper_2411_02206_gb300 import frames
    u = _truth(counts, len(what), **kw)
    dev = {}
    for k, v in frames.to_torch(u, "cuda:0").items():  # offset 1: arrays aligned to one element
        buf = torch.empty(v.numel() + 1, dtype=v.dtype, device=v.device)
        dev[k] = buf[offset:offset + v.numel()].copy_(v)
    for _ in range(2):  # the second call finds the first one's scratch
        out = dec.encode_unattached(dev)
    torch.cuda.synchronize()
    assert int(out["status"].item()) == 0
    ref = _oracle(u)
    for k, dt in UNATT_OUT:
        assert np.array_equal(frames.to_numpy(out[k], dt), ref[k]), f"{what}: {k} differs"
