"""The unattached encoder on uneven frames: few large bins, crowded and equal
times, times of 2^24 and more.  Byte for byte against the oracle at the sizes
where its sorts hand over, and without the times that one block per bin and the
sort of everything left over once took."""
import statistics

import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import synth
from test_gpu_unatt_encode import UNATT_OUT, _oracle, dec  # noqa: F401

pytestmark = pytest.mark.gpu

SLICE, BLOCK, BIG = 12288, 4096, 1 << 18  # clusters: per time slice, largest block bin, largest sliced


def _truth(counts, seed, times=128_000, pads=8000, spread=None):
    """Clusters of bins 97 k + 11 with the given counts, in random order; times
    below `times`, or `spread` (values) at random."""
    rng = np.random.default_rng(seed)
    binid = np.repeat(97 * np.arange(len(counts)) + 11, counts)
    rng.shuffle(binid)
    n = len(binid)
    u = synth.make_unattached_truth(rng, n)
    u["row_u"] = (binid % synth.NROW).astype(np.uint8)
    u["sector_u"] = (binid // synth.NROW).astype(np.uint8)
    u["pad_u"] = rng.integers(0, pads, n).astype(np.uint16)
    u["time_u"] = (rng.choice(np.asarray(spread, np.uint32), n) if spread
                   else rng.integers(0, times, n).astype(np.uint32))
    return u


def _check(dec, u, what):  # noqa: F811
    import torch
    from paper_2411_02206_gb300 import frames
    dev = frames.to_torch(u, "cuda:0")
    for _ in range(2):  # the second call finds the first one's scratch
        out = dec.encode_unattached(dev)
    torch.cuda.synchronize()
    assert int(out["status"].item()) == 0
    ref = _oracle(u)
    for k, dt in UNATT_OUT:
        assert np.array_equal(frames.to_numpy(out[k], dt), ref[k]), f"{what}: {k} differs"


TOP = 0xFFFFFF


@pytest.mark.parametrize("what, counts, kw", [
    # a block's bins, sorted as a whole: full, one more than a power of two, small
    ("one time", [129, 513, 1025, 4095, 4096], dict(times=1)),
    ("one cluster over and over", [129, 2048, 2049, 4095, 4096], dict(times=1, pads=1)),
    ("first and last time", [200, 3000, 4096, 9000], dict(spread=[0, TOP])),
    ("crowd beside lone times", [1000, 4096, 30000], dict(spread=[5] * 99 + list(range(100, 4000)))),
    # slices: none before, some before, empty ones between, one full, one too full
    ("slices", [BLOCK + 1, SLICE, SLICE + 1, 3 * SLICE, 5 * SLICE + 1, 100_000], {}),
    ("few times", [SLICE + 1, 40_000, 120_000], dict(times=64)),
    ("empty slices", [60_000, 130_000], dict(spread=list(range(700)) + [TOP - 1, TOP])),
    ("slice of one time", [16384, 4097, 50], dict(times=1, pads=250)),
    ("more than a slice of one time", [16385, 4097, 50, 60_000], dict(times=1, pads=250)),
    ("largest sliced bin and larger", [BIG, BIG + 1, 10], {}),
    # the general sort: some bins of many, all of them, a single one, nothing to sort by
    ("two of many", [BIG + 7, 20_000] + [37] * 40, dict(spread=[9] * 20 + [10])),
    ("all general", [BIG + 1, BIG + 2049], {}),
    ("one bin, one cluster", [BIG + 1], dict(times=1, pads=1)),
    ("every time bit", [300, 5000, 1], dict(spread=[0, 1, 1 << 24, 1 << 31, 0xFFFFFFFF])),
    ("latest time only", [300, 5000, 1], dict(spread=[0xFFFFFFFF])),
    ("one wide cluster", [1], dict(spread=[0xFFFFFFFE], pads=1)),
])
def test_skewed_frames(dec, what, counts, kw):  # noqa: F811
    _check(dec, _truth(counts, len(what), **kw), what)


def _time(dec, u):  # noqa: F811
    """Median device time of a call, ms."""
    import torch
    from paper_2411_02206_gb300 import frames
    dev = frames.to_torch(u, "cuda:0")
    ms = []
    for i in range(25):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        dec.encode_unattached(dev)
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return statistics.median(ms[5:])


@pytest.mark.parametrize("what, n, same, limit", [
    # the radix sort over all clusters that came before these paths took 3.1 and
    # 2.4 times the even frame's time now; one block per bin and the general sort
    # of crowded bins took 20 and 3.8 times
    ("one bin", 200_000, ("row_u", "sector_u"), 4.0),
    ("one time and pad", 2_000_000, ("time_u", "pad_u"), 3.0),
])
def test_skewed_frames_keep_their_time(dec, what, n, same, limit):  # noqa: F811
    rng = np.random.default_rng(5)
    even = synth.make_unattached_truth(rng, n)
    skewed = {k: np.full_like(v, 7) if k in same else v for k, v in even.items()}
    t, flat = _time(dec, skewed), _time(dec, even)
    assert t <= limit * flat, f"{what}: {t:.3f} ms against {flat:.3f} ms"
