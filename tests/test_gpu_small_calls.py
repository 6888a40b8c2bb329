"""Decoding at the sizes where the kernels of small calls hand over to the
general ones: 16384 tracks (track preparation), one group of 32 ranking tiles
(group sums)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import synth

import gpu_helpers as G
from test_gpu_unatt_encode import dec  # noqa: F401

pytestmark = pytest.mark.gpu

CLUSTERS = 80  # per track: 13107 tracks fill 32 tiles of 32768 clusters (but for 16)


def _truth(n_tracks):
    """n_tracks tracks of 80 clusters, repeated from a sample of longer ones."""
    u = synth.make_truth(n_tracks=900, n_unatt=30_000, seed=77, max_legs=3)
    ncl = u["ncl"].astype(np.int64)
    start = np.cumsum(ncl) - ncl
    pick = np.nonzero(ncl >= CLUSTERS)[0]
    pick = pick[np.arange(n_tracks) % len(pick)]
    place = (start[pick][:, None] + np.arange(CLUSTERS)).ravel()
    for k, _, kind in O.TRUTH_FIELDS:
        if kind == "att":
            u[k] = u[k][place]
        elif kind == "track":
            u[k] = u[k][pick]
    u["ncl"] = np.full(n_tracks, CLUSTERS, np.uint16)
    return u


@pytest.mark.parametrize("n_tracks", [1023, 1025, 13107, 13108, 16384, 16385])
def test_hand_over(dec, n_tracks):  # noqa: F811
    u = _truth(n_tracks)
    enc, _, gpu = G.gpu_encode_decode(dec, u)
    of = G.oracle_frame(u)
    assert enc["status"] == 0
    for k in ("pad_res", "time_res", "row_diff", "slice_leg_diff"):
        assert np.array_equal(enc[k], of[k]), f"encoder field {k} differs"
    G.assert_same_decode(gpu, O.decode(of), f"{n_tracks} tracks")


@pytest.mark.parametrize("bad", ["zero length", "one cluster more", "unattached count"])
def test_wrong_counts_set_the_status(dec, bad):  # noqa: F811
    u = _truth(1025)
    f = G.oracle_frame(u)
    if bad == "zero length":
        f["ncl"][5] = 0
    elif bad == "one cluster more":
        f["ncl"][5] += 1
    else:
        f["n_unatt"][100] += 1
    assert G.gpu_decode_np(dec, f)[3] & O.ST_COUNT
