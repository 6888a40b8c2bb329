"""Paths that only larger calls take: both staging variants of the track decoder
at every number of tracks per warp, and the allocation-free decode of a frame
of more than one group of ranking tiles."""
import numpy as np
import pytest

from oracle import oracle as O

import gpu_helpers as G
from test_gpu_small_calls import CLUSTERS, _truth
from test_gpu_unatt_encode import dec  # noqa: F401

pytestmark = pytest.mark.gpu

TILE, GROUP = 32768, 32  # attached clusters per ranking tile, tiles per group


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("variant", [0, 1])
def test_decoder_variants_at_all_lanes(dec, lanes, variant):  # noqa: F811
    """The largest call of `lanes` tracks per warp (12 warps per SM), and for 32
    the first one."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_tracks = lanes * 12 * sms if lanes < 32 else 16 * 12 * sms + 1
    of = G.oracle_frame(_truth(n_tracks))
    assert len(of["ncl"]) == n_tracks
    old = dec.tmd_tune_get("decode_variant")
    dec.tmd_tune_set("decode_variant", variant)
    try:
        G.assert_same_decode(G.gpu_decode_np(dec, of), O.decode(of),
                             f"variant {variant}, {lanes} lanes")
    finally:
        dec.tmd_tune_set("decode_variant", old)


@pytest.mark.parametrize("tiles", [GROUP, GROUP + 1, 2 * GROUP + 1])
def test_noalloc_over_groups_of_tiles(tiles):
    import torch
    from paper_2411_02206_gb300 import build, frames, tmd
    build.build()
    n_tracks = (tiles - 1) * TILE // CLUSTERS + 1
    of = G.oracle_frame(_truth(n_tracks))
    assert -(-O.frame_counts(of)[1] // TILE) == tiles
    dev = frames.to_torch(of, "cuda:0")
    n = sum(O.frame_counts(of)[1:])
    out = (torch.full((n, 12), 0xAB, dtype=torch.uint8, device="cuda:0"),
           *(torch.full((k,), -1, dtype=torch.int32, device="cuda:0") for k in (5473, 5472, 1)))
    rc, msg = tmd.tmd_decode_frame_noalloc(tmd.frame_in(dev), tmd.frame_out(*out))
    torch.cuda.synchronize()
    assert rc == tmd.TMD_OK, msg
    G.assert_same_decode((out[0].cpu().numpy(), frames.to_numpy(out[1], np.uint32),
                          frames.to_numpy(out[2], np.uint32), int(out[3].item())),
                         O.decode(of), f"{tiles} tiles")
