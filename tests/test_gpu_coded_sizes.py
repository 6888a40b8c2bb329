"""Coded frames at the chunk counts where the entropy decoder's blocks change
size (32 and 56 chunks per SM) and where the later streams stop starting at
once (24 chunks per SM)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import frames, synth

import gpu_helpers as G
from test_gpu_rans import CHUNK, _same_streams, _upload, dec  # noqa: F401

pytestmark = pytest.mark.gpu

TRACKS = 300


def _chunks(f: dict) -> int:
    return sum(max(1, -(-len(f[name]) // CHUNK)) for name, _, _ in O.FRAME_FIELDS)


@pytest.mark.parametrize("per_sm", [24, 32, 56])
@pytest.mark.parametrize("over", [0, 1])
def test_block_and_start_rules(dec, per_sm, over):  # noqa: F811
    """The largest frame within the limit, and the next chunk of each
    unattached stream."""
    import torch
    from paper_2411_02206_gb300 import tmd
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    kinds = [kind for _, _, kind in O.FRAME_FIELDS]
    small = G.oracle_frame(synth.make_truth(n_tracks=TRACKS, n_unatt=1, seed=31))
    others = _chunks(small) - kinds.count("unatt")
    whole = (per_sm * sms - others) // kinds.count("unatt") + over
    f = G.oracle_frame(synth.make_truth(n_tracks=TRACKS, n_unatt=whole * CHUNK - 5, seed=31))
    assert (_chunks(f) > per_sm * sms) == bool(over)
    coded = _upload(tmd.rans_encode(f))
    counts = O.frame_counts(f)
    got, status = dec.rans_decode(coded, *counts)
    assert int(status.item()) == 0
    _same_streams(got, f, f"{_chunks(f)} chunks")
    a = dec.decode_coded(coded, *counts)
    torch.cuda.synchronize()
    native, rs, att, st = a
    G.assert_same_decode((native.cpu().numpy(), frames.to_numpy(rs, np.uint32),
                          frames.to_numpy(att, np.uint32), int(st.item())),
                         O.decode(f), f"{_chunks(f)} chunks")
