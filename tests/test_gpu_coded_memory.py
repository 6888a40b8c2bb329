"""The coded host pipeline's second set of streams never costs a call its
memory: where the device has room for one set and the decoding scratch, the
frames are decoded; and the set makes way for other allocations."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_02206_gb300 import frames, synth

import gpu_helpers as G
from test_gpu_rans import dec  # noqa: F401

pytestmark = pytest.mark.gpu

MIB = 1 << 20


class _Case:
    """A frame with its coded form, the bytes that a handle takes for each part
    of its decoding (measured on a handle of its own, which also loads every
    kernel), and a filler for the rest of the device."""

    def __init__(self, n_tracks=24_000, n_unatt=600_000):
        import torch
        from paper_2411_02206_gb300 import tmd
        self.torch, self.tmd = torch, tmd
        u = synth.make_truth(n_tracks=1500, n_unatt=n_unatt, seed=5)
        rep = n_tracks // 1500
        for k, _, kind in O.TRUTH_FIELDS:
            if kind in ("att", "track"):
                u[k] = np.tile(u[k], rep)
        self.host = G.oracle_frame(u)
        self.dev = frames.to_torch(self.host, "cuda:0")
        self.counts = O.frame_counts(self.host)
        self.ref = O.decode(self.host)
        self.blob = torch.from_numpy(tmd.rans_encode(self.host).copy()).pin_memory()
        self.coded = torch.from_numpy(self.blob.numpy()).to("cuda:0")
        n = self.counts[1] + self.counts[2]
        self.out = [[torch.zeros(s, dtype=d, device=w) for s, d in
                     (((n, 12), torch.uint8), (5473, torch.int32), (5472, torch.int32),
                      (1, torch.int32))] for w in ("cuda:0", "cpu", "cpu", "cpu")]
        self.fill = None
        h = tmd.Decoder(0)
        at = [self.free()]
        self.decode(h)
        at.append(self.free())
        h.tmd_decode_coded_frame(self.coded, self.coded.numel(), *self.counts,
                                 tmd.frame_out(*self.out[0]))
        at.append(self.free())
        self.stream(h, 1)
        at.append(self.free())
        h.close()
        self.scratch, self.set, self.slot = (a - b for a, b in zip(at, at[1:]))
        assert min(self.scratch, self.set, self.slot) >= 20 * MIB  # cudaMalloc rounds to 2 MiB

    def free(self):
        self.torch.cuda.synchronize()
        return self.torch.cuda.mem_get_info()[0]

    def leave(self, n_bytes):
        """Occupies the device's memory but for n_bytes."""
        self.torch.cuda.empty_cache()
        self.fill = self.torch.empty(self.free() - n_bytes, dtype=self.torch.uint8, device="cuda:0")

    def decode(self, h):
        h.tmd_decode_frame(self.tmd.frame_in(self.dev), self.tmd.frame_out(*self.out[0]))
        self.torch.cuda.synchronize()

    def stream(self, h, n):
        c = self.tmd.tmd_coded_frame(self.blob.data_ptr(), self.blob.numel(), *self.counts)
        h.tmd_decode_coded_host_stream([c] * n, [self.tmd.frame_out(*o) for o in self.out[1:n + 1]])

    def check(self, o, what):
        G.assert_same_decode((o[0].cpu().numpy(), frames.to_numpy(o[1], np.uint32),
                              frames.to_numpy(o[2], np.uint32), int(o[3].item())), self.ref, what)

    def close(self):
        self.fill = None
        self.torch.cuda.empty_cache()


@pytest.fixture(scope="module")
def case(dec):  # noqa: F811
    c = _Case()
    yield c
    c.close()


@pytest.mark.parametrize("spare", ["half the scratch", "half a set"])
def test_frames_decode_without_room_for_the_second_set(case, spare):
    """Room for the slots, one set and the scratch, but not for two sets: two
    sets fit before the scratch is asked for, or not even they."""
    from paper_2411_02206_gb300 import tmd
    h = tmd.Decoder(0)
    try:
        case.leave(2 * case.slot + (2 * case.set + case.scratch // 2 if spare == "half the scratch"
                                    else case.set + case.scratch + case.set // 2))
        for turn in range(2):
            for o in case.out[1:]:
                for t in o:
                    t.fill_(7)
            case.stream(h, 2)
            assert h._L.tmd_last_error_string(h.h) == b""
            for i in (1, 2):
                case.check(case.out[i], f"{spare}, call {turn}, frame {i}")
    finally:
        h.close()
        case.close()


def test_second_set_makes_way(case):
    """After a pipelined call, an allocation that fits only in the second set's
    place is made, and the next pipelined call still works."""
    from paper_2411_02206_gb300 import tmd
    h = tmd.Decoder(0)
    try:
        case.stream(h, 3)
        # a batch's own scratch, about as large as the handle's
        case.leave(case.scratch // 2)
        b = h.tmd_batch_create([tmd.frame_in(case.dev)], [tmd.frame_out(*case.out[0])])
        h.tmd_batch_launch(b)
        case.torch.cuda.synchronize()
        case.check(case.out[0], "batch")
        case.stream(h, 3)
        for i in (1, 2, 3):
            case.check(case.out[i], f"frame {i}")
        h.tmd_batch_destroy(b)
    finally:
        h.close()
        case.close()
