"""Timed cases of the track-model decoder: what a user of the library has it do.

Each case is one call through the public binding (paper_2411_02206_gb300.tmd),
on synthetic frames of the library's own input recipe (synth.py: helices from
the origin in B = 0.5 T crossing the pad rows, unattached clusters uniform or
in hot bins, log-normal charges), generated on the GPU so that a frame of
57 M clusters takes well under a second.

Kinds:
  decode        Decoder.decode: one device-resident compressed frame
  batch         Decoder.tmd_batch_launch: a planned batch of frames, one graph launch
  coded         Decoder.decode_coded: entropy decoding, then track-model decoding
  coded_host    Decoder.tmd_decode_coded_host_stream: coded frames in pinned host memory,
                results back in pinned host memory
  encode_tracks Decoder.encode: track-model encoding of attached clusters
  encode_unatt  Decoder.encode_unattached: sorting and differencing of unattached clusters
  xyz           Decoder.global_xyz: positions of a decoded cluster list
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_02206_gb300 import frames, synth, tmd

NBIN, NROW = synth.NBIN, synth.NROW
DEV = "cuda:0"

# Track mixes (arguments of synth.make_truth) and the mean clusters per track
# that they give; "small", "pbpb" and "stress" are synth.SHAPES, "pp" is the
# pp-like end of synth.batch_specs (few, mostly primary tracks).
MIXES = {
    "small": dict(looper=0.17, secondary=0.65, pt_mean=0.5, legs=3, per_track=104.0),
    "pbpb": dict(looper=0.17, secondary=0.85, pt_mean=0.5, legs=3, per_track=94.4),
    "pp": dict(looper=0.05, secondary=0.60, pt_mean=0.5, legs=3, per_track=103.2),
    "stress": dict(looper=0.30, secondary=0.65, pt_mean=0.2, legs=6, per_track=107.7),
}
# unattached clusters of the stress shape: 40 % of the bins empty, 90 % of the
# clusters in 10 % of the bins
HOT = dict(empty=0.4, frac=0.1, share=0.9)


def listed():
    return [
        # the smallest frames of the repository's workloads (2 k tracks + 100 k
        # unattached clusters): a call of launches and latencies
        dict(name="decode_small", kind="decode", mix="small", n_tracks=2000, n_unatt=100_000),
        # a pp-like frame, mostly unattached clusters, ragged counts
        dict(name="decode_pp", kind="decode", mix="pp", n_tracks=11_111, n_unatt=2_500_003),
        # the full Pb-Pb-shaped frame, the headline workload
        dict(name="decode_pbpb", kind="decode", mix="pbpb", n_tracks=400_000,
             n_unatt=20_000_000),
        # low-pT loopers of up to 6 legs and unattached clusters in hot bins:
        # the stress shape at 0.4 of its size
        dict(name="decode_stress", kind="decode", mix="stress", n_tracks=400_000,
             n_unatt=24_000_000),
        # frames of very different sizes and mixes decoded together, as the
        # batched and the serving workloads do
        dict(name="batch_mixed", kind="batch", n_frames=16, lo=100_000, hi=4_000_000, spec_seed=7),
        # entropy-coded frames: a small one and a quarter of the Pb-Pb frame
        dict(name="coded_small", kind="coded", mix="small", n_tracks=2000, n_unatt=100_000),
        dict(name="coded_pbpb", kind="coded", mix="pbpb", n_tracks=100_000, n_unatt=5_000_000),
        # coded frames arriving in host memory, results wanted there
        dict(name="coded_host", kind="coded_host", mix="pbpb", n_tracks=15_000, n_unatt=750_000,
             n_frames=4),
        # the encoding side: the tracks and the unattached clusters of a
        # Pb-Pb-shaped frame, and the unattached clusters of a small frame
        dict(name="encode_tracks", kind="encode_tracks", mix="pbpb", n_tracks=200_003),
        dict(name="encode_unatt", kind="encode_unatt", n_unatt=20_000_000, hot=False),
        dict(name="encode_unatt_small", kind="encode_unatt", n_unatt=100_003, hot=False),
        # global positions of a Pb-Pb-shaped cluster list, the step after decoding
        dict(name="xyz_pbpb", kind="xyz", n=57_800_001),
    ]


def n_attached(n_tracks, mix):
    """Attached clusters of a frame: 96 % of the mix's mean, so that a sample
    of tracks has at least as many."""
    return int(n_tracks * MIXES[mix]["per_track"] * 0.96)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "batch", "coded", "coded", "coded_host",
                       "encode_tracks", "encode_unatt", "encode_unatt", "xyz"])
    mix = rng.choice(sorted(MIXES))
    if kind in ("decode", "coded"):
        # total clusters from 2e4 up, of which 25 to 70 % attached (the
        # repository's range from pp-like to central Pb-Pb)
        total = _log(rng, 20_000, 50_000_000 if kind == "decode" else 10_000_000)
        att = rng.uniform(0.25, 0.70)
        return dict(kind=kind, mix=mix,
                    n_tracks=max(1, int(total * att / MIXES[mix]["per_track"])),
                    n_unatt=int(total * (1 - att)))
    if kind == "batch":
        return dict(kind=kind, n_frames=rng.randint(2, 16), lo=_log(rng, 20_000, 200_000),
                    hi=_log(rng, 300_000, 4_000_000), spec_seed=rng.randint(0, 10 ** 6))
    if kind == "coded_host":
        return dict(kind=kind, mix=mix, n_tracks=_log(rng, 200, 15_000),
                    n_unatt=_log(rng, 10_000, 750_000), n_frames=rng.randint(1, 5))
    if kind == "encode_tracks":
        return dict(kind=kind, mix=mix, n_tracks=_log(rng, 100, 200_000))
    if kind == "encode_unatt":
        return dict(kind=kind, n_unatt=_log(rng, 1_000, 20_000_000), hot=rng.random() < 0.4)
    return dict(kind=kind, n=_log(rng, 10_000, 57_000_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rand(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _crossings(g, m, mix):
    """Pad-row crossings of m helices, axes (track, leg, row along the path):
    mask of the clusters kept, and row, sector, leg, y, t, q/pT code."""
    mx = MIXES[mix]
    legs = mx["legs"]
    loop = _rand(g, m) < mx["looper"]
    pt = torch.where(loop, _rand(g, m, 0.1, 0.17),
                     0.18 - mx["pt_mean"] * torch.log1p(-_rand(g, m)))
    q = torch.where(_rand(g, m) < 0.5, 1.0, -1.0).double()
    phi0, sinh_eta = _rand(g, m, 0.0, 2 * math.pi), torch.sinh(_rand(g, m, -0.9, 0.9))
    t0 = _rand(g, m, 0.0, 3000.0)
    second = (_rand(g, m) < mx["secondary"]) & ~loop
    r_first = torch.where(second, (_rand(g, m) * 130).long(), 0)
    xrow = torch.as_tensor(synth.XROW, device=DEV)
    radius = pt / synth.B_CM
    sig = -q
    cx, cy = -sig * radius * torch.sin(phi0), sig * radius * torch.cos(phi0)
    a0 = torch.atan2(-cy, -cx)
    nleg = torch.where(2.0 * radius < xrow[-1] / math.cos(math.radians(10.0)), legs, 1)

    def ax(v):  # a per-track value along the (leg, row) axes
        return v[:, None, None]

    up = torch.arange(NROW, device=DEV)
    leg = torch.arange(legs, device=DEV)[None, :, None]
    row = torch.where(leg % 2 == 0, up[None, None, :], NROW - 1 - up[None, None, :])
    rho, R = xrow[row], ax(radius)
    ok = (leg < ax(nleg)) & (rho < 2.0 * R) & ((leg > 0) | (row >= ax(r_first)))
    ok &= torch.rand(ok.shape, generator=g, device=DEV) >= 0.1
    beta = torch.arccos((1.0 - rho * rho / (2.0 * R * R)).clamp(-1.0, 1.0))
    beta = torch.where(leg % 2 == 1, 2 * math.pi - beta, beta)
    z = R * (beta + (leg // 2) * (2 * math.pi)) * ax(sinh_eta)
    ok &= z.abs() < synth.ZMAX - 1.0
    th = ax(a0) + ax(sig) * beta
    px, py = ax(cx) + R * torch.cos(th), ax(cy) + R * torch.sin(th)
    sec0 = (torch.remainder(torch.atan2(py, px), 2 * math.pi) / synth.SEC_RAD).long().clamp(max=17)
    y, sector = torch.full_like(px, math.nan), sec0.clone()
    for d in (0, 1, -1):  # the sector of the crossing, else its neighbours
        sc = torch.remainder(sec0 + d, 18)
        psi = sc * synth.SEC_RAD + synth.SEC_RAD / 2
        u0, u1 = torch.cos(psi), torch.sin(psi)
        ccx, ccy = ax(cx) * u0 + ax(cy) * u1, -ax(cx) * u1 + ax(cy) * u0
        disc = R * R - (rho - ccx) ** 2
        root, ref = torch.sqrt(disc.clamp(min=0.0)), -px * u1 + py * u0
        yy = torch.where((ccy + root - ref).abs() < (ccy - root - ref).abs(), ccy + root, ccy - root)
        good = torch.isnan(y) & (disc >= 0) & (yy.abs() < rho * synth.TAN10)
        y, sector = torch.where(good, yy, y), torch.where(good, sc, sector)
    ok &= ~torch.isnan(y)
    ok &= torch.cumsum(ok.reshape(m, -1), 1).reshape(ok.shape) <= 152
    y = y + 0.1 * torch.randn(y.shape, generator=g, device=DEV)
    z = z + 0.1 * torch.randn(z.shape, generator=g, device=DEV)
    sector = sector + 18 * (z < 0)
    t = ax(t0) + (synth.ZMAX - z.abs()) / 0.5
    code = (q / pt / 0.078125 + 127.5).round().clamp(0, 255)
    return ok, row.expand_as(ok), sector, leg.expand_as(ok), y, t, code


def _charges(g, n):
    def byte():
        return torch.randint(0, 256, (n,), generator=g, device=DEV, dtype=torch.uint8)
    qtot = torch.exp(5.0 + 0.6 * torch.randn(n, generator=g, device=DEV)).round().clamp(1, 65535)
    qtot = qtot.to(torch.int32)
    wob = torch.randint(-3, 4, (n,), generator=g, device=DEV, dtype=torch.int32)
    qmax = ((qtot >> 2) + wob).clamp(min=1)
    flags = (torch.rand(n, generator=g, device=DEV) < 0.01).to(torch.uint8)
    return qtot.to(torch.int16), qmax.to(torch.int16), flags, byte(), byte()


def _tracks(g, n_tracks, mix):
    """Attached-cluster truth (the track encoder's input) with its charges."""
    npads = torch.as_tensor(synth.NPADS, device=DEV)
    wpad = torch.as_tensor(synth.WPAD, device=DEV)
    att = n_attached(n_tracks, mix)
    parts, have = {k: [] for k in ("qpt", "ncl", "row", "sector", "leg", "pad", "time")}, 0
    while have < n_tracks:
        want = n_tracks - have  # tracks of fewer than 20 clusters are drawn again
        ok, row, sector, leg, y, t, code = _crossings(g, min(24_000, want + want // 3 + 64), mix)
        n = ok.sum((1, 2))
        good = torch.nonzero(n >= 20).flatten()[:want]
        ok, n, code = ok[good], n[good], code[good]
        row, sector, leg = row[good][ok], sector[good][ok], leg[good][ok]
        y, t = y[good][ok], t[good][ok]
        pad = ((y / wpad[row] + npads[row] / 2.0) * 64.0).round()
        pad = torch.minimum(pad.clamp(min=0), (npads[row] * 64 - 1).double())
        parts["qpt"].append(code.to(torch.uint8))
        parts["ncl"].append(n.to(torch.int16))
        for k, v in (("row", row), ("sector", sector), ("leg", leg)):
            parts[k].append(v.to(torch.uint8))
        parts["pad"].append(pad.to(torch.int32).to(torch.int16))
        parts["time"].append((t * 32.0).round().clamp(0, synth.TIME_CODES - 1).to(torch.int32))
        have += len(good)
    f = {k: torch.cat(v) for k, v in parts.items()}
    over = f["row"].numel() - att
    if over < 0:  # a short sample of few tracks
        return _tracks(g, n_tracks, mix)
    # the frame's number of clusters is part of the case: the tracks lose what
    # they have too many at their ends, in proportion to their length
    n = f["ncl"].long()
    cut = ((n - 20) * (over / max(1, int((n - 20).sum())))).long()
    room = n - 20 - cut > 0
    cut += room & (torch.cumsum(room, 0) <= over - int(cut.sum()))
    start = torch.cumsum(n, 0) - n
    place = torch.arange(f["row"].numel(), device=DEV) - torch.repeat_interleave(start, n)
    keep = place < torch.repeat_interleave(n - cut, n)
    f["ncl"] = (n - cut).to(torch.int16)
    f.update({k: f[k][keep] for k in ("row", "sector", "leg", "pad", "time")})
    names = ("qtot_a", "qmax_a", "flags_a", "sigma_pad_a", "sigma_time_a")
    f.update(zip(names, _charges(g, f["row"].numel())))
    return f


def _bins(g, n, hot):
    """Bin of every unattached cluster."""
    w = torch.ones(NBIN, device=DEV)
    if hot:
        perm = torch.randperm(NBIN, generator=g, device=DEV)
        n_empty, n_hot = round(HOT["empty"] * NBIN), round(HOT["frac"] * NBIN)
        w[perm[:n_empty]] = 0.0
        w[perm[n_empty:n_empty + n_hot]] = HOT["share"] / n_hot
        w[perm[n_empty + n_hot:]] = (1.0 - HOT["share"]) / (NBIN - n_empty - n_hot)
    edge = torch.cumsum(w.double(), 0)
    return torch.searchsorted(edge, _rand(g, n) * edge[-1], right=True).clamp(max=NBIN - 1)


def _unattached(g, n, hot):
    """Unattached streams of a compressed frame: counts per bin, geometric
    time spacings that fill the frame, differences of uniform pads."""
    cnt = torch.bincount(_bins(g, n, hot), minlength=NBIN)
    binid = torch.repeat_interleave(torch.arange(NBIN, device=DEV), cnt)
    p = (cnt / synth.TIME_CODES).clamp(1e-9, 0.999999)[binid].double()
    tdiff = (torch.log1p(-_rand(g, n)) / torch.log1p(-p)).floor().clamp(max=2.0 ** 30)
    npu = torch.as_tensor(synth.NPADS * 64, device=DEV)[binid % NROW]
    pdiff = (_rand(g, n) * npu).long() - (_rand(g, n) * npu).long()
    f = {"n_unatt": cnt.to(torch.int32), "time_diff_u": tdiff.to(torch.int32),
         "pad_diff_u": pdiff.to(torch.int16)}
    f.update(zip(("qtot_u", "qmax_u", "flags_u", "sigma_pad_u", "sigma_time_u"), _charges(g, n)))
    return f


def _unattached_truth(g, n, hot):
    """Unattached clusters in generation order, the unattached encoder's input."""
    binid = _bins(g, n, hot)
    npu = torch.as_tensor(synth.NPADS * 64, device=DEV)[binid % NROW]
    f = {"row_u": (binid % NROW).to(torch.uint8), "sector_u": (binid // NROW).to(torch.uint8),
         "pad_u": (_rand(g, n) * npu).to(torch.int16),
         "time_u": torch.randint(0, synth.TIME_CODES, (n,), generator=g, device=DEV,
                                 dtype=torch.int32)}
    f.update(zip(("qtot_u", "qmax_u", "flags_u", "sigma_pad_u", "sigma_time_u"), _charges(g, n)))
    return f


def _frame(dec, g, n_tracks, n_unatt, mix):
    """A compressed frame on the device."""
    truth = _tracks(g, n_tracks, mix)
    truth.update(_unattached(g, n_unatt, mix == "stress"))
    return frames.assemble(truth, dec.encode(truth))


def _coded(frame):
    """The entropy-coded frame (host bytes) of a device frame."""
    return tmd.rans_encode({k: frame[k].cpu() for k, _, _ in tmd.FRAME_FIELDS})


def _outputs(frame_counts, host=False):
    """Empty results of a frame: native list, row offsets, attached counts, status."""
    _, na, nu = frame_counts
    kw = dict(pin_memory=True) if host else dict(device=DEV)
    return (torch.empty((na + nu, tmd.REC_BYTES), dtype=torch.uint8, **kw),
            torch.empty(NBIN + 1, dtype=torch.int32, **kw),
            torch.empty(NBIN, dtype=torch.int32, **kw), torch.empty(1, dtype=torch.int32, **kw))


def _batch_mix(case):
    """(tracks, unattached clusters, mix) of the batch's frames: log-uniform
    totals, pp-like to central Pb-Pb-like."""
    rng = np.random.default_rng(case["spec_seed"])
    out = []
    for _ in range(case["n_frames"]):
        total = math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))
        att = rng.uniform(0.25, 0.65)
        mix = "pp" if att < 0.4 else "small" if att < 0.5 else "pbpb"
        out.append((max(1, int(total * att / MIXES[mix]["per_track"])), int(total * (1 - att)), mix))
    return out


def _native(g, n):
    """A decoded cluster list: records with pads of their row and times of
    the 4000-bin frame, and its row offsets."""
    cnt = torch.bincount(_bins(g, n, False), minlength=NBIN)
    row_start = torch.zeros(NBIN + 1, dtype=torch.int32, device=DEV)
    row_start[1:] = torch.cumsum(cnt, 0)
    binid = torch.repeat_interleave(torch.arange(NBIN, device=DEV), cnt)
    npu = torch.as_tensor(synth.NPADS * 64, device=DEV)[binid % NROW]
    word = torch.empty((n, 3), dtype=torch.int32, device=DEV)
    word[:, 0] = torch.randint(0, synth.TIME_CODES, (n,), generator=g, device=DEV)
    sig = torch.randint(0, 1 << 15, (n,), generator=g, device=DEV)
    word[:, 1] = (_rand(g, n) * npu).to(torch.int32) | (sig << 16).to(torch.int32)
    word[:, 2] = torch.randint(0, 1 << 30, (n,), generator=g, device=DEV)
    return word.view(torch.uint8), row_start


class _State:
    """A decoder with a user's inputs; gives back what the decoder planned."""

    def __init__(self, kind):
        self.kind, self.dec, self.batch = kind, tmd.Decoder(0), None

    def __del__(self):
        if self.batch is not None:
            self.dec.tmd_batch_destroy(self.batch)
        self.dec.close()


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    s = _State(case["kind"])
    if s.kind in ("decode", "coded", "coded_host"):
        one = [_frame(s.dec, g, case["n_tracks"], case["n_unatt"], case["mix"])
               for _ in range(case.get("n_frames", 1))]
        s.counts = [tmd.counts(f) for f in one]
        if s.kind == "decode":
            s.frame = one[0]
        elif s.kind == "coded":
            s.coded = torch.from_numpy(_coded(one[0])).to(DEV)
        else:
            s.blobs = [torch.from_numpy(_coded(f)).pin_memory() for f in one]
            s.coded = [tmd.tmd_coded_frame(b.data_ptr(), b.numel(), *c)
                       for b, c in zip(s.blobs, s.counts)]
            s.out = [_outputs(c, host=True) for c in s.counts]
            s.fouts = [tmd.frame_out(*o) for o in s.out]
    elif s.kind == "batch":
        s.frames = [_frame(s.dec, g, *spec) for spec in _batch_mix(case)]
        s.out = [_outputs(tmd.counts(f)) for f in s.frames]
        s.batch = s.dec.tmd_batch_create([tmd.frame_in(f) for f in s.frames],
                                         [tmd.frame_out(*o) for o in s.out])
    elif s.kind == "encode_tracks":
        s.truth = _tracks(g, case["n_tracks"], case["mix"])
    elif s.kind == "encode_unatt":
        s.truth = _unattached_truth(g, case["n_unatt"], case["hot"])
    else:
        s.native, s.row_start = _native(g, case["n"])
    torch.cuda.synchronize()
    return s


def run(state):
    s, st = state, torch.cuda.current_stream()
    if s.kind == "decode":
        return s.dec.decode(s.frame, st)
    if s.kind == "coded":
        return s.dec.decode_coded(s.coded, *s.counts[0], stream=st)
    if s.kind == "coded_host":
        s.dec.tmd_decode_coded_host_stream(s.coded, s.fouts, st)
        return s.out
    if s.kind == "batch":
        s.dec.tmd_batch_launch(s.batch, st)
        return s.out
    if s.kind == "encode_tracks":
        return s.dec.encode(s.truth, st)
    if s.kind == "encode_unatt":
        return s.dec.encode_unattached(s.truth, st)
    return s.dec.global_xyz(s.native, s.row_start, st)


# ---------------------------------------------------------------------------
# least work and exact values
# ---------------------------------------------------------------------------
def _decode_bytes(nt, na, nu):
    """15 B of streams in and a 12 B record out per attached cluster (8 of the
    15 only after the first of a track), 13 + 12 B per unattached cluster, 11 B
    per track, the bin counts, row offsets and attached counts."""
    return 11 * nt + 7 * na + 8 * (na - nt) + 13 * nu + 12 * (na + nu) + 4 * NBIN * 3


def work(case):
    kind = case["kind"]
    if kind == "batch":
        spec = _batch_mix(case)
        na = [n_attached(nt, mix) for nt, _, mix in spec]
        # ~50 binary32 operations of the track model per attached cluster
        return {"bytes": sum(_decode_bytes(nt, a, nu) for (nt, nu, _), a in zip(spec, na)),
                "flops": 100 * sum(na)}
    if kind == "encode_unatt":  # 15 B in, 13 B out per cluster
        return {"bytes": 28 * case["n_unatt"] + 4 * NBIN, "flops": 0}
    if kind == "xyz":  # a 12 B record in, three floats out; about 8 operations
        return {"bytes": 24 * case["n"] + 4 * NBIN, "flops": 8 * case["n"]}
    nt = case["n_tracks"]
    na = n_attached(nt, case["mix"])
    if kind == "encode_tracks":  # 9 B in and 8 B out per cluster, 3 + 11 B per track
        return {"bytes": 17 * na + 14 * nt, "flops": 100 * na}
    nu, n = case["n_unatt"], case.get("n_frames", 1)
    if kind == "decode":
        return {"bytes": _decode_bytes(nt, na, nu), "flops": 100 * na}
    # coded frames: about 6.7 B per cluster come in coded, the records go out
    return {"bytes": n * (6.7 + 12) * (na + nu), "flops": n * 100 * na}


def exact(case, seed):
    """Global positions in 64 bits; every other output is an integer or a byte."""
    if case["kind"] != "xyz":
        return None
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    native, row_start = _native(g, case["n"])
    word = native.view(torch.int32)
    cnt = (row_start[1:] - row_start[:-1]).long()
    binid = torch.repeat_interleave(torch.arange(NBIN, device=DEV), cnt)
    row, sec = binid % NROW, binid // NROW
    x = 85.0 + row.double()
    npads = (66 + (72 * row) // 151).double()
    y = ((word[:, 1] & 0xFFFF).double() / 64.0 - npads / 2.0) * (
        2.0 * x * math.tan(math.radians(10.0)) / npads)
    psi = ((sec % 18) * 20 + 10).double() * (math.pi / 180.0)
    z = 250.0 - 0.5 * ((word[:, 0] & 0xFFFFFF).double() / 32.0)
    return (x * torch.cos(psi) - y * torch.sin(psi), x * torch.sin(psi) + y * torch.cos(psi),
            torch.where(sec < 18, z, -z))
