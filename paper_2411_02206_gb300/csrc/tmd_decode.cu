// tmd_decode.cu -- attached-cluster decoding and encoding (arXiv:2411.02206,
// Sec. 4: the attached-cluster kernel gives each thread one track; the thread
// carries the track model along the track through the TPC and restores each
// cluster's absolute coordinates from the stored residual and the model).
//
// Decoding of the attached clusters runs in three kernels:
//
//   k_track_decode  one lane per track, warps take up to 32 tracks at a time
//                   (task_lanes) from the length-sorted order (longest first,
//                   so lanes of a warp run loops of similar length and the tail
//                   is short).  For
//                   every cluster the lane applies the row and sector/leg
//                   differences, propagates the model to the row, adds the
//                   modular residuals to the quantised prediction and updates
//                   the model with the decoded cluster.  It writes, in input
//                   order j, the cluster's (sector,row) key, pad code and time
//                   code.
//   k_count_rank    (tmd_rank.cu) per-tile counts of the keys and the stable
//                   rank of every cluster within its (ranking tile, bin).
//   k_att_scatter   (tmd_scatter.cu) assembles the 12-byte native record of
//                   every attached cluster from the decoded coordinates and
//                   the charge streams and writes it at
//                   tileBase[tile(j)][key] + rank[j] (deterministic, no
//                   atomics).
//
// The lane-per-track walk reads each stream at 32 unrelated positions per
// warp.  Read directly, every lane pulls whole sectors for a few bytes and
// the L2 has to hold one line per lane and stream until the lane has walked
// past it.  k_track_decode therefore moves data in rounds of R steps (R = 16
// or 8, a tuning variant): each lane copies its own track's next round of
// differences into its half of a double buffer in shared memory with
// asynchronous copies while it runs the model through the current round, and
// the round's outputs leave through shared memory with coalesced stores.
//
// Encoder: the same walk with the truth as measurement; it writes the header
// and the residual streams (the synchronous side of the method).
#include <algorithm>

#include "tmd_internal.cuh"

namespace tmd {

namespace {

__device__ __forceinline__ uint32_t next_task(uint32_t* counter) {
  uint32_t task = 0;
  if ((threadIdx.x & 31) == 0) task = atomicAdd(counter, 1u);
  return __shfl_sync(0xffffffffu, task, 0);
}

constexpr uint32_t kFull = 0xffffffffu;

}  // namespace

// ---------------------------------------------------------------------------
// Asynchronous staging.  Each lane copies its own track's next round of
// differences into its own part of a double buffer with cp.async, so the
// copies of round r + 1 are in flight while the lane runs the model through
// round r, and no lane waits for another lane's copies.  The round's outputs
// still leave through shared memory with coalesced stores.
//
// A copy moves one 16-byte aligned window (it lies in the same 16 bytes as an
// element of the caller's array).  Every lane's copy is its own L1 request,
// and the requests, not the bytes, are what staging costs: a round of 16 steps
// takes 12 copies per lane (2 + 2 + 3 + 5) where copies of the aligned 4-byte
// words took 35 (431 -> 407 us for the 37.8 M clusters of a
// Pb-Pb-shaped frame).
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Copies the 16-byte windows from the one that holds `first` up to byte `end`
// (at most W of them).
template <int W>
__device__ __forceinline__ void cp_windows(const uint32_t* dst_smem, const void* first,
                                           const void* end) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_smem);
  const uintptr_t w = reinterpret_cast<uintptr_t>(first) & ~(uintptr_t)15;
  const uintptr_t e = reinterpret_cast<uintptr_t>(end);
#pragma unroll
  for (int c = 0; c < W; c++)
    if (w + 16 * c < e)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 16 * c), "l"(w + 16 * c)
                   : "memory");
}

// Offset of a byte in its window.
__device__ __forceinline__ int win_off(const void* p) {
  return (int)(reinterpret_cast<uintptr_t>(p) & 15);
}

// Windows that R elements of `size` bytes can touch.
constexpr int windows(int R, int size) { return (16 - size + R * size + 15) / 16; }

// Words per lane and buffer: windows of row_diff, sld, pad_res and time_res.
template <int R>
struct AsyncLayout {
  static constexpr int kW1 = windows(R, 1), kW2 = windows(R, 2), kW4 = windows(R, 4);
  static constexpr int kSl = 4 * kW1, kPr = 8 * kW1, kTr = kPr + 4 * kW2;
  static constexpr int kWin = 2 * kW1 + kW2 + kW4;
  static constexpr int kLane = 4 * (kWin | 1);  // an odd number of windows: the lanes' 16-byte
                                                // parts spread over the banks
};

template <int R>
struct AsyncStage {
  uint32_t buf[2][32 * AsyncLayout<R>::kLane];
  uint32_t kp[32 * (R + 1)];  // outputs key | pad << 16 of the round; [R]: the first
                              // cluster's time code
};

// Element offsets of step 0 of a round inside a lane's windows (one before
// the first element in round 0, whose step 0 has no difference).
struct RoundBase {
  int rd, sl, pr, tr;
};

// Issue the copies of the differences of steps [k0, k0 + R) of one track
// (cluster k uses difference dm1 + k; cluster 0 has none) into lane buffer lb.
template <int R>
__device__ __forceinline__ RoundBase issue_round(uint32_t* lb, uint32_t k0, uint32_t n,
                                                 uint32_t dm1, const uint8_t* rd_s,
                                                 const uint8_t* sld_s, const uint16_t* pr_s,
                                                 const uint32_t* tr_s) {
  using Lay = AsyncLayout<R>;
  const uint32_t k_lo = k0 > 1u ? k0 : 1u;
  const uint32_t k_hi = k0 + R < n ? k0 + R : n;
  if (k_lo >= k_hi) return RoundBase{0, 0, 0, 0};
  const uint32_t x_lo = dm1 + k_lo, x_hi = dm1 + k_hi;  // differences [x_lo, x_hi)
  const int skip = (int)(k_lo - k0);                    // 1 in round 0, else 0
  cp_windows<Lay::kW1>(lb, rd_s + x_lo, rd_s + x_hi);
  cp_windows<Lay::kW1>(lb + Lay::kSl, sld_s + x_lo, sld_s + x_hi);
  cp_windows<Lay::kW2>(lb + Lay::kPr, pr_s + x_lo, pr_s + x_hi);
  cp_windows<Lay::kW4>(lb + Lay::kTr, tr_s + x_lo, tr_s + x_hi);
  return RoundBase{win_off(rd_s + x_lo) - skip, win_off(sld_s + x_lo) - skip,
                   win_off(pr_s + x_lo) / 2 - skip, win_off(tr_s + x_lo) / 4 - skip};
}

}  // namespace

// Writes the (sector,row) key, the pad code and the time code of every
// attached cluster.
template <int R, int MINB>
__global__ void __launch_bounds__(kDecodeThreads, MINB)
    k_track_decode(const FrameDev* frames, PlanDev plan, uint32_t n_tasks) {
  static_assert(R == 8 || R == 16, "round length");
  using Lay = AsyncLayout<R>;
  constexpr int P = R + 1;   // pitch of the output rows
  constexpr int G = 32 / R;  // tracks per write-out instruction
  __shared__ RowGeo geo_s;
  extern __shared__ __align__(16) uint32_t s_stage[];
  fill_row_geo(&geo_s);
  chain_wait();
  __syncthreads();
  const RowGeo* geo = &geo_s;
  const uint32_t lane = threadIdx.x & 31, lanes = plan.lanes;
  const uint32_t sq = lane % R, sg = lane / R;
  AsyncStage<R>& S = reinterpret_cast<AsyncStage<R>*>(s_stage)[threadIdx.x >> 5];
  for (;;) {
    const uint32_t task = next_task(&plan.counters[0]);
    if (task >= n_tasks) break;
    const uint32_t f = find_frame(plan.pre_kt, plan.n_frames, task);
    const FrameDev& F = frames[f];
    const uint32_t idx =
        lane < lanes ? (task - plan.pre_kt[f]) * lanes + lane : 0xFFFFFFFFu;
    // the status and the task's order entries are loaded together
    const uint32_t nt = F.n_tracks;
    const uint32_t t_ord = idx < nt ? F.order[idx] : 0u;
    if (*F.status & kStCount) continue;
    const uint8_t* __restrict__ rd_s = F.row_diff;
    const uint8_t* __restrict__ sld_s = F.sld;
    const uint16_t* __restrict__ pr_s = F.pad_res;
    const uint32_t* __restrict__ tr_s = F.time_res;
    uint16_t* __restrict__ key_o = F.keys;
    uint16_t* __restrict__ pad_o = F.kf_pad;
    uint32_t* __restrict__ time_o = F.kf_time;
    uint32_t j0 = 0, n = 0, dm1 = 0, pad0 = 0, time0 = 0, st = 0, tmax = 0;
    Track s;
    s.max_row = 0;
    if (idx < nt) {
      const uint32_t t = t_ord;
      j0 = F.track_start[t];
      n = F.ncl[t];
      dm1 = j0 - t - 1u;
      pad0 = F.pad[t];
      time0 = F.time[t];
      const uint32_t raw = F.row[t], sec = F.slice[t];
      if (raw >= (uint32_t)kNRow || sec >= (uint32_t)kNSec) st |= kStRow;
      seed(geo, s, F.qpt[t], (int)raw, sec < (uint32_t)kNSec ? (int)sec : kNSec - 1, pad0,
           time0);
    }
    const uint32_t nmax = __reduce_max_sync(kFull, n);
    const uint32_t n_rounds = (nmax + R - 1) / R;
    uint32_t* lb0 = S.buf[0] + lane * Lay::kLane;
    uint32_t* lb1 = S.buf[1] + lane * Lay::kLane;
    RoundBase cur = issue_round<R>(lb0, 0u, n, dm1, rd_s, sld_s, pr_s, tr_s);
    cp_commit();
    for (uint32_t r = 0; r < n_rounds; r++) {
      const uint32_t k0 = r * R;
      uint32_t* lb = (r & 1) ? lb1 : lb0;
      RoundBase nxt{0, 0, 0, 0};
      if (r + 1 < n_rounds) {
        nxt = issue_round<R>((r & 1) ? lb0 : lb1, k0 + R, n, dm1, rd_s, sld_s, pr_s, tr_s);
        cp_commit();
        cp_wait<1>();
      } else {
        cp_wait<0>();
      }
      const uint32_t rem = n > k0 ? n - k0 : 0u;
      // the round's differences as byte and halfword loads from the lane's
      // buffer (step q at element base + q of each stream; the base is -1 in
      // round 0, whose step 0 reads none)
      const uint8_t* rd_b = reinterpret_cast<const uint8_t*>(lb);
      const uint8_t* sl_b = reinterpret_cast<const uint8_t*>(lb + Lay::kSl);
      const uint16_t* pr_b = reinterpret_cast<const uint16_t*>(lb + Lay::kPr);
      uint32_t* tr_b = lb + Lay::kTr + cur.tr;  // becomes the time code
      // What a step needs and no decoded coordinate enters (its differences, its
      // row and the row's geometry) is fetched a step ahead, before the stores
      // of the step in between: three shared-memory latencies one after the
      // other outside the model chain (decode kernel 39.9 ->
      // 37.1 us for 2000 tracks, 388 -> 385 us for 400 k; encoder 299 -> 290 us).  The fetch after the round's
      // last step stays within the lane's windows and is not used.
      struct Ahead {
        int raw;
        uint32_t sl, pr, tr;
        float4 G;
      } nx;
      auto fetch = [&](uint32_t q) {
        nx.raw = (s.raw_row + (int)rd_b[cur.rd + (int)q]) & 255;
        nx.sl = sl_b[cur.sl + (int)q];
        nx.pr = pr_b[cur.pr + (int)q];
        nx.tr = tr_b[q];
        nx.G = geo->row[clamp_row(nx.raw)];
      };
      // one model step: cluster k0 + q >= 1 of the lane's track
      auto step = [&](uint32_t q) {
        const Ahead c = nx;
        const float4& G = c.G;
        row_step(s, c.raw);
        fetch(q + 1);
        turn_step(geo, s, c.sl);
        uint32_t ppad, ptime;
        propagate_predict(G, s, ppad, ptime);
        const uint32_t padq = (ppad + c.pr) & 0xFFFFu;
        const uint32_t timeq = ptime + c.tr;
        update(G, s, padq, timeq);
        tmax = max(tmax, timeq);
        S.kp[lane * P + q] = (uint32_t)(s.sec * kNRow + s.row) | (padq << 16);
        tr_b[q] = timeq;
      };
      uint32_t q0 = 0;
      if (k0 == 0) {  // the track's first cluster, stored absolute
        if (rem > 0) {
          tmax = max(tmax, time0);
          S.kp[lane * P] = (uint32_t)(s.sec * kNRow + s.row) | (pad0 << 16);
          S.kp[lane * P + R] = time0;
        }
        q0 = 1;
      }
      if (rem > 0) fetch(q0);
      // rounds in which every lane has all R steps left run without the
      // per-step bound test (the common case for the long tracks decoded first)
      const bool full = __all_sync(kFull, rem >= (uint32_t)R || lane >= lanes);
      if (full) {
        if (lane < lanes) {
#pragma unroll 4
          for (uint32_t q = q0; q < (uint32_t)R; q++) step(q);
        }
      } else {
#pragma unroll 1
        for (uint32_t q = q0; q < (uint32_t)R; q++)
          if (q < rem) step(q);
      }
      __syncwarp();
      const uint32_t k = k0 + sq;
      const uint32_t* bb = ((r & 1) ? S.buf[1] : S.buf[0]) + Lay::kTr + (int)sq - 1;
#pragma unroll
      for (int i0 = 0; i0 < 32; i0 += G) {
        if (i0 >= (int)lanes) break;
        const uint32_t i = i0 + sg;
        const uint32_t ji = __shfl_sync(kFull, j0, i);
        // length and time offset of track i; in a full round every track has step k
        const uint32_t no = __shfl_sync(kFull, n | ((uint32_t)(cur.tr + 1) << 16), i);
        if (full || k < (no & 0xFFFFu)) {
          const uint32_t a = S.kp[i * P + sq];
          const uint32_t* t = k ? bb + i * Lay::kLane + (no >> 16) : S.kp + i * P + R;
          key_o[ji + k] = (uint16_t)(a & 0xFFFFu);
          pad_o[ji + k] = (uint16_t)(a >> 16);
          time_o[ji + k] = *t;
        }
      }

      __syncwarp();
      cur = nxt;
    }
    if (s.max_row >= kNRow) st |= kStRow;
    if (tmax > 0xFFFFFFu) st |= kStTime;
    st = __reduce_or_sync(kFull, st);
    if (st && lane == 0) atomicOr(frames[f].status, st);
  }
}

template <int R>
constexpr int kDecodeSmem = (kDecodeThreads / 32) * (int)sizeof(AsyncStage<R>);

// Variants: 0 -> rounds of 16 steps (3 blocks per SM), 1 -> rounds of 8
// steps (5 blocks per SM).
void launch_track_decode(int variant, uint32_t grid, cudaStream_t st, const FrameDev* frames,
                         PlanDev plan, uint32_t n_tasks) {
  if (variant == 1)
    launch_chained(k_track_decode<8, 5>, grid, kDecodeThreads, kDecodeSmem<8>, st, frames,
                   plan, n_tasks);
  else
    launch_chained(k_track_decode<16, 3>, grid, kDecodeThreads, kDecodeSmem<16>, st, frames,
                   plan, n_tasks);
}

cudaError_t prepare_track_decode(int variant, int* blocks_per_sm) {
  const auto kern = variant == 1 ? k_track_decode<8, 5> : k_track_decode<16, 3>;
  const int smem = variant == 1 ? kDecodeSmem<8> : kDecodeSmem<16>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, kDecodeThreads, smem);
}

// Float-path trace: one thread per selected track walks it through the
// compressed frame like the decoder (one global load per stream and step; a
// debugging path, not a fast one) and writes the binary32 model state after
// every cluster: x, y, dy/dx, d2y/dx2, the six y-covariance terms, t, dt/dx,
// the three t-covariance terms, row and sector (as floats).
__global__ void k_track_trace(const FrameDev* frames, const uint32_t* ids, uint32_t n_ids,
                              float* state) {
  __shared__ RowGeo geo;
  fill_row_geo(&geo);
  __syncthreads();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const FrameDev& F = frames[0];
  if (i >= n_ids || (*F.status & kStCount)) return;
  const uint32_t t = ids[i];
  if (t >= F.n_tracks) return;
  const uint32_t j0 = F.track_start[t], n = F.ncl[t], dm1 = j0 - t - 1u;
  const uint32_t raw = F.row[t], sec = F.slice[t];
  Track s;
  seed(&geo, s, F.qpt[t], (int)raw, sec < (uint32_t)kNSec ? (int)sec : kNSec - 1, F.pad[t],
       F.time[t]);
  for (uint32_t k = 0; k < n && k < (uint32_t)kNRow; k++) {
    if (k > 0) {
      const uint32_t d = dm1 + k;
      row_step(s, (s.raw_row + (int)F.row_diff[d]) & 255);
      turn_step(&geo, s, F.sld[d]);
      uint32_t ppad, ptime;
      const float4 G = geo.row[s.row];
      propagate_predict(G, s, ppad, ptime);
      update(G, s, (ppad + F.pad_res[d]) & 0xFFFFu, ptime + F.time_res[d]);
    }
    float* o = state + ((size_t)i * kNRow + k) * 17;
    o[0] = s.x; o[1] = s.y; o[2] = s.ty; o[3] = s.c;
    o[4] = s.c00; o[5] = s.c01; o[6] = s.c02; o[7] = s.c11; o[8] = s.c12; o[9] = s.c22;
    o[10] = s.t; o[11] = s.tt; o[12] = s.d00; o[13] = s.d01; o[14] = s.d11;
    o[15] = (float)s.row; o[16] = (float)s.sec;
  }
}

// ---------------------------------------------------------------------------
// Encoder staging: 14 windows per lane and round of 16 clusters (row, sector
// and leg 2 each, pad 3, time 5).  A round advances every stream by a multiple
// of 16 bytes, so the offset of a round's first cluster in its windows is a
// constant of the track.
// ---------------------------------------------------------------------------
namespace {

constexpr int kEncRound = 16;

struct EncStage {
  static constexpr int kSec = 8, kLeg = 16, kPad = 24, kTime = 36;  // first words (row: 0)
  static constexpr int kLane = 60;     // 56 words; an odd number of 16-byte units
  static constexpr int kPitch = kEncRound + 1;
  uint32_t buf[2][32 * kLane];
  uint32_t res[32 * kPitch];   // row difference | sector/leg << 8 | pad residual << 16
};

// Copies, for every track of the warp, the 16-byte windows that hold elements
// [x, x + cnt) of `src` (SZ bytes each) into the track's part of the buffer
// (`pitch` words apart from dst): window c of track t by lane (t W + c) % 32,
// so that a track's windows are one or two L1 requests, where each is its
// own in cp_windows: 14.9 M against 18.4 M requests to L2 and 299 against 343 us
// for 200 k tracks.  Lane t holds track t's x and cnt (0: nothing).
// The decoder, nearer to its issue limit, gains nothing: 382 against 388 us for
// 400 k tracks, and 45 against 40 us for 2000.
template <int W, int SZ>
__device__ __forceinline__ void cp_windows_of_warp(const uint32_t* dst_smem, int pitch, const void* src,
                                           uint32_t x_own, uint32_t cnt_own, uint32_t lanes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_smem), lane = threadIdx.x & 31;
  const uintptr_t base = reinterpret_cast<uintptr_t>(src);
#pragma unroll
  for (int i = 0; i < W; i++) {
    if (32u * i >= W * lanes) break;
    const uint32_t t = (32 * i + lane) / W, c = (32 * i + lane) % W;
    const uint32_t x = __shfl_sync(0xffffffffu, x_own, t);
    const uint32_t cnt = __shfl_sync(0xffffffffu, cnt_own, t);
    const uintptr_t a = base + (uintptr_t)x * SZ;
    if (cnt != 0 && (uint32_t)(a & 15) + cnt * SZ > 16 * c)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 4 * (t * pitch) + 16 * c),
                   "l"((a & ~(uintptr_t)15) + 16 * c)
                   : "memory");
  }
}

struct Truth {
  const uint8_t *row, *sector, *leg;
  const uint16_t* pad;
  const uint32_t* time;
};

// Truth of clusters [j, j + m) of every track of the warp, m <= kEncRound.
__device__ __forceinline__ void issue_truth(uint32_t* buf, const Truth& E, uint32_t j, uint32_t m,
                                            uint32_t lanes) {
  using S = EncStage;
  cp_windows_of_warp<5, 4>(buf + S::kTime, S::kLane, E.time, j, m, lanes);
  cp_windows_of_warp<3, 2>(buf + S::kPad, S::kLane, E.pad, j, m, lanes);
  cp_windows_of_warp<2, 1>(buf, S::kLane, E.row, j, m, lanes);
  cp_windows_of_warp<2, 1>(buf + S::kSec, S::kLane, E.sector, j, m, lanes);
  cp_windows_of_warp<2, 1>(buf + S::kLeg, S::kLane, E.leg, j, m, lanes);
}

}  // namespace

// Writes the headers and the residual streams of the attached clusters.  One
// lane per track like the decoder, with the truth staged a round ahead and the
// residuals leaving through shared memory: read and written directly, 13
// unrelated sectors per lane and step, the walk took 2.72 ms for 200 k tracks
// (18 M clusters); staged it takes 0.30 ms.
__global__ void __launch_bounds__(kDecodeThreads, 3)
    k_track_encode(const EncDev* enc, const FrameDev* frames, PlanDev plan, uint32_t n_tasks,
                   uint32_t too_short) {
  constexpr int R = kEncRound, P = EncStage::kPitch;
  __shared__ RowGeo geo;
  extern __shared__ __align__(16) uint32_t s_stage[];
  fill_row_geo(&geo);
  chain_wait();
  __syncthreads();
  EncStage& S = reinterpret_cast<EncStage*>(s_stage)[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31, lanes = plan.lanes;
  const uint32_t sq = lane % R, sg = lane / R;
  for (;;) {
    const uint32_t task = next_task(&plan.counters[0]);
    if (task >= n_tasks) break;
    const uint32_t f = find_frame(plan.pre_warp, plan.n_frames, task);
    const FrameDev& F = frames[f];
    const EncDev& D = enc[f];
    if (*F.status & kStCount) continue;
    const uint32_t idx =
        lane < lanes ? (task - plan.pre_warp[f]) * lanes + lane : 0xFFFFFFFFu;
    // in registers: stores to the output bytes may alias the descriptor
    const Truth E{D.row, D.sector, D.leg, D.pad, D.time};
    uint8_t* __restrict__ rd_o = D.o_row_diff;
    uint8_t* __restrict__ sld_o = D.o_sld;
    uint16_t* __restrict__ pr_o = D.o_pad_res;
    uint32_t* __restrict__ tr_o = D.o_time_res;
    uint32_t st = 0, t = 0, j0 = 0, n = 0, rmax = 0, smax = 0;
    Track s;
    if (idx < F.n_tracks) {
      t = F.order[idx];
      j0 = F.track_start[t];
      n = D.ncl[t];
    }
    const uint32_t dm1 = j0 - t - 1u;  // cluster k >= 1 has difference dm1 + k
    const uint32_t nmax = __reduce_max_sync(kFull, n);
    if (nmax <= too_short) break;  // this task and those after it: k_track_encode_short
    const uint32_t rounds = (nmax + R - 1) / R;
    uint32_t* lb0 = S.buf[0] + lane * EncStage::kLane;
    uint32_t* lb1 = S.buf[1] + lane * EncStage::kLane;
    issue_truth(S.buf[0], E, j0, min(n, (uint32_t)R), lanes);
    cp_commit();
    // offsets of a round's first cluster in its windows
    const int o_row = win_off(E.row + j0), o_sec = win_off(E.sector + j0);
    const int o_leg = win_off(E.leg + j0), o_pad = win_off(E.pad + j0) / 2;
    const int o_time = win_off(E.time + j0) / 4;
    uint32_t r0 = 0, s0 = 0, l0 = 0;  // row, sector, leg of the cluster before
    for (uint32_t r = 0; r < rounds; r++) {
      const uint32_t k0 = r * R;
      uint32_t* lb = (r & 1) ? lb1 : lb0;
      if (r + 1 < rounds) {
        issue_truth(S.buf[(r & 1) ^ 1], E, j0 + k0 + R, n > k0 + R ? min(n - k0 - R, (uint32_t)R) : 0u,
                    lanes);
        cp_commit();
        cp_wait<1>();
      } else {
        cp_wait<0>();
      }
      __syncwarp();  // the other lanes' copies too
      const uint8_t* row_b = reinterpret_cast<const uint8_t*>(lb) + o_row;
      const uint8_t* sec_b = reinterpret_cast<const uint8_t*>(lb + EncStage::kSec) + o_sec;
      const uint8_t* leg_b = reinterpret_cast<const uint8_t*>(lb + EncStage::kLeg) + o_leg;
      const uint16_t* pad_b = reinterpret_cast<const uint16_t*>(lb + EncStage::kPad) + o_pad;
      uint32_t* time_b = lb + EncStage::kTime + o_time;  // becomes the time residual
      const uint32_t rem = n > k0 ? n - k0 : 0u;
      uint32_t q0 = 0;
      if (k0 == 0) {  // the first cluster is stored absolute
        if (rem > 0) {
          r0 = row_b[0];
          s0 = sec_b[0];
          l0 = leg_b[0];
          const uint32_t pad = pad_b[0], time = time_b[0];
          rmax = r0;
          smax = s0;
          const uint8_t qpt = D.qpt[t];
          D.o_qpt[t] = qpt;
          D.o_ncl[t] = (uint16_t)n;
          D.o_row[t] = (uint8_t)r0;
          D.o_slice[t] = (uint8_t)s0;
          D.o_pad[t] = (uint16_t)pad;
          D.o_time[t] = time;
          seed(&geo, s, qpt, (int)r0, s0 < (uint32_t)kNSec ? (int)s0 : kNSec - 1, pad, time);
        }
        q0 = 1;
      }
      // the truth of the next step and its row's geometry, a step ahead as in
      // the decoder
      struct Ahead {
        uint32_t row, sec, leg, pad, time;
        float4 G;
      } nx;
      auto fetch = [&](uint32_t q) {
        nx.row = row_b[q];
        nx.sec = sec_b[q];
        nx.leg = leg_b[q];
        nx.pad = pad_b[q];
        nx.time = time_b[q];
        nx.G = geo.row[clamp_row((int)nx.row)];
      };
      auto step = [&](uint32_t q) {
        const Ahead c = nx;
        const float4& G = c.G;
        fetch(q + 1);
        rmax = max(rmax, c.row);
        smax = max(smax, c.sec);
        const uint32_t rd = (c.row - r0) & 255u;
        const uint32_t sld = (c.leg != l0 ? (uint32_t)kNSec : 0u) + (c.sec - s0 + 8u * kNSec) % kNSec;
        r0 = c.row;
        s0 = c.sec;
        l0 = c.leg;
        row_step(s, (int)c.row);  // the walk of the differences ends at the row itself
        turn_step(&geo, s, sld);
        uint32_t ppad, ptime;
        propagate_predict(G, s, ppad, ptime);
        const uint32_t padq = c.pad, timeq = c.time;
        S.res[lane * P + q] = rd | (sld << 8) | ((padq - ppad) << 16);
        time_b[q] = timeq - ptime;
        update(G, s, padq, timeq);
      };
      if (rem > 0) fetch(q0);
      const bool full = __all_sync(kFull, rem >= (uint32_t)R || lane >= lanes);
      if (full) {
        if (lane < lanes) {
#pragma unroll 4
          for (uint32_t q = q0; q < (uint32_t)R; q++) step(q);
        }
      } else {
#pragma unroll 1
        for (uint32_t q = q0; q < (uint32_t)R; q++)
          if (q < rem) step(q);
      }
      __syncwarp();
      const uint32_t k = k0 + sq;
      const uint32_t* bb = (r & 1) ? S.buf[1] : S.buf[0];
#pragma unroll
      for (int i0 = 0; i0 < 32; i0 += 32 / R) {
        if (i0 >= (int)lanes) break;
        const uint32_t i = i0 + sg;
        const uint32_t di = __shfl_sync(kFull, dm1, i) + k;
        const uint32_t no = __shfl_sync(kFull, n | ((uint32_t)o_time << 16), i);
        if (k < (no & 0xFFFFu) && k > 0) {
          const uint32_t a = S.res[i * P + sq];
          rd_o[di] = (uint8_t)a;
          sld_o[di] = (uint8_t)(a >> 8);
          pr_o[di] = (uint16_t)(a >> 16);
          tr_o[di] = bb[i * EncStage::kLane + EncStage::kTime + (no >> 16) + sq];
        }
      }
      __syncwarp();
    }
    if (rmax >= (uint32_t)kNRow || smax >= (uint32_t)kNSec) st |= kStRow;
    st = __reduce_or_sync(kFull, st);
    if (st && lane == 0) atomicOr(F.status, st);
  }
}

constexpr int kEncodeSmem = (kDecodeThreads / 32) * (int)sizeof(EncStage);

// The same walk for tracks of up to kShortTrack clusters, read and written directly:
// a warp's time is that of fetching its task, and what counts is warps per SM.  Tasks
// with a longer track are left to k_track_encode.
constexpr uint32_t kShortTrack = 4;
constexpr int kShortThreads = 256;
__global__ void __launch_bounds__(kShortThreads, 4)
    k_track_encode_short(const EncDev* enc, const FrameDev* frames, PlanDev plan,
                         uint32_t n_tasks) {
  __shared__ RowGeo geo;
  fill_row_geo(&geo);
  chain_wait();
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31, lanes = plan.lanes;
  const FrameDev& F = frames[0];  // an encoding call has one frame
  const EncDev& D = enc[0];
  if (*F.status & kStCount) return;
  const Truth E{D.row, D.sector, D.leg, D.pad, D.time};
  for (;;) {
    const uint32_t ticket = next_task(&plan.counters[1]);
    if (ticket >= n_tasks) break;
    const uint32_t idx = lane < lanes ? ticket * lanes + lane : 0xFFFFFFFFu;
    uint32_t st = 0, t = 0, j0 = 0, n = 0, r0 = 0, s0 = 0, l0 = 0, pad = 0, time = 0;
    uint8_t qpt = 0;
    Track s;
    if (idx < F.n_tracks) {
      t = F.order[idx];
      j0 = F.track_start[t];
      n = D.ncl[t];
      r0 = E.row[j0];
      s0 = E.sector[j0];
      l0 = E.leg[j0];
      pad = E.pad[j0], time = E.time[j0];
      qpt = D.qpt[t];
    }
    const uint32_t nmax = __reduce_max_sync(kFull, n);
    if (nmax > kShortTrack) continue;
    if (n > 0) {
      if (r0 >= (uint32_t)kNRow || s0 >= (uint32_t)kNSec) st |= kStRow;
      D.o_qpt[t] = qpt;
      D.o_ncl[t] = (uint16_t)n;
      D.o_row[t] = (uint8_t)r0;
      D.o_slice[t] = (uint8_t)s0;
      D.o_pad[t] = (uint16_t)pad;
      D.o_time[t] = time;
      if (n > 1) seed(&geo, s, qpt, (int)r0, s0 < (uint32_t)kNSec ? (int)s0 : kNSec - 1, pad, time);
    }
    for (uint32_t k = 1; k < nmax; k++) {
      if (k >= n) continue;
      const uint32_t d = j0 - t + k - 1, j = j0 + k;
      const uint32_t r1 = E.row[j], s1 = E.sector[j], l1 = E.leg[j];
      const uint32_t padq = E.pad[j], timeq = E.time[j];
      if (r1 >= (uint32_t)kNRow || s1 >= (uint32_t)kNSec) st |= kStRow;
      const uint32_t sld = (l1 != l0 ? (uint32_t)kNSec : 0u) + (s1 - s0 + 8u * kNSec) % kNSec;
      D.o_row_diff[d] = (uint8_t)(r1 - r0);
      D.o_sld[d] = (uint8_t)sld;
      r0 = r1;
      s0 = s1;
      l0 = l1;
      row_step(s, (int)r1);
      turn_step(&geo, s, sld);
      uint32_t ppad, ptime;
      const float4 G = geo.row[s.row];
      propagate_predict(G, s, ppad, ptime);
      D.o_pad_res[d] = (uint16_t)((padq - ppad) & 0xFFFFu);
      D.o_time_res[d] = timeq - ptime;
      update(G, s, padq, timeq);
    }
    st = __reduce_or_sync(kFull, st);
    if (st && lane == 0) atomicOr(F.status, st);
  }
}

// Calls of up to kShortTrack clusters per track go to both kernels, the others to
// the staged one alone.  A million tracks of 1, 2, 3, 4, 6 and 8 clusters: 96, 103, 124, 157,
// 234 and 321 us by the short walk, 149, 173, 177, 181, 203 and 218 us staged; 300 k: 66, 70,
// 79, 91, 110 and 136 against 86, 96, 95, 98, 100 and 106 us.  The short walk goes first: behind
// the staged kernel, whose shared memory leaves it little L1, 4 M tracks of 4 clusters
// take 565 instead of 454 us.
void launch_track_encode(uint64_t n_tracks, uint64_t n_attached, uint32_t sms,
                         const int* blocks_per_sm, cudaStream_t st, const EncDev* enc,
                         const FrameDev* frames, PlanDev plan, uint32_t n_tasks) {
  const bool both = n_attached <= kShortTrack * n_tracks;
  auto grid = [&](uint32_t threads, int bps) {
    const uint32_t per_block = threads / 32;
    return std::min<uint32_t>((n_tasks + per_block - 1) / per_block, sms * (uint32_t)bps);
  };
  if (both)
    launch_chained(k_track_encode_short, grid(kShortThreads, blocks_per_sm[1]), kShortThreads, 0, st,
                   enc, frames, plan, n_tasks);
  launch_chained(k_track_encode, grid(kDecodeThreads, blocks_per_sm[0]), kDecodeThreads, kEncodeSmem,
                 st, enc, frames, plan, n_tasks, both ? kShortTrack : 0u);
}

cudaError_t prepare_track_encode(int* blocks_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_track_encode, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kEncodeSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[0], k_track_encode,
                                                      kDecodeThreads, kEncodeSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[1], k_track_encode_short,
                                                      kShortThreads, 0);
  return e;
}

}  // namespace tmd
