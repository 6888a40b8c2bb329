// tmd_unatt_encode.cu -- unattached-cluster encoding on the GPU (the
// synchronous side of arXiv:2411.02206, Sec. 4: the clusters that no track
// claimed are sorted by their position in the TPC and each is stored as the
// difference to the cluster before it).
//
// Per (sector,row) bin the clusters are ordered by (time, pad), ties in input
// order, and stored as pad / time differences to the preceding cluster of the
// bin (the first to zero), mod 2^16 / 2^32, with their charges, flags and
// sigmas in the same order; the bins follow each other in bin order.
//
// The sort goes from the most significant digit down, so that a cluster moves
// through memory once as one 16-byte record (its native record and its input
// index) and everything else happens on chip:
//
//   k_ue_init     outputs that are summed into, control block
//   k_ue_count    clusters per bin
//   k_ue_plan     first output position of every bin; bins by size
//   k_ue_scatter  every record to its bin's range, in any order within it
//   k_ue_sort_warp / _block / _big
//                 sort one bin by (time, pad, index) and write its streams: a
//                 warp for up to kUeWarpMax clusters, a block for up to
//                 kUeBlockMax, a large block per time slice beyond that
//   k_ue_general  least-significant-digit radix sort of whatever the others
//                 leave (leaves at once when there is nothing): frames with
//                 times of 2^24 and more, which the record does not hold, and
//                 bins that are too large or more than a slice of whose
//                 clusters crowd on one time
//
// A bin's sort is a distribution sort: as many buckets as clusters, equally
// wide between the bin's first and last time, so a bucket holds about one
// cluster and a few comparisons finish it.  The previous form, eight stable
// radix passes over 64-bit keys and a random gather of the charges, moved each
// cluster nine times: 3.60 ms for 20 M clusters against 0.59 ms now, and 0.193 ms
// in 35 launches for 100 k clusters against 0.054 ms in 8.
#include <algorithm>
#include <cstring>

#include "tmd_api_internal.h"
#include "tmd_internal.cuh"

namespace tmd {
namespace {

constexpr uint32_t kUeWarpMax = 128;      // clusters of a bin sorted by one warp
constexpr uint32_t kUeBlockMax = 4096;    // by one block of kUeBlockThreads
constexpr int kUeBlockThreads = 512;
constexpr uint32_t kUeSliceCap = 16384;   // by one block of kUeBigThreads, per time slice
constexpr uint32_t kUeSliceMean = 12288;  // aimed at, leaving room for uneven times
constexpr int kUeBigThreads = 1024;
// Larger bins go to the general sort: a slice reads its whole bin, so the work grows
// with the square.  Bins of 250 k: 36 of them 0.97 ms by slices and 1.13 ms in the
// general sort; a single one 0.21 and 0.15 ms, 300 of 120 k 2.5 and 5.8 ms.
constexpr uint32_t kUeBigMax = 1u << 18;
constexpr uint32_t kUeSlices = (kUeBigMax + kUeSliceMean - 1) / kUeSliceMean;
constexpr uint32_t kUeWhole = 255;        // instead of a slice: all of the bin's
constexpr uint32_t kUeWholeSlices = 4;    // see k_ue_sort_big
static_assert(kUeSlices < kUeWhole, "a slice in the low byte of its list entry");
constexpr uint32_t kUeBucketMax = 64;     // clusters of a bucket that one thread may sort
constexpr int kUeScatThreads = 512;

constexpr int kRsThreads = 256;
constexpr int kRsPerThread = 8;
constexpr uint32_t kRsTile = kRsThreads * kRsPerThread;  // keys per tile
constexpr int kRsWarps = kRsThreads / 32;

// Zeroed by k_ue_init, lists and counts written by k_ue_plan.
struct UeCtl {
  uint32_t wide;               // a time of 2^24 or more: everything in the general sort
  uint32_t n_general;          // bins marked for the general sort
  uint32_t n_block, n_big;     // bins, bins or slices in the lists
  uint32_t next_block, next_big;
  uint32_t barrier;            // arrivals at the general sort's grid barriers
  uint32_t not_tmin, tmax, pmax;  // of the general sort's clusters (~earliest, latest time)
  uint32_t general[kNBin];     // marks
};
struct UePlan {
  uint32_t start[kNBin + 1];   // first output position of every bin
  uint32_t cursor[kNBin];      // next free record of every bin during the scatter
  uint32_t block[kNBin];       // bins
};
// bin << 8 | time slice or kUeWhole
struct UeBig {
  uint32_t item[kNBin * kUeSlices];
};

struct UeArgs {
  uint32_t n;
  const uint8_t* row;
  const uint8_t* sector;
  const uint16_t* pad;
  const uint32_t* time;
  const uint16_t* qtot;
  const uint16_t* qmax;
  const uint8_t* flags;
  const uint8_t* sigp;
  const uint8_t* sigt;
  uint32_t* n_unatt;
  uint16_t* pad_diff;
  uint32_t* time_diff;
  uint16_t* qtot_o;
  uint16_t* qmax_o;
  uint8_t* flags_o;
  uint8_t* sigp_o;
  uint8_t* sigt_o;
  uint32_t* status;
  int vec;  // every input aligned for loads of four clusters
};

// Bin of a cluster; a row >= 152 or a sector >= 36 counts in bin 5471.
__device__ __forceinline__ uint32_t ue_bin(uint32_t row, uint32_t sector, uint32_t& st) {
  if (row >= (uint32_t)kNRow || sector >= (uint32_t)kNSec) {
    st = kStRow;
    return kNBin - 1;
  }
  return sector * kNRow + row;
}

__global__ void __launch_bounds__(256) k_ue_init(UeArgs a, UeCtl* ctl) {
  const uint32_t i = blockIdx.x * 256 + threadIdx.x;
  if (i < (uint32_t)kNBin) a.n_unatt[i] = 0u;
  if (i < sizeof(UeCtl) / 4) reinterpret_cast<uint32_t*>(ctl)[i] = 0u;
  if (i == 0) *a.status = 0u;
}

// Clusters per bin: counters in shared memory, added to the output once per
// block (so a block takes at least a few thousand clusters).
__global__ void __launch_bounds__(1024) k_ue_count(UeArgs a) {
  chain_wait();
  __shared__ uint32_t s_cnt[kNBin];
  for (int i = threadIdx.x; i < kNBin; i += 1024) s_cnt[i] = 0u;
  __syncthreads();
  uint32_t st = 0;
  const uint32_t groups = a.n / 4 + (a.n % 4 != 0);
  for (uint32_t g = blockIdx.x * 1024 + threadIdx.x; g < groups; g += gridDim.x * 1024) {
    const uint32_t i = g * 4;
    if (a.vec && a.n - i >= 4) {
      const uint32_t r = *reinterpret_cast<const uint32_t*>(a.row + i);
      const uint32_t s = *reinterpret_cast<const uint32_t*>(a.sector + i);
#pragma unroll
      for (int q = 0; q < 4; q++)
        atomicAdd(&s_cnt[ue_bin((r >> (8 * q)) & 255u, (s >> (8 * q)) & 255u, st)], 1u);
    } else {
      for (uint32_t q = 0; q < 4 && q < a.n - i; q++)
        atomicAdd(&s_cnt[ue_bin(a.row[i + q], a.sector[i + q], st)], 1u);
    }
  }
  if (__syncthreads_or(st != 0) && threadIdx.x == 0) atomicOr(a.status, kStRow);
  for (int i = threadIdx.x; i < kNBin; i += 1024)
    if (s_cnt[i]) atomicAdd(&a.n_unatt[i], s_cnt[i]);
}

// Exclusive scan over a block of B threads; total in tot.
template <int B>
__device__ __forceinline__ uint32_t ue_scan(uint32_t v, uint32_t& tot) {
  __shared__ uint32_t s_w[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  // every warp scans the warp totals
  const uint32_t t = lane < B / 32 ? s_w[lane] : 0u;
  uint32_t y = t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) y += z;
  }
  tot = __shfl_sync(0xffffffffu, y, 31);
  const uint32_t off = __shfl_sync(0xffffffffu, y - t, w);
  __syncthreads();
  return off + x - v;
}

// One block: output positions of the bins, and which kernel sorts each.  Bins
// are read and written by neighbouring lanes at neighbouring bins, the scan over
// consecutive bins goes through shared memory.
__global__ void __launch_bounds__(1024) k_ue_plan(UeArgs a, UePlan* plan, UeBig* big,
                                                  UeCtl* ctl, uint32_t sms) {
  constexpr int Q = (kNBin + 1023) / 1024;
  static_assert(kNBin % Q == 0, "a thread has all its bins or none");
  __shared__ uint32_t s_bin[kNBin];
  __shared__ uint32_t s_block, s_bins, s_sliced, s_big, s_general;
  chain_wait();
  const uint32_t tid = threadIdx.x, b0 = tid * Q;
  uint32_t n[Q], v[Q], sum = 0, tot;
#pragma unroll
  for (int q = 0; q < Q; q++)
    n[q] = tid + 1024 * q < (uint32_t)kNBin ? a.n_unatt[tid + 1024 * q] : 0u;
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (tid + 1024 * q < (uint32_t)kNBin) s_bin[tid + 1024 * q] = n[q];
  if (tid == 0) s_block = s_bins = s_sliced = s_big = s_general = 0u;
  __syncthreads();
  const bool mine = b0 < (uint32_t)kNBin;
#pragma unroll
  for (int q = 0; q < Q; q++) {
    v[q] = mine ? s_bin[b0 + q] : 0u;
    sum += v[q];
  }
  uint32_t run = ue_scan<1024>(sum, tot);
#pragma unroll
  for (int q = 0; q < Q; q++) {
    if (mine) s_bin[b0 + q] = run;
    run += v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < Q; q++) {
    const uint32_t b = tid + 1024 * q;
    if (b >= (uint32_t)kNBin) break;
    plan->start[b] = plan->cursor[b] = s_bin[b];
    if (n[q] > kUeBigMax) {
      ctl->general[b] = 1u;
      atomicAdd(&s_general, 1u);
    } else if (n[q] > kUeBlockMax) {
      atomicAdd(&s_bins, 1u);
      if (n[q] <= kUeSliceMean) big->item[atomicAdd(&s_big, 1u)] = (b << 8) | kUeWhole;
      else s_sliced = 1u;
    } else if (n[q] > kUeWarpMax) {
      plan->block[atomicAdd(&s_block, 1u)] = b;
    }
  }
  __syncthreads();
  if (s_sliced != 0) {
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const uint32_t b = tid + 1024 * q;
      if (b >= (uint32_t)kNBin || n[q] <= kUeSliceMean || n[q] > kUeBigMax) continue;
      const uint32_t slices = (n[q] + kUeSliceMean - 1) / kUeSliceMean;
      const bool whole = slices <= kUeWholeSlices && s_bins >= sms;
      const uint32_t count = whole ? 1u : slices;
      const uint32_t at = atomicAdd(&s_big, count);
      for (uint32_t k = 0; k < count; k++) big->item[at + k] = (b << 8) | (whole ? kUeWhole : k);
    }
    __syncthreads();
  }
  if (tid == 0) {
    plan->start[kNBin] = tot;
    ctl->n_general = s_general;
    ctl->n_block = s_block;
    ctl->n_big = s_big;
  }
}

// Records to their bins.  A block counts its clusters per bin in shared memory
// (each cluster's count is its place among the block's clusters of the bin),
// reserves the bins' ranges with one global atomic per bin, neighbouring bins
// by neighbouring lanes, and writes 16-byte records.  The order within a bin
// depends on the blocks' timing; the sort does not, because the record carries
// the input index.  Bound by L2 requests, of which every record is one.  Small
// tiles are best although they reserve more often: the records in flight have
// to meet their neighbours of a sector in L2, and tiles of 16384 spilled
// half-written sectors (427 us for 20 M clusters against 295 us with 2048).
// Reserving by the first cluster of each bin, without the pass over the
// counters, makes every reservation a request of its own: 442 us.
__global__ void __launch_bounds__(kUeScatThreads, 3) k_ue_scatter(UeArgs a, uint4* __restrict__ rec,
                                                                 UePlan* plan, UeCtl* ctl) {
  chain_wait();
  constexpr int T = kUeScatThreads;
  __shared__ __align__(16) uint32_t s_cnt[kNBin];
  const uint32_t tid = threadIdx.x;
  const uint32_t base = blockIdx.x * (uint32_t)(T * 4);
  const uint32_t cnt = min((uint32_t)(T * 4), a.n - base);
  const uint32_t l = tid * 4, i = base + l;
  const bool vec = a.vec && l + 4 <= cnt;
  uint32_t r = 0, s = 0, tm[4] = {}, pd[4] = {}, qt[4] = {}, qm[4] = {}, fl = 0, sp = 0, sg = 0;
  if (vec) {
    r = *reinterpret_cast<const uint32_t*>(a.row + i);
    s = *reinterpret_cast<const uint32_t*>(a.sector + i);
    const uint4 t = *reinterpret_cast<const uint4*>(a.time + i);
    const uint2 p = *reinterpret_cast<const uint2*>(a.pad + i);
    const uint2 x = *reinterpret_cast<const uint2*>(a.qtot + i);
    const uint2 y = *reinterpret_cast<const uint2*>(a.qmax + i);
    fl = *reinterpret_cast<const uint32_t*>(a.flags + i);
    sp = *reinterpret_cast<const uint32_t*>(a.sigp + i);
    sg = *reinterpret_cast<const uint32_t*>(a.sigt + i);
    tm[0] = t.x; tm[1] = t.y; tm[2] = t.z; tm[3] = t.w;
    pd[0] = p.x & 0xFFFFu; pd[1] = p.x >> 16; pd[2] = p.y & 0xFFFFu; pd[3] = p.y >> 16;
    qt[0] = x.x & 0xFFFFu; qt[1] = x.x >> 16; qt[2] = x.y & 0xFFFFu; qt[3] = x.y >> 16;
    qm[0] = y.x & 0xFFFFu; qm[1] = y.x >> 16; qm[2] = y.y & 0xFFFFu; qm[3] = y.y >> 16;
  } else {
#pragma unroll
    for (int q = 0; q < 4; q++)
      if (l + q < cnt) {
        r |= (uint32_t)a.row[i + q] << (8 * q);
        s |= (uint32_t)a.sector[i + q] << (8 * q);
        tm[q] = a.time[i + q];
        pd[q] = a.pad[i + q];
        qt[q] = a.qtot[i + q];
        qm[q] = a.qmax[i + q];
        fl |= (uint32_t)a.flags[i + q] << (8 * q);
        sp |= (uint32_t)a.sigp[i + q] << (8 * q);
        sg |= (uint32_t)a.sigt[i + q] << (8 * q);
      }
  }
  static_assert(kNBin % 4 == 0, "");
  for (int z = tid; z < kNBin / 4; z += T)
    reinterpret_cast<uint4*>(s_cnt)[z] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  uint32_t b[4], place[4], st = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    b[q] = ue_bin((r >> (8 * q)) & 255u, (s >> (8 * q)) & 255u, st);
    place[q] = l + q < cnt ? atomicAdd(&s_cnt[b[q]], 1u) : 0u;
  }
  __syncthreads();
  constexpr int Q = (kNBin + T - 1) / T;
  uint32_t c[Q];
#pragma unroll
  for (int q = 0; q < Q; q++) {
    const uint32_t k = tid + q * T;
    c[q] = k < (uint32_t)kNBin ? s_cnt[k] : 0u;
    if (c[q]) c[q] = atomicAdd(&plan->cursor[k], c[q]);
  }
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (tid + q * T < (uint32_t)kNBin) s_cnt[tid + q * T] = c[q];
  __syncthreads();
  bool wide = false;
#pragma unroll
  for (int q = 0; q < 4; q++)
    if (l + q < cnt) {
      wide |= (tm[q] >> 24) != 0;
      rec[s_cnt[b[q]] + place[q]] =
          make_uint4((tm[q] & 0xFFFFFFu) | ((fl >> (8 * q)) << 24),
                     pd[q] | (((sg >> (8 * q)) & 255u) << 16) | ((sp >> (8 * q)) << 24),
                     qm[q] | (qt[q] << 16), i + q);
    }
  if (__syncthreads_or(wide) && tid == 0) ctl->wide = 1u;
}

// The encoded cluster at output position p.
__device__ __forceinline__ void ue_emit(const UeArgs& a, uint32_t p, uint32_t pad_diff,
                                        uint32_t time_diff, const uint4& r) {
  a.pad_diff[p] = (uint16_t)pad_diff;
  a.time_diff[p] = time_diff;
  a.qtot_o[p] = (uint16_t)(r.z >> 16);
  a.qmax_o[p] = (uint16_t)r.z;
  a.flags_o[p] = (uint8_t)(r.x >> 24);
  a.sigp_o[p] = (uint8_t)(r.y >> 24);
  a.sigt_o[p] = (uint8_t)(r.y >> 16);
}

// (time, pad) of a record: 40 bits.
__device__ __forceinline__ uint64_t ue_key(uint32_t x, uint32_t y) {
  return ((uint64_t)(x & 0xFFFFFFu) << 16) | (y & 0xFFFFu);
}

// One warp per bin of up to kUeWarpMax clusters: every lane counts, for each
// of its records, the records that come before it.
__global__ void __launch_bounds__(256) k_ue_sort_warp(UeArgs a, const uint4* __restrict__ rec,
                                                     const UePlan* plan, const UeCtl* ctl) {
  chain_wait();
  constexpr int E = kUeWarpMax / 32;
  __shared__ uint4 s_rec[8][kUeWarpMax];
  __shared__ uint8_t s_ord[8][kUeWarpMax];
  const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t b = blockIdx.x * 8 + w;
  if (b >= (uint32_t)kNBin || ctl->wide) return;
  const uint32_t s0 = plan->start[b], n = plan->start[b + 1] - s0;
  if (n == 0 || n > kUeWarpMax) return;
  uint4 r[E];
  uint32_t rank[E];
#pragma unroll
  for (int u = 0; u < E; u++) {
    const uint32_t e = lane + 32 * u;
    rank[u] = 0;
    r[u] = e < n ? rec[s0 + e] : make_uint4(0, 0, 0, 0);
    if (e < n) s_rec[w][e] = r[u];
  }
  __syncwarp();
  const uint32_t eu = (n + 31) / 32;
  for (uint32_t j = 0; j < n; j++) {
    const uint4 o = s_rec[w][j];
    const uint64_t ko = ue_key(o.x, o.y);
#pragma unroll
    for (int u = 0; u < E; u++)
      if ((uint32_t)u < eu) {
        const uint64_t k = ue_key(r[u].x, r[u].y);
        rank[u] += (ko < k || (ko == k && o.w < r[u].w)) ? 1u : 0u;
      }
  }
#pragma unroll
  for (int u = 0; u < E; u++)
    if (lane + 32 * u < n) s_ord[w][rank[u]] = (uint8_t)(lane + 32 * u);
  __syncwarp();
  for (uint32_t q = lane; q < n; q += 32) {
    const uint4 v = s_rec[w][s_ord[w][q]];
    const uint4 o = q ? s_rec[w][s_ord[w][q - 1]] : make_uint4(0, 0, 0, 0);
    ue_emit(a, s0 + q, v.y - o.y, (v.x & 0xFFFFFFu) - (o.x & 0xFFFFFFu), v);
  }
}

// Buckets of a bin (or time slice): d is the distance of a cluster's leading
// 32 key bits (time, high byte of the pad) from the first one's, below width.
struct UeBuckets {
  uint32_t mul;  // 0: one bucket per value
  __device__ __forceinline__ void init(uint64_t width, uint32_t n_buckets) {
    // at most n_buckets / width * 2^32: the factor covers the three roundings
    mul = width <= n_buckets
              ? 0u
              : (uint32_t)(__fdividef((float)n_buckets * 4294967296.0f, (float)width) * 0.99999f);
  }
  __device__ __forceinline__ uint32_t of(uint32_t d) const { return mul ? __umulhi(d, mul) : d; }
};

// Insertion sort of one bucket's entries ((time, pad) << 24 | place in the
// bin); equal (time, pad) by input index.
__device__ __forceinline__ void ue_sort_bucket(uint64_t* k, uint32_t lo, uint32_t hi,
                                               const uint4* rec) {
  for (uint32_t i = lo + 1; i < hi; i++) {
    const uint64_t x = k[i];
    uint32_t j = i;
    while (j > lo) {
      const uint64_t y = k[j - 1];
      bool after = y > x;
      if ((y >> 24) == (x >> 24))
        after = rec[(uint32_t)y & 0xFFFFFFu].w > rec[(uint32_t)x & 0xFFFFFFu].w;
      if (!after) break;
      k[j] = y;
      j--;
    }
    k[j] = x;
  }
}

// Entry of a crowded bin or slice: (time, pad) and the input index, then the
// place in the bin -- no two are equal.
__device__ __forceinline__ void ue_put_whole(uint64_t* k, uint32_t* v, uint32_t i, const uint4& r,
                                             uint32_t place) {
  k[i] = (ue_key(r.x, r.y) << 24) | (r.w >> 8);
  v[i] = (r.w << 24) | place;
}

// Bitonic sort by the block of the entries put into [0, n), then the form that
// ue_emit_sorted reads.  Its time does not depend on the keys.
template <int B>
__device__ __forceinline__ void ue_sort_whole(uint64_t* k, uint32_t* v, uint32_t n) {
  const uint32_t size = n > 1 ? 1u << (32 - __clz(n - 1)) : 1u;
  for (uint32_t i = n + threadIdx.x; i < size; i += B) {
    k[i] = ~0ull;
    v[i] = ~0u;
  }
  __syncthreads();
  for (uint32_t len = 2; len <= size; len <<= 1)
    for (uint32_t j = len >> 1; j > 0; j >>= 1) {
      for (uint32_t t = threadIdx.x; t < size / 2; t += B) {
        const uint32_t a = ((t & ~(j - 1)) << 1) | (t & (j - 1)), b = a | j;
        const uint64_t ka = k[a], kb = k[b];
        const uint32_t va = v[a], vb = v[b];
        const bool greater = ka > kb || (ka == kb && va > vb);
        if (greater == ((a & len) == 0)) {
          k[a] = kb;
          k[b] = ka;
          v[a] = vb;
          v[b] = va;
        }
      }
      __syncthreads();
    }
  for (uint32_t i = threadIdx.x; i < n; i += B)
    k[i] = (k[i] & ~0xFFFFFFull) | (v[i] & 0xFFFFFFu);
  __syncthreads();
}

// Streams of n sorted entries from output position p0; prev is the entry
// before the first (0: none, differences to zero).
template <int B>
__device__ __forceinline__ void ue_emit_sorted(const UeArgs& a, uint32_t p0, uint32_t n,
                                               const uint64_t* k, uint64_t prev,
                                               const uint4* __restrict__ rec) {
#pragma unroll 2
  for (uint32_t q = threadIdx.x; q < n; q += B) {
    const uint64_t x = k[q], y = q ? k[q - 1] : prev;
    const uint4 r = rec[(uint32_t)x & 0xFFFFFFu];
    ue_emit(a, p0 + q, (uint32_t)(x >> 24) - (uint32_t)(y >> 24),
            (uint32_t)(x >> 40) - (uint32_t)(y >> 40), r);
  }
}

__device__ __forceinline__ void ue_mark_general(UeCtl* ctl, uint32_t b) {
  if (atomicExch(&ctl->general[b], 1u) == 0u) atomicAdd(&ctl->n_general, 1u);
}

// Smallest and largest value over the block, through s (2 x 32 words).
__device__ __forceinline__ void ue_minmax(uint32_t& lo, uint32_t& hi, uint32_t* s, int warps) {
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t lane = threadIdx.x & 31;
  if (lane == 0) {
    s[threadIdx.x >> 5] = lo;
    s[32 + (threadIdx.x >> 5)] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, lane < (uint32_t)warps ? s[lane] : 0xFFFFFFFFu);
  hi = __reduce_max_sync(0xffffffffu, lane < (uint32_t)warps ? s[32 + lane] : 0u);
}

// Blocks take the listed bins in turn.  A thread keeps its eight clusters'
// keys in registers; their records are read again, from the caches, when the
// sorted streams are written.
__global__ void __launch_bounds__(kUeBlockThreads, 3) k_ue_sort_block(UeArgs a, const uint4* rec,
                                                                     const UePlan* plan,
                                                                     UeCtl* ctl) {
  chain_wait();
  constexpr int T = kUeBlockThreads, E = kUeBlockMax / T;
  extern __shared__ uint64_t s_dyn[];
  uint64_t* s_key = s_dyn;                                            // kUeBlockMax
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_dyn + kUeBlockMax);  // kUeBlockMax
  __shared__ uint32_t s_task, s_mm[64];
  const uint32_t tid = threadIdx.x;
  const uint32_t n_list = ctl->wide ? 0u : ctl->n_block;
  for (;;) {
    if (tid == 0) s_task = atomicAdd(&ctl->next_block, 1u);
    __syncthreads();
    const uint32_t task = s_task;
    if (task >= n_list) break;
    const uint32_t b = plan->block[task];
    const uint32_t s0 = plan->start[b], n = plan->start[b + 1] - s0;
    const uint4* __restrict__ r0 = rec + s0;
    uint2 w[E];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int u = 0; u < E; u++) {
      const uint32_t e = tid + u * T;
      if (e < n) w[u] = *reinterpret_cast<const uint2*>(r0 + e);
    }
#pragma unroll
    for (int u = 0; u < E; u++) s_cnt[tid + u * T] = 0u;
#pragma unroll
    for (int u = 0; u < E; u++)
      if (tid + u * T < n) {
        const uint32_t d = (w[u].x << 8) | ((w[u].y >> 8) & 255u);
        lo = min(lo, d);
        hi = max(hi, d);
      }
    ue_minmax(lo, hi, s_mm, T / 32);
    UeBuckets bk;
    bk.init((uint64_t)(hi - lo) + 1, n);
    uint32_t br[E];
#pragma unroll
    for (int u = 0; u < E; u++)
      if (tid + u * T < n) {
        const uint32_t d = (w[u].x << 8) | ((w[u].y >> 8) & 255u);
        const uint32_t k = bk.of(d - lo);
        br[u] = k | (atomicAdd(&s_cnt[k], 1u) << 16);
      }
    __syncthreads();
    // first entry of every bucket, E consecutive buckets per thread
    uint32_t c[E], sum = 0, most = 0, tot;
#pragma unroll
    for (int u = 0; u < E; u++) {
      c[u] = s_cnt[tid * E + u];
      sum += c[u];
      most = max(most, c[u]);
    }
    uint32_t run = ue_scan<T>(sum, tot);
#pragma unroll
    for (int u = 0; u < E; u++) {
      s_cnt[tid * E + u] = run;
      run += c[u];
    }
    if (__syncthreads_or(most > kUeBucketMax)) {
      if (tid == 0) ue_mark_general(ctl, b);
      continue;
    }
#pragma unroll
    for (int u = 0; u < E; u++)
      if (tid + u * T < n)
        s_key[s_cnt[br[u] & 0xFFFFu] + (br[u] >> 16)] =
            (ue_key(w[u].x, w[u].y) << 24) | (tid + u * T);
    __syncthreads();
    for (uint32_t k = tid; k < n; k += T) {
      const uint32_t k0 = s_cnt[k], k1 = k + 1 < n ? s_cnt[k + 1] : n;
      if (k1 > k0 + 1) ue_sort_bucket(s_key, k0, k1, r0);
    }
    __syncthreads();
    ue_emit_sorted<T>(a, s0, n, s_key, 0ull, r0);
  }
}

// Larger bins: cut into equal time slices of about kUeSliceMean clusters, which
// large blocks sort: all of a bin, one slice after the other, or a slice each.  A
// block reads its whole bin, from L2, for the first and last time and twice per
// slice: to count its clusters per bucket (and those before it, where the block has
// not sorted them itself), and to pick them out.  A single bin of 100, 131 and 262 k
// clusters takes 0.13, 0.15 and 0.22 ms by slices, 0.56, 0.80 and 2.41 ms as a whole.
// With a bin for every block, bins of up to kUeWholeSlices slices are the faster as a
// whole (152 of 20 k: 146 against 158 us; 547 of 40 k: 1.03 against 1.07 ms), larger
// ones by slices (152 of 50 k: 0.40 against 0.44 ms; 300 of 60 k: 0.90 against 1.05).
__global__ void __launch_bounds__(kUeBigThreads, 1) k_ue_sort_big(UeArgs a, const uint4* rec,
                                                                 const UePlan* plan,
                                                                 const UeBig* big, UeCtl* ctl) {
  chain_wait();
  constexpr int T = kUeBigThreads, E = kUeSliceCap / T;
  extern __shared__ uint64_t s_dyn[];
  uint64_t* s_key = s_dyn;                                            // kUeSliceCap
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_dyn + kUeSliceCap);  // kUeSliceCap
  __shared__ uint32_t s_task, s_mm[64], s_before, s_at;
  __shared__ unsigned long long s_last;
  const uint32_t tid = threadIdx.x;
  const uint32_t n_list = ctl->wide ? 0u : ctl->n_big;
  auto lead = [](const uint2& w) { return (w.x << 8) | ((w.y >> 8) & 255u); };
  for (;;) {
    if (tid == 0) {
      s_task = atomicAdd(&ctl->next_big, 1u);
      s_before = 0u;
      s_last = 0ull;
    }
    __syncthreads();
    const uint32_t task = s_task;
    if (task >= n_list) break;
    const uint32_t b = big->item[task] >> 8, part = big->item[task] & 255u;
    const uint32_t s0 = plan->start[b], n = plan->start[b + 1] - s0;
    const uint4* __restrict__ r0 = rec + s0;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll 4
    for (uint32_t e = tid; e < n; e += T) {
      const uint32_t d = lead(*reinterpret_cast<const uint2*>(r0 + e));
      lo = min(lo, d);
      hi = max(hi, d);
    }
    ue_minmax(lo, hi, s_mm, T / 32);
    const uint32_t slices = (n + kUeSliceMean - 1) / kUeSliceMean;
    const uint64_t width = (uint64_t)(hi - lo) / slices + 1;
    UeBuckets bk;
    bk.init(width, kUeSliceCap);
    const bool whole = part == kUeWhole;
    const uint32_t s_end = whole ? slices : part + 1;
    uint32_t out = 0;    // clusters before the slice
    uint64_t prev = 0ull;  // the last of them
    for (uint32_t s = whole ? 0u : part; s < s_end && out < n; s++) {
      const uint64_t first = (uint64_t)lo + s * width;
      if (first > hi) break;  // nothing there, nor after it
      const uint32_t d0 = (uint32_t)first, d1 = (uint32_t)min(first + width - 1, (uint64_t)hi);
#pragma unroll
      for (int u = 0; u < E; u++) s_cnt[tid + u * T] = 0u;
      if (tid == 0) s_at = 0u;
      __syncthreads();
      if (whole || s == 0) {
#pragma unroll 4
        for (uint32_t e = tid; e < n; e += T) {
          const uint32_t d = lead(*reinterpret_cast<const uint2*>(r0 + e));
          if (d >= d0 && d <= d1) atomicAdd(&s_cnt[bk.of(d - d0)], 1u);
        }
      } else {
        uint32_t before = 0;
        uint64_t last = 0;
#pragma unroll 4
        for (uint32_t e = tid; e < n; e += T) {
          const uint2 w = *reinterpret_cast<const uint2*>(r0 + e);
          const uint32_t d = lead(w);
          if (d < d0) {
            before++;
            last = max(last, ue_key(w.x, w.y));
          } else if (d <= d1) {
            atomicAdd(&s_cnt[bk.of(d - d0)], 1u);
          }
        }
        before = __reduce_add_sync(0xffffffffu, before);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        if ((tid & 31) == 0 && before) {
          atomicAdd(&s_before, before);
          atomicMax(&s_last, (unsigned long long)last);
        }
      }
      __syncthreads();
      if (!whole) {
        out = s_before;
        prev = (uint64_t)s_last << 24;
      }
      uint32_t c[E], sum = 0, most = 0, m;
#pragma unroll
      for (int u = 0; u < E; u++) {
        c[u] = s_cnt[tid * E + u];
        sum += c[u];
        most = max(most, c[u]);
      }
      uint32_t run = ue_scan<T>(sum, m);
      if (m > kUeSliceCap) {  // the same for every thread
        if (tid == 0) ue_mark_general(ctl, b);
        break;  // the general sort writes the whole bin
      }
#pragma unroll
      for (int u = 0; u < E; u++) {
        s_cnt[tid * E + u] = run;
        run += c[u];
      }
      if (__syncthreads_or(most > kUeBucketMax)) {
        for (uint32_t e = tid; e < n; e += T) {
          const uint4 w = r0[e];
          const uint32_t d = lead(make_uint2(w.x, w.y));
          if (d >= d0 && d <= d1) ue_put_whole(s_key, s_cnt, atomicAdd(&s_at, 1u), w, e);
        }
        ue_sort_whole<T>(s_key, s_cnt, m);
      } else {
#pragma unroll 4
        for (uint32_t e = tid; e < n; e += T) {
          const uint2 w = *reinterpret_cast<const uint2*>(r0 + e);
          const uint32_t d = lead(w);
          if (d >= d0 && d <= d1)
            s_key[atomicAdd(&s_cnt[bk.of(d - d0)], 1u)] = (ue_key(w.x, w.y) << 24) | e;
        }
        __syncthreads();  // s_cnt[k] is now the end of bucket k
#pragma unroll 1
        for (uint32_t k = tid; k < kUeSliceCap; k += T) {
          const uint32_t k0 = k ? s_cnt[k - 1] : 0u, k1 = s_cnt[k];
          if (k1 > k0 + 1) ue_sort_bucket(s_key, k0, k1, r0);
        }
        __syncthreads();
      }
      ue_emit_sorted<T>(a, s0 + out, m, s_key, prev, r0);
      if (m) prev = s_key[m - 1];
      out += m;
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------
// General sort: a stable radix sort, 8 bits per pass, least significant first,
// by one cooperative launch.  Its clusters are taken in input order, so that
// ties need no digits of their own, and the key holds only the bits in which
// they differ: rank of the bin among the sorted ones, time - first time, pad.
// ---------------------------------------------------------------------------
struct RsKeys {
  uint64_t* key;
  uint32_t* idx;
};

// Clusters of a tile: warp w takes [256 w, 256 w + 256) in steps of 32.
__device__ __forceinline__ uint32_t rs_place(int u) {
  return (threadIdx.x >> 5) * (32u * kRsPerThread) + 32u * u + (threadIdx.x & 31);
}

__device__ __forceinline__ void rs_upsweep(const uint64_t* key, uint32_t m, uint32_t tile,
                                           uint32_t n_tiles, int shift, uint32_t* counts,
                                           uint32_t* s_c) {
  s_c[threadIdx.x] = 0u;
  __syncthreads();
  const uint32_t base = tile * kRsTile;
  uint64_t k[kRsPerThread];
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++) {
    const uint32_t l = u * kRsThreads + threadIdx.x;
    k[u] = l < m - base ? __ldcg(key + base + l) : 0ull;
  }
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++)
    if (u * kRsThreads + threadIdx.x < m - base)
      atomicAdd(&s_c[(uint32_t)(k[u] >> shift) & 255u], 1u);
  __syncthreads();
  counts[(size_t)threadIdx.x * n_tiles + tile] = s_c[threadIdx.x];
  __syncthreads();
}

// Exclusive sums of n counts in place, by one block; returns the total.
__device__ __forceinline__ uint32_t rs_scan_row(uint32_t* c, uint32_t n) {
  constexpr uint32_t E = 8;
  uint32_t run = 0;
  for (uint64_t t0 = 0; t0 < n; t0 += E * kRsThreads) {
    const uint64_t t = t0 + E * threadIdx.x;
    uint32_t v[E], sum = 0, tot;
#pragma unroll
    for (uint32_t q = 0; q < E; q++) {
      v[q] = t + q < n ? __ldcg(c + t + q) : 0u;
      sum += v[q];
    }
    uint32_t at = run + ue_scan<kRsThreads>(sum, tot);
#pragma unroll
    for (uint32_t q = 0; q < E; q++) {
      if (t + q < n) c[t + q] = at;
      at += v[q];
    }
    run += tot;
  }
  return run;
}

// A tile on chip: its entries in digit order, and by digit its first position in
// the output minus its first place in the tile.
struct RsTile {
  uint64_t key[kRsTile];
  uint32_t idx[kRsTile];
};

// Stable scatter of one tile, through shared memory: an entry's place in the tile
// is its digit's first place plus the entries of that digit in the tile's earlier
// warps and earlier steps and lanes; then neighbouring threads write neighbouring
// places, runs of about eight entries (written straight from the ranking threads,
// two requests to L2 per entry: 4.38 against 3.31 ms for 20 M clusters of times of
// 2^24 and more).
__device__ __forceinline__ void rs_downsweep(RsKeys src, RsKeys dst, uint32_t m, uint32_t tile,
                                             uint32_t n_tiles, int shift, const uint32_t* counts,
                                             const uint32_t* s_base, uint32_t* s_off,
                                             uint32_t (*s_wc)[256], RsTile& S) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) (&s_wc[0][0])[i] = 0u;
  const uint32_t base = tile * kRsTile, left = min(m - base, kRsTile);
  uint64_t key[kRsPerThread];
  uint32_t idx[kRsPerThread], rk[kRsPerThread];
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++) {
    const uint32_t l = rs_place(u);
    key[u] = l < left ? __ldcg(src.key + base + l) : 0ull;
    idx[u] = l < left ? __ldcg(src.idx + base + l) : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++) {
    const bool in = rs_place(u) < left;
    const uint32_t act = __ballot_sync(0xffffffffu, in);
    rk[u] = 0;
    if (in) {
      const uint32_t d = (uint32_t)(key[u] >> shift) & 255u;
      const uint32_t peers = __match_any_sync(act, d);
      rk[u] = s_wc[w][d] + __popc(peers & lanemask_lt());
      __syncwarp(act);
      if (lane == __ffs(peers) - 1) s_wc[w][d] += __popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  {  // per digit: first place in the tile, then the earlier warps' entries
    const uint32_t d = threadIdx.x;
    uint32_t c[kRsWarps], sum = 0, tot;
#pragma unroll
    for (int ww = 0; ww < kRsWarps; ww++) sum += c[ww] = s_wc[ww][d];
    uint32_t run = ue_scan<kRsThreads>(sum, tot);
    s_off[d] = s_base[d] + __ldcg(counts + (size_t)d * n_tiles + tile) - run;
#pragma unroll
    for (int ww = 0; ww < kRsWarps; ww++) {
      s_wc[ww][d] = run;
      run += c[ww];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++)
    if (rs_place(u) < left) {
      const uint32_t l = s_wc[w][(uint32_t)(key[u] >> shift) & 255u] + rk[u];
      S.key[l] = key[u];
      S.idx[l] = idx[u];
    }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kRsPerThread; u++) {
    const uint32_t l = u * kRsThreads + threadIdx.x;
    if (l < left) {
      const uint64_t k = S.key[l];
      const uint32_t p = s_off[(uint32_t)(k >> shift) & 255u] + l;
      dst.key[p] = k;
      dst.idx[p] = S.idx[l];
    }
  }
  __syncthreads();
}

// Bits of the values 0 .. top.
__device__ __forceinline__ int rs_bits(uint32_t top) { return 32 - __clz(top); }

union GeneralSmem {
  struct {
    union {
      // rank: of the bins to sort, the others kNone; delta: by rank, output
      // position minus place among the sorted
      struct {
        uint16_t rank[kNBin];
        uint32_t delta[kNBin];
      } bins;
      RsTile tile;
    };
    uint32_t wc[kRsWarps][256];
    uint32_t base[256], off[256];
  };
  struct {
    uint64_t key[kUeBlockMax];
    uint32_t v[kUeBlockMax];
  } whole;
};

__global__ void __launch_bounds__(kRsThreads, 3) k_ue_general(UeArgs a, uint4* r0, uint4* r1,
                                                          const UePlan* plan, UeCtl* ctl,
                                                          uint32_t* counts, uint32_t* digit_tot) {
  const bool wide = ctl->wide != 0u;
  if (!wide && ctl->n_general == 0u) return;  // the same for every block
  extern __shared__ uint64_t s_dyn[];
  GeneralSmem& S = *reinterpret_cast<GeneralSmem*>(s_dyn);
  constexpr uint16_t kNone = 0xFFFFu;
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t gid = blockIdx.x * kRsThreads + tid, gn = gridDim.x * kRsThreads;
  uint32_t target = 0, m, n_bins;
  auto plan_bins = [&] {
    constexpr uint32_t Q = (kNBin + kRsThreads - 1) / kRsThreads;
    uint32_t cnt[Q], sum = 0, some = 0;
#pragma unroll
    for (uint32_t q = 0; q < Q; q++) {
      const uint32_t b = tid * Q + q;
      cnt[q] = b < (uint32_t)kNBin && (wide || ctl->general[b]) ? plan->start[b + 1] - plan->start[b]
                                                                : 0u;
      if (!wide && cnt[q] <= kUeBlockMax) cnt[q] = 0u;  // done
      sum += cnt[q];
      some += cnt[q] != 0;
    }
    uint32_t first = ue_scan<kRsThreads>(sum, m), rank = ue_scan<kRsThreads>(some, n_bins);
#pragma unroll
    for (uint32_t q = 0; q < Q; q++) {
      const uint32_t b = tid * Q + q;
      if (b >= (uint32_t)kNBin) break;
      S.bins.rank[b] = cnt[q] ? (uint16_t)rank : kNone;
      if (cnt[q]) S.bins.delta[rank++] = plan->start[b] - first;
      first += cnt[q];
    }
    __syncthreads();
  };
  if (!wide)  // crowded bins of k_ue_sort_block, as a whole
    for (uint32_t b = blockIdx.x; b < (uint32_t)kNBin; b += gridDim.x) {
      const uint32_t s0 = plan->start[b], n = plan->start[b + 1] - s0;
      if (!ctl->general[b] || n > kUeBlockMax) continue;
      const uint4* rec = r0 + s0;
      for (uint32_t e = tid; e < n; e += kRsThreads)
        ue_put_whole(S.whole.key, S.whole.v, e, rec[e], e);
      ue_sort_whole<kRsThreads>(S.whole.key, S.whole.v, n);
      ue_emit_sorted<kRsThreads>(a, s0, n, S.whole.key, 0ull, rec);
      __syncthreads();
    }
  plan_bins();
  if (m == 0) return;  // the same for every block
  auto rank_of = [&](uint32_t i) {
    uint32_t st = 0;
    return S.bins.rank[ue_bin(a.row[i], a.sector[i], st)];
  };
  // Ranges of time and pad; clusters to sort per input tile.
  const bool all = m == a.n;
  const uint32_t in_tiles = a.n / kRsTile + (a.n % kRsTile != 0);
  uint32_t not_tmin = 0, tmax = 0, pmax = 0;
  for (uint32_t t = blockIdx.x; t < in_tiles; t += gridDim.x) {
    const uint32_t base = t * kRsTile, left = a.n - base;
    uint32_t mine = 0;
#pragma unroll
    for (int u = 0; u < kRsPerThread; u++) {
      const uint32_t l = rs_place(u);
      if (l < left && (all || rank_of(base + l) != kNone)) {
        const uint32_t time = a.time[base + l];
        not_tmin = max(not_tmin, ~time);
        tmax = max(tmax, time);
        pmax = max(pmax, (uint32_t)a.pad[base + l]);
        mine++;
      }
    }
    if (all) continue;
    uint32_t tot;
    ue_scan<kRsThreads>(mine, tot);
    if (tid == 0) counts[t] = tot;
  }
  not_tmin = __reduce_max_sync(0xffffffffu, not_tmin);
  tmax = __reduce_max_sync(0xffffffffu, tmax);
  pmax = __reduce_max_sync(0xffffffffu, pmax);
  if (lane == 0 && (not_tmin || tmax || pmax)) {
    atomicMax(&ctl->not_tmin, not_tmin);
    atomicMax(&ctl->tmax, tmax);
    atomicMax(&ctl->pmax, pmax);
  }
  bool ok = grid_barrier(&ctl->barrier, target);
  if (ok && !all) {
    if (blockIdx.x == 0) rs_scan_row(counts, in_tiles);
    ok = grid_barrier(&ctl->barrier, target);
  }
  const uint32_t tmin = ~__ldcg(&ctl->not_tmin);
  const int pad_bits = rs_bits(__ldcg(&ctl->pmax));
  const int low_bits = pad_bits + rs_bits(__ldcg(&ctl->tmax) - tmin);
  const int bits = low_bits + rs_bits(n_bins - 1);  // at most 13 + 32 + 16
  RsKeys src{reinterpret_cast<uint64_t*>(r1), reinterpret_cast<uint32_t*>(r1) + 2 * (size_t)a.n};
  RsKeys dst{reinterpret_cast<uint64_t*>(r0), reinterpret_cast<uint32_t*>(r0) + 2 * (size_t)a.n};
  for (uint32_t t = blockIdx.x; t < in_tiles && ok; t += gridDim.x) {
    const uint32_t base = t * kRsTile, left = a.n - base;
    uint32_t rank[kRsPerThread], mask[kRsPerThread], before = 0;
#pragma unroll
    for (int u = 0; u < kRsPerThread; u++) {
      const uint32_t l = rs_place(u);
      rank[u] = l < left ? rank_of(base + l) : kNone;
      mask[u] = __ballot_sync(0xffffffffu, rank[u] != kNone);
      before += __popc(mask[u]);
    }
    // place of the warp's first cluster; with all of them, places are inputs
    uint32_t at = base + w * (32u * kRsPerThread);
    if (!all) {
      uint32_t tot;
      const uint32_t e = ue_scan<kRsThreads>(lane == 0 ? before : 0u, tot);
      at = __ldcg(counts + t) + __shfl_sync(0xffffffffu, e, 0);
    }
#pragma unroll
    for (int u = 0; u < kRsPerThread; u++) {
      const uint32_t i = base + rs_place(u);
      if (rank[u] != kNone) {
        const uint32_t p = at + __popc(mask[u] & lanemask_lt());
        src.key[p] = ((uint64_t)rank[u] << low_bits) |
                     ((uint64_t)(a.time[i] - tmin) << pad_bits) | a.pad[i];
        src.idx[p] = i;
      }
      at += __popc(mask[u]);
    }
  }
  if (ok) ok = grid_barrier(&ctl->barrier, target);
  const uint32_t n_tiles = m / kRsTile + (m % kRsTile != 0);
  for (int shift = 0; shift < bits && ok; shift += 8) {
    for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x)
      rs_upsweep(src.key, m, t, n_tiles, shift, counts, S.base);
    if (!(ok = grid_barrier(&ctl->barrier, target))) break;
    for (uint32_t d = blockIdx.x; d < 256; d += gridDim.x) {
      const uint32_t tot = rs_scan_row(counts + (size_t)d * n_tiles, n_tiles);
      if (tid == 0) digit_tot[d] = tot;
    }
    if (!(ok = grid_barrier(&ctl->barrier, target))) break;
    uint32_t tot;
    const uint32_t e = ue_scan<kRsThreads>(__ldcg(digit_tot + tid), tot);
    S.base[tid] = e;
    for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x)
      rs_downsweep(src, dst, m, t, n_tiles, shift, counts, S.base, S.off, S.wc, S.tile);
    const RsKeys x = src;
    src = dst;
    dst = x;
    ok = grid_barrier(&ctl->barrier, target);
  }
  if (!ok) {
    if (tid == 0) atomicOr(a.status, kStTimeout);
    return;
  }
  plan_bins();
  for (uint64_t q = gid; q < m; q += gn) {
    const uint64_t x = __ldcg(src.key + q), y = q ? __ldcg(src.key + q - 1) : ~0ull;
    const bool same = q && x >> low_bits == y >> low_bits;
    auto pad_of = [&](uint64_t k) { return (uint32_t)k & ((1u << pad_bits) - 1u); };
    auto time_of = [&](uint64_t k) {
      return (uint32_t)((k & ((1ull << low_bits) - 1ull)) >> pad_bits) + tmin;
    };
    const uint32_t p = (uint32_t)q + S.bins.delta[(uint32_t)(x >> low_bits)];
    const uint32_t i = __ldcg(src.idx + q);
    a.pad_diff[p] = (uint16_t)(pad_of(x) - (same ? pad_of(y) : 0u));
    a.time_diff[p] = time_of(x) - (same ? time_of(y) : 0u);
    a.qtot_o[p] = a.qtot[i];
    a.qmax_o[p] = a.qmax[i];
    a.flags_o[p] = a.flags[i];
    a.sigp_o[p] = a.sigp[i];
    a.sigt_o[p] = a.sigt[i];
  }
}

constexpr size_t kUeBlockSmem = (size_t)kUeBlockMax * 12;
constexpr size_t kUeBigSmem = (size_t)kUeSliceCap * 12;

}  // namespace

cudaError_t prepare_unatt_encode(int* blocks_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_ue_sort_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kUeBlockSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_ue_sort_big, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kUeBigSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_ue_general, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(GeneralSmem));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_ue_general, kRsThreads,
                                                      sizeof(GeneralSmem));
  return e;
}

}  // namespace tmd

using namespace tmd;

extern "C" int tmd_encode_unattached(tmd_handle* h, const tmd_unatt_truth_in* in,
                                     const tmd_unatt_out* out, void* stream) {
  if (!h) return TMD_ERR_ARG;
  if (!in || !out) return tmd_set_error(h, TMD_ERR_ARG, "null descriptor");
  const uint32_t n = in->n;
  if (!out->n_unatt || !out->status)
    return tmd_set_error(h, TMD_ERR_ARG, "n_unatt and status are required");
  const void* need[] = {in->row,     in->sector,      in->pad,       in->time,       in->qtot,
                        in->qmax,    in->flags,       in->sigma_pad, in->sigma_time, out->pad_diff_u,
                        out->time_diff_u, out->qtot_u, out->qmax_u,  out->flags_u,   out->sigma_pad_u,
                        out->sigma_time_u};
  for (const void* p : need)
    if (n && !p) return tmd_set_error(h, TMD_ERR_ARG, "per-cluster array is NULL");
  auto mis = [](const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) != 0; };
  if (mis(in->pad, 2) || mis(in->time, 4) || mis(in->qtot, 2) || mis(in->qmax, 2) ||
      mis(out->pad_diff_u, 2) || mis(out->time_diff_u, 4) || mis(out->qtot_u, 2) ||
      mis(out->qmax_u, 2) || mis(out->n_unatt, 4) || mis(out->status, 4))
    return tmd_set_error(h, TMD_ERR_ARG, "array not aligned to its element size");
  int rc = tmd_cuda_check(h, cudaSetDevice(h->device), "cudaSetDevice");
  if (rc != TMD_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const uint32_t n_tiles = n / kRsTile + 1;
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t o_r0 = 0, o_r1 = up((size_t)n * 16 + 16), o_cnt = o_r1 + up((size_t)n * 16 + 16),
               o_dig = o_cnt + up((size_t)256 * n_tiles * 4), o_plan = o_dig + up(256 * 4),
               o_ctl = o_plan + up(sizeof(UePlan)), o_big = o_ctl + up(sizeof(UeCtl)),
               total = o_big + up(sizeof(UeBig));
  if ((rc = h->ensure_scratch(total)) != TMD_OK) return rc;
  bool order = false;
  if ((rc = h->order_after_previous(st, &order)) != TMD_OK) return rc;
  char* base = static_cast<char*>(h->scratch);
  uint4* r0 = reinterpret_cast<uint4*>(base + o_r0);
  uint4* r1 = reinterpret_cast<uint4*>(base + o_r1);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(base + o_cnt);
  uint32_t* dig = reinterpret_cast<uint32_t*>(base + o_dig);
  UePlan* plan = reinterpret_cast<UePlan*>(base + o_plan);
  UeCtl* ctl = reinterpret_cast<UeCtl*>(base + o_ctl);
  UeBig* big = reinterpret_cast<UeBig*>(base + o_big);
  UeArgs a;
  a.n = n;
  a.row = in->row; a.sector = in->sector; a.pad = in->pad; a.time = in->time;
  a.qtot = in->qtot; a.qmax = in->qmax; a.flags = in->flags; a.sigp = in->sigma_pad;
  a.sigt = in->sigma_time;
  a.n_unatt = out->n_unatt; a.pad_diff = out->pad_diff_u; a.time_diff = out->time_diff_u;
  a.qtot_o = out->qtot_u; a.qmax_o = out->qmax_u; a.flags_o = out->flags_u;
  a.sigp_o = out->sigma_pad_u; a.sigt_o = out->sigma_time_u; a.status = out->status;
  a.vec = !(mis(a.row, 4) || mis(a.sector, 4) || mis(a.flags, 4) || mis(a.sigp, 4) ||
            mis(a.sigt, 4) || mis(a.pad, 8) || mis(a.qtot, 8) || mis(a.qmax, 8) || mis(a.time, 16));
  const uint32_t sms = (uint32_t)h->sms;
  k_ue_init<<<(sizeof(UeCtl) / 4 + 255) / 256, 256, 0, st>>>(a, ctl);
  if (n) {
    launch_chained(k_ue_count, std::min(2 * sms, n / 8192 + 1), 1024, 0, st, a);
    launch_chained(k_ue_plan, 1, 1024, 0, st, a, plan, big, ctl, sms);
    launch_chained(k_ue_scatter, n / (kUeScatThreads * 4) + (n % (kUeScatThreads * 4) != 0),
                   kUeScatThreads, 0, st, a, r0, plan, ctl);
    launch_chained(k_ue_sort_warp, (kNBin + 7) / 8, 256, 0, st, a, r0, plan, ctl);
    if (n > kUeWarpMax)
      launch_chained(k_ue_sort_block, std::min(3 * sms, n / kUeWarpMax), kUeBlockThreads,
                     kUeBlockSmem, st, a, r0, plan, ctl);
    if (n > kUeBlockMax)
      launch_chained(k_ue_sort_big, std::min(sms, n / kUeBlockMax), kUeBigThreads, kUeBigSmem, st,
                     a, r0, plan, big, ctl);
    void* args[] = {&a, &r0, &r1, &plan, &ctl, &cnt, &dig};
    const uint32_t grid = std::min(n_tiles, sms * (uint32_t)h->occ_ue);
    rc = tmd_cuda_check(h, cudaLaunchCooperativeKernel((const void*)k_ue_general, dim3(grid),
                                                       dim3(kRsThreads), args, sizeof(GeneralSmem), st),
                        "general sort launch");
    if (rc != TMD_OK) return rc;
  }
  rc = tmd_cuda_check(h, cudaGetLastError(), "unattached encoder launch");
  if (rc != TMD_OK) return rc;
  return h->mark_scratch_done(st, order);
}
