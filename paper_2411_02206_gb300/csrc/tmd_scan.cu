// tmd_scan.cu -- track preparation and row offsets of the decoder.
//
// Track preparation (replaces the CPU-precomputed SoA indices of Sec. 4 of
// arXiv:2411.02206 with device scans): trackStart = exclusive scan of the
// track lengths, and a decode order with the longest tracks first (bucketed by
// length), so that warps of the persistent decoder take similar tracks and
// the tail is short.
//
// Row offsets: per (sector,row) bin the attached count (summed from the
// per-tile histograms of k_count_rank) plus the unattached count, exclusive
// scan -> rowStart; then per (tile, bin) the first native index of the tile's
// clusters in that bin.
#include <cstring>

#include "tmd_internal.cuh"

namespace tmd {

// Exclusive scan over a block of B threads: returns the exclusive prefix of v
// and sets total to the block total (all threads).
template <int B>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t& total) {
  __shared__ uint32_t warp_tot[B / 32];
  __shared__ uint32_t block_tot;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    const uint32_t t = lane < B / 32 ? warp_tot[lane] : 0u;
    uint32_t s = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < B / 32) warp_tot[lane] = s - t;
    if (lane == 31) block_tot = s;
  }
  __syncthreads();
  const uint32_t r = warp_tot[w] + x - v;
  total = block_tot;
  __syncthreads();
  return r;
}

// The launch record (frame descriptors and prefix tables) travels to the
// device as the parameter of this kernel, not by a host-to-device copy: a
// copy would queue on the copy engine behind whatever bulk uploads other
// streams have in flight (the pipelined host entry point uploads the next
// frame's inputs while this one decodes), and the decode would wait for them.
// The same launch clears the scratch region that must start at zero.
// With n_status > 0 the chunk holds the n_status frame descriptors at byte
// offset frames_off, and the launch also clears their status words (the
// chain's first write to them).
template <int W>
__global__ void k_put_record(RecordChunk<W> c, uint32_t n16, uint4* __restrict__ dst,
                             uint4* __restrict__ zero, uint32_t zero_n16, uint32_t frames_off,
                             uint32_t n_status) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride) dst[i] = c.w[i];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < zero_n16; i += stride)
    zero[i] = make_uint4(0u, 0u, 0u, 0u);
  if (blockIdx.x == 0) {
    const FrameDev* fd =
        reinterpret_cast<const FrameDev*>(reinterpret_cast<const char*>(c.w) + frames_off);
    for (uint32_t f = threadIdx.x; f < n_status; f += blockDim.x) *fd[f].status = 0u;
  }
}

bool put_record_zeroes_status(size_t frames_off, uint32_t n_frames) {
  return frames_off + (size_t)n_frames * sizeof(FrameDev) <= sizeof(RecordChunk<kRecordChunkBig>);
}

cudaError_t put_record(const void* host, size_t bytes, void* dev, void* zero, size_t zero_bytes,
                       cudaStream_t st, size_t frames_off, uint32_t n_status) {
  const char* h = static_cast<const char*>(host);
  char* d = static_cast<char*>(dev);
  uint4* z = static_cast<uint4*>(zero);
  uint32_t zn = (uint32_t)(zero_bytes / 16);
  do {
    const size_t small = sizeof(RecordChunk<kRecordChunkSmall>);
    const size_t big = sizeof(RecordChunk<kRecordChunkBig>);
    const size_t take = bytes <= small ? bytes : (bytes < big ? bytes : big);
    const uint32_t n16 = (uint32_t)(take / 16);
    const uint32_t work = n16 > zn ? n16 : zn;
    uint32_t grid = (work + 255) / 256;
    grid = grid < 1 ? 1 : (grid > 256 ? 256 : grid);
    // the first chunk clears the status words if it holds every descriptor
    const uint32_t ns = (n_status && frames_off + (size_t)n_status * sizeof(FrameDev) <= take)
                            ? n_status : 0u;
    if (take <= small) {
      RecordChunk<kRecordChunkSmall> c;
      if (take) memcpy(c.w, h, take);
      k_put_record<kRecordChunkSmall><<<grid, 256, 0, st>>>(c, n16, reinterpret_cast<uint4*>(d),
                                                            z, zn, (uint32_t)frames_off, ns);
    } else {
      RecordChunk<kRecordChunkBig> c;
      memcpy(c.w, h, take);
      k_put_record<kRecordChunkBig><<<grid, 256, 0, st>>>(c, n16, reinterpret_cast<uint4*>(d), z,
                                                          zn, (uint32_t)frames_off, ns);
    }
    n_status = 0;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    h += take;
    d += take;
    bytes -= take;
    zn = 0;
  } while (bytes);
  return cudaSuccess;
}

__global__ void k_zero_status(const FrameDev* frames, uint32_t n_frames) {
  for (uint32_t f = blockIdx.x * blockDim.x + threadIdx.x; f < n_frames;
       f += gridDim.x * blockDim.x)
    *frames[f].status = 0u;
}

// Block totals of the track lengths, zero-length check, length histogram.
__global__ void __launch_bounds__(256) k_track_scan1(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  __shared__ uint32_t hist[kLenBuckets];
  uint32_t tot;
  const uint32_t f = find_frame(plan.pre_tblk, plan.n_frames, blockIdx.x);
  const FrameDev& F = frames[f];
  const uint32_t lb = blockIdx.x - plan.pre_tblk[f];
  for (int i = threadIdx.x; i < kLenBuckets; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  const uint32_t t0 = lb * kTrackBlk + threadIdx.x * 8;
  uint32_t sum = 0;
  bool zero = false;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const uint32_t t = t0 + k;
    if (t < F.n_tracks) {
      const uint32_t n = F.ncl[t];
      sum += n;
      zero |= (n == 0);
      atomicAdd(&hist[n < kLenBuckets ? n : kLenBuckets - 1], 1u);
    }
  }
  if (__syncthreads_or(zero) && threadIdx.x == 0) atomicOr(F.status, kStCount);
  block_excl_scan<256>(sum, tot);
  if (threadIdx.x == 0) F.blk_sum[lb] = tot;
  for (int i = threadIdx.x; i < kLenBuckets; i += blockDim.x)
    if (hist[i]) atomicAdd(&F.len_cursor[i], hist[i]);
}

// Exclusive scan of one value per bin (value(b), put(b, prefix)) by a block of
// 1024 threads; returns the total.  Values and prefixes pass through shared
// memory so that neighbouring lanes read and write neighbouring bins (six
// consecutive bins per thread in global memory are six times the L1 requests of
// a block that has its SM to itself: 8.1 against 7.6 us for the row offsets,
// timing events included).
template <class Value, class Put>
__device__ __forceinline__ uint32_t scan_bins(Value value, Put put) {
  constexpr int Q = (kNBin + 1023) / 1024;
  static_assert(kNBin % Q == 0, "a thread has all its bins or none");
  __shared__ uint32_t s_bin[kNBin];
  const uint32_t tid = threadIdx.x, b0 = tid * Q;
  uint32_t v[Q], sum = 0, tot;
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (tid + 1024 * q < (uint32_t)kNBin) v[q] = value(tid + 1024 * q);
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (tid + 1024 * q < (uint32_t)kNBin) s_bin[tid + 1024 * q] = v[q];
  __syncthreads();
  const bool mine = b0 < (uint32_t)kNBin;
#pragma unroll
  for (int q = 0; q < Q; q++) {
    v[q] = mine ? s_bin[b0 + q] : 0u;
    sum += v[q];
  }
  uint32_t run = block_excl_scan<1024>(sum, tot);
#pragma unroll
  for (int q = 0; q < Q; q++) {
    if (mine) s_bin[b0 + q] = run;
    run += v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (tid + 1024 * q < (uint32_t)kNBin) put(tid + 1024 * q, s_bin[tid + 1024 * q]);
  return tot;
}

// Starts of the unattached bins, their total checked, and the attached counts
// per bin cleared; one block of 1024 threads.
__device__ __forceinline__ void unatt_bins(const FrameDev& F) {
  const uint32_t tid = threadIdx.x;
  const uint32_t* __restrict__ cnt = F.n_unatt_bin;
  uint32_t* __restrict__ start = F.unatt_start;
  uint32_t* __restrict__ att = F.att_count;
  // attached counts: summed into by k_count_rank or k_group_sum (an encoding
  // call has none)
  const uint32_t tot = scan_bins([&](uint32_t b) { return cnt[b]; },
                                 [&](uint32_t b, uint32_t v) {
                                   start[b] = v;
                                   if (att) att[b] = 0u;
                                 });
  if (tid == 0) {
    start[kNBin] = tot;
    if (tot != F.n_unatt) atomicOr(F.status, kStCount);
  }
}

// Per frame: offsets of the track blocks, decode-order bucket offsets (longest
// first), unattached bin starts, count checks.
__global__ void __launch_bounds__(1024) k_frame_scan(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  uint32_t tot;
  const FrameDev& F = frames[blockIdx.x];
  const uint32_t tid = threadIdx.x;
  unsigned long long carry = 0;
  for (uint32_t base = 0; base < F.n_tblocks; base += 1024) {
    const uint32_t i = base + tid;
    const uint32_t v = i < F.n_tblocks ? F.blk_sum[i] : 0u;
    const uint32_t e = block_excl_scan<1024>(v, tot);
    if (i < F.n_tblocks) F.blk_sum[i] = (uint32_t)carry + e;
    carry += tot;
  }
  if (tid == 0 && carry != F.n_att) atomicOr(F.status, kStCount);
  {
    const uint32_t b = kLenBuckets - 1 - tid;  // descending length
    const uint32_t v = F.len_cursor[b];
    const uint32_t e = block_excl_scan<1024>(v, tot);
    F.len_cursor[b] = e;
  }
  unatt_bins(F);
}

// trackStart and decode order.  A block first counts its tracks per length
// bucket in shared memory and reserves each bucket's range of the order with
// one global atomic per bucket; the order of tracks of equal length is
// arbitrary (it only changes which warp decodes a track, not a result).
__global__ void __launch_bounds__(256) k_track_scan2(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  __shared__ uint32_t s_cnt[kLenBuckets];
  uint32_t tot;
  const uint32_t f = find_frame(plan.pre_tblk, plan.n_frames, blockIdx.x);
  const FrameDev& F = frames[f];
  if (*F.status & kStCount) return;
  for (int i = threadIdx.x; i < kLenBuckets; i += blockDim.x) s_cnt[i] = 0u;
  const uint32_t lb = blockIdx.x - plan.pre_tblk[f];
  const uint32_t t0 = lb * kTrackBlk + threadIdx.x * 8;
  const uint32_t nt = F.n_tracks;
  uint32_t n[8], slot[8];
  uint32_t sum = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const uint32_t t = t0 + k;
    n[k] = t < nt ? (uint32_t)F.ncl[t] : 0u;
    sum += n[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; k++)
    if (t0 + k < nt) slot[k] = atomicAdd(&s_cnt[n[k] < kLenBuckets ? n[k] : kLenBuckets - 1], 1u);
  uint32_t start = F.blk_sum[lb] + block_excl_scan<256>(sum, tot);  // synchronises the block
  for (int i = threadIdx.x; i < kLenBuckets; i += blockDim.x) {
    const uint32_t c = s_cnt[i];
    if (c) s_cnt[i] = atomicAdd(&F.len_cursor[i], c);
  }
  __syncthreads();
  uint32_t* __restrict__ track_start = F.track_start;
  uint32_t* __restrict__ order = F.order;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const uint32_t t = t0 + k;
    if (t < nt) {
      track_start[t] = start;
      order[s_cnt[n[k] < kLenBuckets ? n[k] : kLenBuckets - 1] + slot[k]] = t;
      start += n[k];
      if (t == nt - 1) track_start[nt] = start;
    }
  }
}

// The whole track preparation of frames of at most kPrepTracks tracks in one
// launch, two blocks per frame (tracks; unattached bins): a call of small
// frames is a chain of latencies, and the three kernels above take 25 us for 2000
// tracks where this one takes 8 us (28 and 17 us for 11 111 tracks).
__global__ void __launch_bounds__(1024) k_track_prep(const FrameDev* frames) {
  __shared__ uint32_t s_cur[kLenBuckets];
  // lengths, then the order, then track starts by halves: global memory is read
  // and written by neighbouring lanes at neighbouring tracks (see scan_bins)
  extern __shared__ __align__(16) uint32_t s_dyn[];
  uint16_t* s_len = reinterpret_cast<uint16_t*>(s_dyn);  // kPrepTracks
  chain_wait();
  const FrameDev& F = frames[blockIdx.x];
  if (blockIdx.y == 1) {
    unatt_bins(F);
    return;
  }
  constexpr int E = kPrepTracks / 1024;
  const uint32_t tid = threadIdx.x, nt = F.n_tracks;
  const uint32_t per = (nt + 1023) / 1024;  // consecutive tracks per thread, at most E
  const uint16_t* __restrict__ ncl = F.ncl;
  static_assert(kLenBuckets == 1024, "one bucket per thread");
  s_cur[tid] = 0u;
#pragma unroll
  for (int k = 0; k < E; k++)
    if (tid + 1024 * k < nt) s_len[tid + 1024 * k] = ncl[tid + 1024 * k];
  __syncthreads();
  uint32_t n[E], sum = 0, tot;
  bool zero = false;
#pragma unroll
  for (int k = 0; k < E; k++) {
    const uint32_t t = tid * per + k;
    const bool in = (uint32_t)k < per && t < nt;
    n[k] = in ? (uint32_t)s_len[t] : 0u;
    sum += n[k];
    zero |= in && n[k] == 0;
    if (in) atomicAdd(&s_cur[min(n[k], (uint32_t)kLenBuckets - 1)], 1u);
  }
  uint32_t start = block_excl_scan<1024>(sum, tot);  // at most 2^14 * 65535: no overflow
  if (__syncthreads_or(zero) || tot != F.n_att) {
    if (tid == 0) atomicOr(F.status, kStCount);
    return;
  }
  // buckets in descending length
  const uint32_t b = kLenBuckets - 1 - tid, v = s_cur[b];
  const uint32_t e = block_excl_scan<1024>(v, tot);
  s_cur[b] = e;
  __syncthreads();  // also: every length is in registers
#pragma unroll
  for (int k = 0; k < E; k++) {
    const uint32_t t = tid * per + k;
    if ((uint32_t)k < per && t < nt)
      s_len[atomicAdd(&s_cur[min(n[k], (uint32_t)kLenBuckets - 1)], 1u)] = (uint16_t)t;
  }
  __syncthreads();
  uint32_t* __restrict__ order = F.order;
#pragma unroll
  for (int k = 0; k < E; k++)
    if (tid + 1024 * k < nt) order[tid + 1024 * k] = s_len[tid + 1024 * k];
  uint32_t* __restrict__ track_start = F.track_start;
  constexpr uint32_t H = kPrepTracks / 2;
  for (uint32_t h = 0; h < nt; h += H) {
    __syncthreads();
    uint32_t at = start;
#pragma unroll
    for (int k = 0; k < E; k++) {
      const uint32_t t = tid * per + k;
      if ((uint32_t)k < per && t < nt) {
        if (t >= h && t < h + H) s_dyn[t - h] = at;
        at += n[k];
      }
    }
    __syncthreads();
    for (uint32_t t = h + tid; t < nt && t < h + H; t += 1024) track_start[t] = s_dyn[t - h];
  }
  if (tid == 0) track_start[nt] = F.n_att;
}

// Sum of the tile histograms over groups of kGroup tiles, per bin; the group
// sums are also added into the bin's attached count (cleared by k_frame_scan).
// Calls with a frame of several groups; see launch_count_rank.
__global__ void __launch_bounds__(kBinBlk) k_group_sum(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  const uint32_t f = find_frame(plan.pre_grp, plan.n_frames, blockIdx.x);
  const FrameDev& F = frames[f];
  if (*F.status & kStCount) return;
  const uint32_t lb = blockIdx.x - plan.pre_grp[f];
  const uint32_t g = lb / kBinBlocks;
  const uint32_t b = (lb % kBinBlocks) * kBinBlk + threadIdx.x;
  if (b >= (uint32_t)kNBin) return;
  const uint32_t t0 = g * kGroup, nt = min((uint32_t)kGroup, F.n_tiles - t0);
  const uint16_t* __restrict__ hist = F.tile_hist + (size_t)t0 * kNBin + b;
  uint32_t s = 0;
#pragma unroll
  for (uint32_t k = 0; k < (uint32_t)kGroup; k++)  // all loads in flight at once
    s += k < nt ? (uint32_t)hist[(size_t)k * kNBin] : 0u;
  F.group_sum[(size_t)g * kNBin + b] = s;
  if (s) atomicAdd(&F.att_count[b], s);
}

// rowStart = exclusive scan of attached + unattached counts per bin, one block
// of 1024 threads per frame.
__device__ __forceinline__ void row_start_scan(const FrameDev& F) {
  const uint32_t* __restrict__ att = F.att_count;
  const uint32_t* __restrict__ un = F.n_unatt_bin;
  uint32_t* __restrict__ rs = F.row_start;
  const uint32_t tot = scan_bins([&](uint32_t b) { return att[b] + un[b]; },
                                 [&](uint32_t b, uint32_t v) { rs[b] = v; });
  if (threadIdx.x == 0) rs[kNBin] = tot;
}

// Per frame: rowStart (the attached counts are there).
__global__ void __launch_bounds__(1024) k_row_offsets(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  const FrameDev& F = frames[blockIdx.x];
  if (*F.status & kStCount) return;
  row_start_scan(F);
}

// First native index of every (tile, bin): rowStart plus the counts of the
// bin in the groups and tiles before.
__global__ void __launch_bounds__(kBinBlk) k_tile_base(const FrameDev* frames, PlanDev plan) {
  chain_wait();
  const uint32_t f = find_frame(plan.pre_grp, plan.n_frames, blockIdx.x);
  const FrameDev& F = frames[f];
  if (*F.status & kStCount) return;
  const uint32_t lb = blockIdx.x - plan.pre_grp[f];
  const uint32_t g = lb / kBinBlocks;
  const uint32_t b = (lb % kBinBlocks) * kBinBlk + threadIdx.x;
  if (b >= (uint32_t)kNBin) return;
  const uint32_t* __restrict__ gsum = F.group_sum;
  uint32_t* __restrict__ tbase = F.tile_base;
  const uint32_t t0 = g * kGroup, nt = min((uint32_t)kGroup, F.n_tiles - t0);
  const uint16_t* __restrict__ hist = F.tile_hist + (size_t)t0 * kNBin + b;
  // the group's tile counts first (all loads in flight), then the bases
  uint32_t c[kGroup];
#pragma unroll
  for (uint32_t k = 0; k < (uint32_t)kGroup; k++) c[k] = k < nt ? (uint32_t)hist[(size_t)k * kNBin] : 0u;
  uint32_t run = F.row_start[b];
#pragma unroll 8
  for (uint32_t gg = 0; gg < g; gg++) run += gsum[(size_t)gg * kNBin + b];
#pragma unroll
  for (uint32_t k = 0; k < (uint32_t)kGroup; k++) {
    if (k < nt) tbase[(size_t)(t0 + k) * kNBin + b] = run;
    run += c[k];
  }
}

}  // namespace tmd
