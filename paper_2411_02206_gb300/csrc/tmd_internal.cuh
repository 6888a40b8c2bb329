// tmd_internal.cuh -- device-side frame descriptors and launch helpers shared
// by the decoder's CUDA translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "tmd_model.cuh"

namespace tmd {

// Work decomposition (fixed by the decoder, independent of the GPU model).
constexpr int kTrackBlk = 2048;          // tracks per block of the track scan
constexpr int kTile = 32768;             // attached clusters per ranking tile
constexpr int kGroup = 32;               // tiles per group of the tile scan
constexpr int kBinBlk = 256;             // bins per block of the tile scan
constexpr int kBinBlocks = (kNBin + kBinBlk - 1) / kBinBlk;
constexpr int kChunk = 2048;             // unattached clusters per scan chunk
constexpr int kLenBuckets = 1024;        // track-length buckets of the decode order
constexpr int kDecodeThreads = 128;      // threads per block of the track decoder
constexpr int kScatThreads = 256;        // threads per block of the record scatter

// One frame as the kernels see it: caller inputs, caller outputs, scratch.
struct FrameDev {
  uint32_t n_tracks, n_att, n_unatt;
  uint32_t n_tblocks, n_tiles, n_groups, n_chunks;
  // per track
  const uint8_t* qpt;
  const uint8_t* row;
  const uint8_t* slice;
  const uint16_t* pad;
  const uint32_t* time;
  const uint16_t* ncl;
  // per attached cluster
  const uint16_t* qtot_a;
  const uint16_t* qmax_a;
  const uint8_t* flags_a;
  const uint8_t* sigp_a;
  const uint8_t* sigt_a;
  // per attached cluster after the first of its track
  const uint8_t* row_diff;
  const uint8_t* sld;
  const uint16_t* pad_res;
  const uint32_t* time_res;
  // per (sector,row)
  const uint32_t* n_unatt_bin;
  // per unattached cluster
  const uint16_t* pad_diff_u;
  const uint32_t* time_diff_u;
  const uint16_t* qtot_u;
  const uint16_t* qmax_u;
  const uint8_t* flags_u;
  const uint8_t* sigp_u;
  const uint8_t* sigt_u;
  // outputs
  uint8_t* native;
  uint32_t* row_start;
  uint32_t* att_count;
  uint32_t* status;
  // scratch
  uint32_t* track_start;   // n_tracks + 1
  uint32_t* order;         // n_tracks, longest tracks first
  uint16_t* keys;          // n_att: (sector,row) bin of every attached cluster
  uint16_t* kf_pad;        // n_att: decoded pad code of every attached cluster
  uint32_t* kf_time;       // n_att: decoded time code of every attached cluster
  uint16_t* rank;          // n_att: rank of a cluster within its (tile, bin)
  uint16_t* tile_hist;     // n_tiles x kNBin
  uint32_t* group_sum;     // n_groups x kNBin
  uint32_t* tile_base;     // n_tiles x kNBin: first native index of (tile, bin)
  uint32_t* unatt_start;   // kNBin + 1
  uint32_t* blk_sum;       // n_tblocks
  uint32_t* len_cursor;    // kLenBuckets (zeroed)
  unsigned long long* lookback;  // n_chunks (zeroed)
};

// Encoder view of a frame: attached truth in, compressed attached streams out.
struct EncDev {
  uint32_t n_tracks, n_att;
  const uint8_t* qpt;
  const uint16_t* ncl;
  const uint8_t* row;
  const uint8_t* sector;
  const uint8_t* leg;
  const uint16_t* pad;
  const uint32_t* time;
  uint8_t* o_qpt;
  uint8_t* o_row;
  uint8_t* o_slice;
  uint16_t* o_pad;
  uint32_t* o_time;
  uint16_t* o_ncl;
  uint8_t* o_row_diff;
  uint8_t* o_sld;
  uint16_t* o_pad_res;
  uint32_t* o_time_res;
};

// Launch plan of a batch: for each kernel family the exclusive prefix over
// frames of its work items, so that a block can find its frame.
struct PlanDev {
  uint32_t n_frames;
  const uint32_t* pre_tblk;   // track-scan blocks
  const uint32_t* pre_tile;   // ranking tiles
  const uint32_t* pre_grp;    // tile-group blocks (n_groups * kBinBlocks)
  const uint32_t* pre_warp;   // encoder: warp tasks
  const uint32_t* pre_chunk;  // unattached chunks
  const uint32_t* pre_kt;     // decoder: warp tasks
  uint32_t lanes;             // tracks per warp task (task_lanes)
  uint32_t* counters;         // [0] decode/encode task, [1] unattached ticket, short
                              // tracks of an encoding call (zeroed)
};

// Tracks per warp task of the track decoder and encoder, one lane each.  A call
// whose tracks fill all resident warps takes 32.  A smaller call is as long as
// its longest track's chain of steps, and a step is the longer the more lanes
// share it (a lane's sector change holds up the others; every track of the
// warp is written out): it takes fewer lanes as long as its tasks are resident
// together.  2000 tracks: 61 us at 32 lanes, 41 us at 4; 11 111 tracks: 62 us at
// 32, 51 us at 8.
inline uint32_t task_lanes(uint64_t n_tracks, uint32_t sms) {
  const uint64_t warps = 12ull * sms;  // 3 blocks of 4 warps per SM
  for (uint32_t l = 4; l < 32; l *= 2)
    if (n_tracks <= l * warps) return l;
  return 32;
}

// Largest f with pre[f] <= item (pre has n+1 entries, pre[0] = 0).
__device__ __forceinline__ uint32_t find_frame(const uint32_t* pre, uint32_t n, uint32_t item) {
  uint32_t lo = 0, hi = n;  // answer in [lo, hi)
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(pre + mid) <= item) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ uint32_t lanemask_le() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
  return m;
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Overlapped launches.  A kernel of a chain begins with chain_wait, before it
// touches memory: launched by launch_chained its blocks are placed while the
// kernel before finishes and wait there; launched plainly it returns at once.
// The next kernel is let in only after the wait, so that no more than one
// kernel waits, and it is placed only when every block of this one is running:
// waiting blocks take no place that a running kernel still needs.  (Let in
// before the wait, whole chains of waiting blocks had slowed the large frames.)
// Small frame 78 -> 75 us, pp-like frame 147 -> 131 us, small coded frame 157 ->
// 147 us, full frame 1120 -> 1102 us, 2 M unattached clusters encoded 127 -> 116 us.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Barrier of all blocks of a cooperative launch; arrivals starts at 0, target (of
// each thread) too.  False if they did not all arrive within kBarrierPolls polls:
// the caller then leaves with kStTimeout.
constexpr uint32_t kBarrierPolls = 1u << 22;
__device__ __forceinline__ bool grid_barrier(uint32_t* arrivals, uint32_t& target) {
  __shared__ int s_ok;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrivals, 1u);
    int ok = 0;
    for (uint32_t i = 0; i < kBarrierPolls && !ok; i++) {
      ok = (int32_t)(*(volatile uint32_t*)arrivals - target) >= 0;
      if (!ok) __nanosleep(64);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Kernels (launched by tmd_api.cu).
// Launch-record upload as a kernel parameter (no copy engine), in chunks of
// 2 KiB or 16 KiB; bytes and zero_bytes are multiples of 16.  Also clears
// zero_bytes at `zero`.  Returns the launch error, if any.
constexpr int kRecordChunkSmall = 128, kRecordChunkBig = 1024;
template <int W>
struct RecordChunk {
  uint4 w[W];
};
cudaError_t put_record(const void* host, size_t bytes, void* dev, void* zero, size_t zero_bytes,
                       cudaStream_t st, size_t frames_off = 0, uint32_t n_status = 0);
// Whether put_record(..., frames_off, n_frames) clears the frames' status
// words itself (all descriptors in its first launch).
bool put_record_zeroes_status(size_t frames_off, uint32_t n_frames);
__global__ void k_zero_status(const FrameDev* frames, uint32_t n_frames);
__global__ void k_track_scan1(const FrameDev* frames, PlanDev plan);
__global__ void k_frame_scan(const FrameDev* frames, PlanDev plan);
__global__ void k_track_scan2(const FrameDev* frames, PlanDev plan);
// The same for frames of at most kPrepTracks tracks (grid: frames x 2).
constexpr int kPrepTracks = 16384;
constexpr int kTrackPrepSmem = kPrepTracks * 2;
__global__ void k_track_prep(const FrameDev* frames);
// Tile histograms and stable ranks of the attached clusters from their keys
// (grid: ranking tiles of all frames).
// With sum, the tiles' counts are added into the bins' attached counts here:
// calls whose frames are of one group of tiles each need no k_group_sum (4.5 us
// and a launch; with many tiles the adds slow the ranking more than that).
void launch_count_rank(uint32_t n_tiles, bool sum, uint32_t sms, cudaStream_t st,
                       const FrameDev* frames, PlanDev plan);
cudaError_t prepare_count_rank();
// Shared-memory attribute of the tiled global transform; its resident blocks.
cudaError_t prepare_global_xyz(int* blocks_per_sm);
// Shared-memory attributes of the unattached encoder; resident blocks per SM
// of its cooperative kernel.
cudaError_t prepare_unatt_encode(int* blocks_per_sm);
__global__ void k_group_sum(const FrameDev* frames, PlanDev plan);
__global__ void k_row_offsets(const FrameDev* frames, PlanDev plan);
__global__ void k_tile_base(const FrameDev* frames, PlanDev plan);
// The track decoder is instantiated in variants of its staging (a tuning
// parameter, every instance computes identical results); host code launches
// it through these two functions.  Its warps take tasks of plan.lanes tracks
// (pre_kt of the plan) from counters[0] and write the key, pad code and time code of
// every attached cluster.
void launch_track_decode(int variant, uint32_t grid, cudaStream_t st, const FrameDev* frames,
                         PlanDev plan, uint32_t n_tasks);
cudaError_t prepare_track_decode(int variant, int* blocks_per_sm);
// Record scatter variants 0, 1 (identical results; see tmd_scatter.cu),
// launched over n_tiles ranking tiles of all frames.
void launch_att_scatter(int variant, uint32_t n_tiles, cudaStream_t st, const FrameDev* frames,
                        PlanDev plan);
// Unattached decode variants 0, 1 (record write-out word by word or one
// record per thread; identical results), launched through these functions.
void launch_unatt_decode(int variant, uint32_t grid, cudaStream_t st, const FrameDev* frames,
                         PlanDev plan, uint32_t n_tickets, bool chained = false);
cudaError_t occupancy_unatt_decode(int* blocks_per_sm);
__global__ void k_selftest_wait(const unsigned long long* never, uint32_t* status);
// One frame.  blocks_per_sm: of the kernel and of the one for short tracks.
void launch_track_encode(uint64_t n_tracks, uint64_t n_attached, uint32_t sms,
                         const int* blocks_per_sm, cudaStream_t st, const EncDev* enc,
                         const FrameDev* frames, PlanDev plan, uint32_t n_tasks);
cudaError_t prepare_track_encode(int* blocks_per_sm);
__global__ void k_track_trace(const FrameDev* frames, const uint32_t* ids, uint32_t n_ids,
                              float* state);

constexpr int kRankTags = 2048;  // per-warp duplicate-test slots of the ranking (bytes)

}  // namespace tmd
