// Device functions of the library checked one by one (test_gpu_device_checks.py
// builds this file and loads it).
#include "../paper_2411_02206_gb300/csrc/tmd_internal.cuh"
#include "../paper_2411_02206_gb300/csrc/tmd_model.cuh"

using namespace tmd;

namespace {

// The forms that the model's shortcuts stand for.
__device__ uint32_t plain_quant(float v, float hi) {
  v = fminf(fmaxf(v, 0.0f), hi);
  return __float2uint_rd(fadd(v, 0.5f));
}
__device__ float plain_pad_to_y(const float4& G, uint32_t padq) {
  return fmul(ffma((float)padq, 0.015625f, -G.w), G.y);
}
__device__ float plain_time_to_t(uint32_t timeq) { return fmul((float)timeq, 0.03125f); }

__device__ bool differ(float a, float b) { return __float_as_uint(a) != __float_as_uint(b); }

// Mismatches over all 2^32 bit patterns: [0], [1] frcp2 in its first and second
// place (the other operand 1, whose reciprocal is exact: the guard is at its
// widest), [2], [3] quant at both limits, [4] time_to_t, [5] pad_to_y over all
// codes and rows.
__global__ void k_sweep(unsigned long long* bad) {
  __shared__ RowGeo geo;
  fill_row_geo(&geo);
  __syncthreads();
  uint32_t n[6] = {};
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += step) {
    const uint32_t u = (uint32_t)i;
    const float x = __uint_as_float(u), want = __frcp_rn(x);
    float a, b;
    frcp2(x, 1.0f, a, b);
    n[0] += differ(a, want) || differ(b, 1.0f);
    frcp2(1.0f, x, a, b);
    n[1] += differ(b, want) || differ(a, 1.0f);
    n[2] += quant(x, kPadHi) - kIntBits != plain_quant(x, kPadHi);
    n[3] += quant(x, kTimeHi) - kIntBits != plain_quant(x, kTimeHi);
    n[4] += differ(time_to_t(u), plain_time_to_t(u));
    if (u < 65536u * kNRow) {
      const float4 G = geo.row[u >> 16];
      n[5] += differ(pad_to_y(G, u & 0xFFFFu), plain_pad_to_y(G, u & 0xFFFFu));
    }
  }
  for (int k = 0; k < 6; k++)
    if (n[k]) atomicAdd(&bad[k], n[k]);
}

// One grid barrier of `extra` more arrivals than there are blocks: with any, its
// wait is bounded.  out[block] = 1 passed, 2 gave up.
__global__ void k_barrier(uint32_t* arrivals, uint32_t extra, uint32_t* out) {
  uint32_t target = extra;
  const bool ok = grid_barrier(arrivals, target);
  if (threadIdx.x == 0) out[blockIdx.x] = ok ? 1u : 2u;
}

}  // namespace

extern "C" int check_sweep(unsigned long long* bad) {
  k_sweep<<<1216, 256>>>(bad);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return (int)e;
}

extern "C" int check_barrier(uint32_t blocks, uint32_t extra, uint32_t* arrivals, uint32_t* out) {
  void* args[] = {&arrivals, &extra, &out};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_barrier, dim3(blocks), dim3(64), args,
                                              0, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return (int)e;
}
