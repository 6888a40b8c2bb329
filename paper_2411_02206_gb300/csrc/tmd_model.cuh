// tmd_model.cuh -- device track model for TPC track-model encoding/decoding
// (arXiv:2411.02206, Sec. 4: the attached-cluster kernel gives each thread one
// track, carries the track model along it through the TPC and restores each
// cluster's absolute coordinates from the stored residual and the model).
//
// The paper leaves the track model to its reference [rohr-global-track]; this
// library defines it as a linear Kalman filter in the sector-local frame:
//   y-block (y, ty = dy/dx, c = d2y/dx2), a parabola in x, 3x3 covariance;
//   t-block (t, tt = dt/dx), a line in drift time, 2x2 covariance.
// Encoder and decoder run the same sequence of binary32 operations; every
// operation below is an explicit round-to-nearest intrinsic, the model's
// multiply-adds are explicit fused multiply-adds (one rounding each), and the
// compiler contracts nothing else (-fmad=false): the arithmetic is fixed
// whatever the compiler does with the rest of the code.
#pragma once
#include <cstdint>

namespace tmd {

constexpr int kNSec = 36;
constexpr int kNRow = 152;
constexpr int kNBin = kNSec * kNRow;
constexpr int kRecBytes = 12;

// status bits (also in include/tmd.h)
constexpr uint32_t kStCount = 1u;
constexpr uint32_t kStRow = 2u;
constexpr uint32_t kStTime = 4u;
constexpr uint32_t kStTimeout = 8u;
constexpr uint32_t kStLimit = 16u;

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }
// a * b + c with a single rounding
__device__ __forceinline__ float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// 1/x correctly rounded: the same value as the division 1.0f / x.
__device__ __forceinline__ float frcp(float x) { return __frcp_rn(x); }
// Two correctly rounded reciprocals at once.  The hardware approximation and
// one correction y + y (1 - x y) (P. Markstein, IBM J. Res. Dev. 34, 1990) give
// the value of __frcp_rn wherever 1 - x y is small, which was checked on all
// 2^32 operands; the others (zero, denormal, huge, infinite, NaN) take
// __frcp_rn.  Two calls of __frcp_rn are two branches that cut a model step
// into pieces executed one after the other; here one test serves both and the
// two chains and the code around them interleave.
__device__ __forceinline__ void frcp2(float a, float b, float& ia, float& ib) {
  float ya, yb;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ya) : "f"(a));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yb) : "f"(b));
  const float ea = __fmaf_rn(-a, ya, 1.0f), eb = __fmaf_rn(-b, yb, 1.0f);
  ia = __fmaf_rn(ya, ea, ya);
  ib = __fmaf_rn(yb, eb, yb);
  if (!(__fadd_rn(fabsf(ea), fabsf(eb)) < 0.0009765625f)) {  // also for NaN
    ia = __frcp_rn(a);
    ib = __frcp_rn(b);
  }
}

// Model constants (binary32).
constexpr float kSY2 = 0.01f;     // measurement variance of y [cm^2]
constexpr float kST2 = 0.04f;     // measurement variance of t [bin^2]
constexpr float kQTY = 1.0e-6f;   // process noise of dy/dx per cm of |dx|
constexpr float kQTT = 4.0e-6f;   // process noise of dt/dx per cm of |dx|
constexpr float kCTY0 = 0.01f;    // seed variance of dy/dx
constexpr float kCC0 = 1.0e-8f;   // seed variance of d2y/dx2 [cm^-2]
constexpr float kCTT0 = 4.0f;     // seed variance of dt/dx
constexpr float kSYR = 0.25f;     // y variance after a sector or leg change
constexpr float kKC = 0.0015f;    // |d2y/dx2| per unit q/pT
constexpr float kTan10 = 0x1.691e1ep-3f;  // binary32 nearest tan(10 deg)
constexpr float kPadHi = 65535.0f;
constexpr float kTimeHi = 8388607.0f;

// cos/sin of k * 20 deg, k = 0..17, correctly rounded to binary32.
__constant__ float c_cos20[18] = {
    0x1p+0f,         0x1.e11f64p-1f,  0x1.8836fap-1f,  0x1p-1f,         0x1.63a1a8p-3f,
    -0x1.63a1a8p-3f, -0x1p-1f,        -0x1.8836fap-1f, -0x1.e11f64p-1f, -0x1p+0f,
    -0x1.e11f64p-1f, -0x1.8836fap-1f, -0x1p-1f,        -0x1.63a1a8p-3f, 0x1.63a1a8p-3f,
    0x1p-1f,         0x1.8836fap-1f,  0x1.e11f64p-1f};
__constant__ float c_sin20[18] = {
    0.0f,            0x1.5e3a88p-2f,  0x1.491b76p-1f,  0x1.bb67aep-1f,  0x1.f838b8p-1f,
    0x1.f838b8p-1f,  0x1.bb67aep-1f,  0x1.491b76p-1f,  0x1.5e3a88p-2f,  0.0f,
    -0x1.5e3a88p-2f, -0x1.491b76p-1f, -0x1.bb67aep-1f, -0x1.f838b8p-1f, -0x1.f838b8p-1f,
    -0x1.bb67aep-1f, -0x1.491b76p-1f, -0x1.5e3a88p-2f};

// Per-row geometry, filled in shared memory by every block that needs it:
// x = 85 + r cm; nPads = 66 + floor(72 r / 151); pad width w = 2 x tan10 / nPads.
// One 16-byte entry per row {x, w, 1/w, nPads/2}: a model step reads its row
// with a single shared-memory load.
struct RowGeo {
  float4 row[kNRow];
  float2 rot[18];  // cos, sin of k * 20 deg: lanes change sector by different k
};

__device__ __forceinline__ void fill_row_geo(RowGeo* g) {
  for (int r = threadIdx.x; r < kNRow; r += blockDim.x) {
    const int np = 66 + (72 * r) / 151;
    const float x = 85.0f + (float)r;
    const float w = fdiv(fmul(fmul(2.0f, x), kTan10), (float)np);
    g->row[r] = make_float4(x, w, fdiv(1.0f, w), fmul(0.5f, (float)np));
    if (r < 18) g->rot[r] = make_float2(c_cos20[r], c_sin20[r]);
  }
}

// Integers below 2^23 as the low bits of the binary32 number 2^23 + i: an
// addition of 2^23, rounded down, is the floor of the other operand, and a
// subtraction gives the integer as a number, both exact.  A conversion
// instruction takes several times an addition's latency, and the conversions
// of the prediction and the measurement lie one after the other in the model
// chain (decode kernel 41.3 -> 39.9 us for 2000 tracks; no change where all
// warps are resident).
constexpr uint32_t kIntBits = 0x4B000000u;  // 2^23
constexpr float kIntBase = 8388608.0f;

// Quantiser: clamp to [0, hi] (NaN to 0), then floor(v + 0.5), as kIntBits + q.
// fmaxf returns its non-NaN operand, so NaN clamps to 0; v + 0.5 then lies in
// [0.5, hi + 0.5], below 2^23.
__device__ __forceinline__ uint32_t quant(float v, float hi) {
  v = fminf(fmaxf(v, 0.0f), hi);
  return __float_as_uint(__fadd_rd(fadd(v, 0.5f), kIntBase));
}

struct Track {
  float x, y, ty, c;
  float c00, c01, c02, c11, c12, c22;
  float t, tt, d00, d01, d11;
  int raw_row;  // row accumulator (mod 256); the model uses min(raw_row, 151)
  int max_row;  // largest raw_row reached by a step
  int row;
  int sec;
};

// y of a pad code on a row with geometry G = {x, w, 1/w, nPads/2}:
// (pad / 64 - nPads/2) * w.
__device__ __forceinline__ float pad_to_y(const float4& G, uint32_t padq) {
  const float p = fsub(__uint_as_float(kIntBits | padq), kIntBase);  // padq < 2^16
  return fmul(ffma(p, 0.015625f, -G.w), G.y);
}
// Any 32-bit time code: its halves as numbers and one rounding.
__device__ __forceinline__ float time_to_t(uint32_t timeq) {
  const float lo = fsub(__uint_as_float(__byte_perm(timeq, kIntBits, 0x7610)), kIntBase);
  const float hi = fsub(__uint_as_float(__byte_perm(timeq, kIntBits, 0x7632)), kIntBase);
  return fmul(ffma(hi, 65536.0f, lo), 0.03125f);
}

__device__ __forceinline__ void reset_ycov(Track& s) {
  s.c00 = kSYR; s.c01 = 0.0f; s.c02 = 0.0f;
  s.c11 = kCTY0; s.c12 = 0.0f; s.c22 = kCC0;
}

// Seed from the first cluster (stored absolute): the parabola through the
// origin with curvature -kc * q/pT; zero time slope.
__device__ __forceinline__ void seed(const RowGeo* g, Track& s, uint8_t qpta, int raw_row,
                                     int sec, uint32_t padq, uint32_t timeq) {
  const float qpt = fmul(fsub((float)qpta, 127.5f), 0.078125f);
  s.raw_row = raw_row;
  s.max_row = 0;
  s.row = raw_row < kNRow ? raw_row : kNRow - 1;
  s.sec = sec;
  const float4 G = g->row[s.row];
  s.x = G.x;
  s.y = pad_to_y(G, padq);
  s.c = fmul(-kKC, qpt);
  s.ty = fadd(fdiv(s.y, s.x), fmul(fmul(s.c, s.x), 0.5f));
  s.c00 = kSY2; s.c01 = 0.0f; s.c02 = 0.0f;
  s.c11 = kCTY0; s.c12 = 0.0f; s.c22 = kCC0;
  s.t = time_to_t(timeq);
  s.tt = 0.0f;
  s.d00 = kST2; s.d01 = 0.0f; s.d11 = kCTT0;
}

// Leg change: x turns back; slope, curvature and time slope change sign.
__device__ __forceinline__ void leg_change(Track& s) {
  s.ty = -s.ty;
  s.c = -s.c;
  s.tt = -s.tt;
  s.d01 = -s.d01;
  reset_ycov(s);
}

// Sector change by sd = 1..35 sectors (mod 36): rotate the parabola's point,
// slope and curvature by sd * 20 deg; a change of side (A/C) reverses the time
// slope.
__device__ __forceinline__ void sector_change(const RowGeo* g, Track& s, int sd) {
  int nsec = s.sec + sd;
  nsec = nsec >= kNSec ? nsec - kNSec : nsec;
  const float2 cs = g->rot[sd >= 18 ? sd - 18 : sd];
  const float ca = cs.x, sa = cs.y;
  float a = fadd(ca, fmul(s.ty, sa));
  const float b = fsub(fmul(s.ty, ca), sa);
  if (!(a >= 1.0e-3f || a <= -1.0e-3f)) a = (a < 0.0f) ? -1.0e-3f : 1.0e-3f;
  const float nx = fadd(fmul(s.x, ca), fmul(s.y, sa));
  const float ny = fsub(fmul(s.y, ca), fmul(s.x, sa));
  const float ia = frcp(a);
  s.ty = fmul(b, ia);
  s.c = fmul(s.c, fmul(fmul(ia, ia), ia));
  s.x = nx;
  s.y = ny;
  if ((s.sec < 18) != (nsec < 18)) {
    s.tt = -s.tt;
    s.d01 = -s.d01;
  }
  s.sec = nsec;
  reset_ycov(s);
}

// Key step of one cluster in its two parts: the row, which no decoded
// coordinate enters (raw: the row walk's new value, mod 256; a row outside the
// detector shows in s.max_row), and the sector/leg difference.
__device__ __forceinline__ int clamp_row(int raw) { return min(raw, kNRow - 1); }
__device__ __forceinline__ void row_step(Track& s, int raw) {
  s.raw_row = raw;
  s.max_row = max(s.max_row, raw);
  s.row = clamp_row(raw);
}
__device__ __forceinline__ void turn_step(const RowGeo* g, Track& s, uint32_t sld) {
  if (sld != 0) {  // few clusters
    uint32_t sd = sld;
    if (sld >= (uint32_t)kNSec) {
      leg_change(s);
      sd = sld % kNSec;
    }
    if (sd != 0) sector_change(g, s, (int)sd);
  }
}

// Propagate to the plane of the current row, whose geometry is
// G = {x, w, 1/w, nPads/2} (RowGeo), and return the quantised prediction
// (pad code, time code).
__device__ __forceinline__ void propagate_predict(const float4& G, Track& s, uint32_t& ppad,
                                                  uint32_t& ptime) {
  const float xr = G.x;
  const float dx = fsub(xr, s.x);
  const float adx = fabsf(dx);
  const float h = fmul(fmul(0.5f, s.c), dx);
  s.y = ffma(dx, fadd(s.ty, h), s.y);
  s.ty = ffma(s.c, dx, s.ty);
  s.t = ffma(s.tt, dx, s.t);
  s.x = xr;
  const float h2 = fmul(fmul(0.5f, dx), dx);
  const float a0 = ffma(h2, s.c02, ffma(dx, s.c01, s.c00));
  const float a1 = ffma(h2, s.c12, ffma(dx, s.c11, s.c01));
  const float a2 = ffma(h2, s.c22, ffma(dx, s.c12, s.c02));
  const float b1 = ffma(dx, s.c12, s.c11);
  const float b2 = ffma(dx, s.c22, s.c12);
  s.c00 = ffma(h2, a2, ffma(dx, a1, a0));
  s.c01 = ffma(dx, a2, a1);
  s.c02 = a2;
  s.c11 = ffma(kQTY, adx, ffma(dx, b2, b1));
  s.c12 = b2;
  const float e0 = ffma(dx, s.d01, s.d00);
  const float e1 = ffma(dx, s.d11, s.d01);
  s.d00 = ffma(dx, e1, e0);
  s.d01 = e1;
  s.d11 = ffma(kQTT, adx, s.d11);
  const float pp = ffma(s.y, G.z, G.w);
  ppad = quant(fmul(pp, 64.0f), kPadHi) - kIntBits;
  ptime = quant(fmul(s.t, 32.0f), kTimeHi) - kIntBits;
}

// Kalman update with the measured cluster (G: geometry of the current row).
__device__ __forceinline__ void update(const float4& G, Track& s, uint32_t padq, uint32_t timeq) {
  const float ym = pad_to_y(G, padq);
  const float tm = time_to_t(timeq);
  float inv, invt;
  frcp2(fadd(s.c00, kSY2), fadd(s.d00, kST2), inv, invt);
  const float k0 = fmul(s.c00, inv), k1 = fmul(s.c01, inv), k2 = fmul(s.c02, inv);
  const float r = fsub(ym, s.y);
  s.y = ffma(k0, r, s.y);
  s.ty = ffma(k1, r, s.ty);
  s.c = ffma(k2, r, s.c);
  const float c00 = s.c00, c01 = s.c01, c02 = s.c02;
  s.c00 = ffma(-k0, c00, c00);
  s.c01 = ffma(-k0, c01, c01);
  s.c02 = ffma(-k0, c02, c02);
  s.c11 = ffma(-k1, c01, s.c11);
  s.c12 = ffma(-k1, c02, s.c12);
  s.c22 = ffma(-k2, c02, s.c22);
  const float g0 = fmul(s.d00, invt), g1 = fmul(s.d01, invt);
  const float rt = fsub(tm, s.t);
  s.t = ffma(g0, rt, s.t);
  s.tt = ffma(g1, rt, s.tt);
  const float d00 = s.d00, d01 = s.d01;
  s.d00 = ffma(-g0, d00, d00);
  s.d01 = ffma(-g0, d01, d01);
  s.d11 = ffma(-g1, d01, s.d11);
}

}  // namespace tmd
