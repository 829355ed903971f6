// emc_common.cuh -- device helpers shared by the libemc kernels (sm_103a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/emc.h"

namespace emc {

// ---------------------------------------------------------------------------
// Device status word: the first error recorded wins.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  if (status) atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------------------
// Two FP32 operations in one instruction, each half rounded as its scalar form.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)),
        "l"(*reinterpret_cast<unsigned long long*>(&c)));
  return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)),
        "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}

// ---------------------------------------------------------------------------
// Double-float ("f2") arithmetic: value = h + l with |l| <= ulp(h)/2, where an
// FP32 sum is not enough and FP64 is rare on this part.
// ---------------------------------------------------------------------------
struct f2 {
  float h, l;
};

__device__ __forceinline__ f2 two_sum(float a, float b) {
  float s = a + b;
  float bb = s - a;
  float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}

// Hamilton rotation matrix of a unit quaternion (w, x, y, z), in FP64.
__host__ __device__ __forceinline__ void quat_to_rot(const double* q, double* R) {
  double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z);     R[2] = 2 * (x * z + w * y);
  R[3] = 2 * (x * y + w * z);     R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
  R[6] = 2 * (x * z - w * y);     R[7] = 2 * (y * z + w * x);     R[8] = 1 - 2 * (x * x + y * y);
}

// Grid coordinate p = R q + N/2 of one pixel, split into the integer corner
// f (floor) and the fraction t in [0, 1], in fixed point. With q = qi 2^-12 + qlo (qi integer,
// |qlo| <= 2^-13) and R = Rh 2^-20 + Rl (Rh integer, |Rl| <= 2^-21),
//   p = N/2 + sum_b Rh_b qi_b 2^-32 + sum_b (Rh_b 2^-20 qlo_b + Rl_b qi_b 2^-12)
// up to |Rl qlo| < 2^-34: the first sum is exact in 64-bit integers (its high
// word the floor, its low word the fraction to 2^-32), the small terms
// (|.| < 1e-3) take six FP32 FMAs. Rhf = Rh 2^-20 and qhf = qi 2^-12 as FP32
// (exact). Error ~1e-10 voxel.
__device__ __forceinline__ void rotate_fx(const int* Rh, const float* Rhf, const float* Rl,
                                          int4 qi, float4 qhf, float4 qlo, int N, int* f,
                                          float* t) {
  const int qiv[3] = {qi.x, qi.y, qi.z};
  const float qhv[3] = {qhf.x, qhf.y, qhf.z}, qlv[3] = {qlo.x, qlo.y, qlo.z};
#pragma unroll
  for (int a = 0; a < 3; a++) {
    long long acc = ((long long)(N >> 1) << 32) + ((N & 1) ? (1LL << 31) : 0LL);
#pragma unroll
    for (int b = 0; b < 3; b++) acc += (long long)Rh[3 * a + b] * (long long)qiv[b];
    const float small =
        fmaf(Rhf[3 * a], qlv[0],
             fmaf(Rhf[3 * a + 1], qlv[1],
                  fmaf(Rhf[3 * a + 2], qlv[2],
                       fmaf(Rl[3 * a], qhv[0], fmaf(Rl[3 * a + 1], qhv[1], Rl[3 * a + 2] * qhv[2])))));
    int fl = (int)(acc >> 32);
    // the 32-bit fraction as FP32 without a conversion instruction: its top 23
    // bits as the mantissa of a number in [1, 2), the low 9 bits likewise
    const unsigned fw = (unsigned)(acc & 0xffffffffLL);
    const float fhi = __uint_as_float(0x3f800000u | (fw >> 9)) - 1.0f;           // exact
    const float flo = __uint_as_float(0x3f800000u | ((fw & 511u) << 14)) - 1.0f;  // exact
    float fr = fhi + fmaf(flo, 0x1p-23f, small);
    if (fr < 0.f) {
      fl -= 1;
      fr += 1.f;
    } else if (fr >= 1.f) {
      fl += 1;
      fr -= 1.f;
    }
    f[a] = fl;
    t[a] = fminf(fmaxf(fr, 0.f), 1.f);
  }
}

// Trilinear value (Eq. 2.8, tent weights) at p = f + t from the grid in its
// cell layout: the eight corners of voxel l = (x N + y) N + z in g4[2 l] =
// (g[x][y][z], g[x][y][z+1], g[x][y+1][z], g[x][y+1][z+1]) and, for x + 1, in
// g4[2 l + 1] (0 beyond the grid). One 32-byte load per point, a whole sector,
// where the plain layout needs eight scattered 4-byte ones: the loads are
// gathers (every lane of a warp reads another cache line), and their
// wavefronts are what the expansion waits for. Corners inside the grid only
// (interior points), N <= 256.
struct Cell {
  float4 a, b;  // corners at x, corners at x + 1
};
__device__ __forceinline__ Cell load_cell(const float4* __restrict__ g4, int voxel) {
  Cell c;
  asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(c.a.x), "=f"(c.a.y), "=f"(c.a.z), "=f"(c.a.w), "=f"(c.b.x), "=f"(c.b.y),
        "=f"(c.b.z), "=f"(c.b.w)
      : "l"(g4 + 2 * voxel));
  return c;
}
__device__ __forceinline__ float cell_value(const Cell& c, const float* t) {
  const float4 a = c.a, b = c.b;
  const float tz = t[2], sz = 1.f - tz, ty = t[1], sy = 1.f - ty;
  const float va = sy * fmaf(tz, a.y, sz * a.x) + ty * fmaf(tz, a.w, sz * a.z);
  const float vb = sy * fmaf(tz, b.y, sz * b.x) + ty * fmaf(tz, b.w, sz * b.z);
  return fmaf(t[0], vb, (1.f - t[0]) * va);
}

// FP32 -> FP64 with integer operations (the conversion instruction runs on the
// FP64 pipe, at 1/64 of the FP32 rate on this part): sign, exponent rebiased by
// 1023 - 127, mantissa moved up 29 bits; a subnormal input a 2^-149 is
// normalised by its leading bit. Exact for every finite input.
__device__ __forceinline__ double f32_to_f64(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t a = u & 0x7fffffffu;
  const unsigned long long sgn = ((unsigned long long)(u >> 31)) << 63;
  unsigned long long d;
  if (a >= 0x00800000u) {
    d = ((unsigned long long)a + (896ull << 23)) << 29;
  } else if (a != 0u) {
    const int p = 31 - __clz(a);  // a = 2^p (1 + f), p < 23
    d = ((unsigned long long)(p - 149 + 1023) << 52) |
        (((unsigned long long)a << (52 - p)) & 0xfffffffffffffull);
  } else {
    d = 0ull;
  }
  return __longlong_as_double((long long)(sgn | d));
}

// ---------------------------------------------------------------------------
// BF16 helpers (round to nearest even).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint16_t bf16_bits(float x) {
  __nv_bfloat16 b = __float2bfloat16_rn(x);
  return *reinterpret_cast<uint16_t*>(&b);
}
__device__ __forceinline__ float bf16_val(uint16_t u) {
  return __uint_as_float(((uint32_t)u) << 16);
}

// FP16 helpers (round to nearest even).
__device__ __forceinline__ uint16_t fp16_bits(float x) {
  __half h = __float2half_rn(x);
  return *reinterpret_cast<uint16_t*>(&h);
}
__device__ __forceinline__ float fp16_val(uint16_t u) {
  return __half2float(*reinterpret_cast<const __half*>(&u));
}

// The fixed grid of the hi term of the BF16 three-term split: multiples of
// 1/8 in [-32, 32); every such value has at most 8 significant bits (exact in
// BF16) and sums of (integer count <= 256) x (hi) stay on the 1/8 grid, so
// FP32 accumulates them exactly while |sum| < 2^21.
constexpr float kHiScale = 8.0f;
constexpr float kHiMin = -32.0f;
constexpr float kHiMax = 32.0f - 0.125f;
// The FP16 two-term split: hi on the 1/64 grid in [-32, 32) (at most 11
// significant bits, exact in FP16); counts <= 2048 are exact in FP16 and the
// products and partial sums stay on the 1/64 grid, exact in FP32 while
// |sum| < 2^18.
constexpr float kHi16Scale = 64.0f;
constexpr float kHi16Max = 32.0f - 1.0f / 64.0f;
// Scores are split for the epilogues into a part on the 1/64 grid (every
// 1/8-grid value lies on it) and a small rest; references (maxima, lse) use
// the same grid so that subtracting them is exact.
constexpr float kGrid = 64.0f;
constexpr double kGridD = 64.0;
// FP16 responsibilities are stored scaled by 2^14 (P <= 1 stays below the
// FP16 maximum, P down to ~4e-9 stays normal); the update removes the scale.
constexpr float kP16Scale = 16384.0f;

// Duplicate pixel columns for counts above 256 (EMC_FLAG_WIDE_COUNTS): at most
// this many, each carrying up to kDupCount photons of its source pixel; their
// geometry entry has w = kDupMark (used pixels 1, padding 0).
constexpr int kDupCols = 64;
constexpr int kDupCount = 256;
constexpr float kDupMark = 2.0f;

// Gaussian model (Eqs. 2.2-2.3): S_jk <= log w_j < 0, and scores further than
// kGaussClamp below zero are clamped -- their exp vanishes next to any
// frame's best rotation, and the clamp keeps every score's 1/64-grid part
// exact in FP32.
constexpr float kGaussClamp = 120000.0f;

// Scale of the Gaussian contraction, from the grid maximum Wmax and the
// largest frame total Nmax (x: s, y: 1/s^2):
//   s  = the largest power of two with s Wmax Nmax <= 2^23 and s Wmax <= 2^15.
//        The integral hi part of s W is at most s Wmax + 1/2, so every partial
//        sum of hi K over a frame stays below 2^24 (exact in FP32) and hi
//        stays far inside the FP16 range.
__host__ __device__ inline float4 gauss_scales(float wmax, long long nmax) {
  if (!(wmax > 0.f) || !(wmax < 3.0e38f)) return make_float4(1.f, 1.f, 0.f, 0.f);
  const double w = (double)wmax, n = (double)(nmax > 0 ? nmax : 1);
  int e = ilogb(8388608.0 / (w * n));
  const int e2 = ilogb(32768.0 / w);
  e = e < e2 ? e : e2;
  e = e < -60 ? -60 : (e > 60 ? 60 : e);
  return make_float4((float)ldexp(1.0, e), (float)ldexp(1.0, -2 * e), 0.f, 0.f);
}

}  // namespace emc
