// expand_tile.cu -- e-step of EMC (Eq. 2.9), a quarter or
// an eighth of a row tile of 128 rotations and a slice of 256 pixels per CTA
// (small CTAs, so that small blocks of rotations fill the SMs and the last wave
// leaves few of them idle).
//
// Each thread owns two neighbouring pixels and takes the CTA's rotations in
// turn, so the pixels' geometry stays in registers and the rotations come from
// shared memory. Per (i, j): the grid point p = R_j q_i + N/2, the trilinear
// value of the model (Eq. 2.8, tent weights), W_ij = max(W, w_floor) and
// log W_ij in the layout of the chosen precision, written two pixels at a time
// (the Gaussian and Poisson-fluence models' own layouts below). The row sums sum_i W_ij of the bias
//   bias_j = log w_j - sum_i W_ij
// are kept as double-float pairs of FP32 (exact two-sums: FP64 is rare on
// this part, and a per-row FP64 reduction kept its pipe 65% busy). A warp
// parks its lanes' pairs of eight rows in shared memory and reduces them
// transposed (each lane sums a quarter of one row, two shuffles finish it),
// a quarter of the instructions of eight butterfly reductions; the CTA adds
// its warps' sums, and a second kernel the slices' partial sums in slice
// order (deterministic).
//
// The grid point is formed in fixed point (rotate_fx): exact 64-bit integer
// products for the large part, six FP32 FMAs for the rest (error ~1e-10
// voxel), the FP32 parts of the two pixels in one instruction. The voxel's
// eight corners come with one 32-byte load, asked for one rotation ahead.
//
// Bound by issue (68%; the FMA pipe next) and the load/store pipe (75%: the
// gathers). 64^3, 10880 rows x 2816 columns, under ncu: 306 us with 128
// rotations a CTA, scalar FP32 and two 16-byte gathers at the point of use (254
// instructions per element); 225 us with two-pixel instructions, rounding without
// the conversion pipe and 32 rotations a CTA (175); 215 us with 32-byte cells; 191 us
// with the gathers a rotation ahead. 32^3 with 3240 rotations: 223 -> 39 us. The
// Gaussian form: 260 us with one CTA per rotation in double-float arithmetic, 171 us here.
//
// With the last iteration's L (DELTA), the CTA also reads the previous planes
// of its elements and keeps, per pixel, the largest rise and fall of the
// represented log W over the tile's rows: the rows t and ntp + t of the
// incremental bound's increments D (prune.cu), rounded up to the operand type
// of the frames, and their magnitude bound A (the rows 2 ntp + t).
#include <cooperative_groups.h>

#include <algorithm>

#include "emc_common.cuh"
#include "emc_internal.h"

namespace cg = cooperative_groups;

namespace emc {

namespace {

constexpr int kTThreads = 128;
constexpr int kTRows = 128;  // rotations of a row tile
constexpr int kTPix = 2 * kTThreads;

// one rotation in shared memory, read as 16-byte words; the FP32 parts twice,
// as operands of two-pixel instructions
struct __align__(16) RowFX {
  int hi[12];
  float2 hf[9];  // hi as FP32 (hi 2^-20, exact)
  float2 lo[9];
};

// The grid points of a thread's two pixels: rotate_fx, bit for bit, in two-pixel
// FP32 instructions. The small part leaves a fraction outside [0, 1) only within
// 10^-3 of a voxel's face, so all six are looked at once and put right in a
// branch that few warps take.
__device__ __forceinline__ void rotate_pair(const RowFX& R, const int4* qi, const float2* qh,
                                            const float2* ql, long long centre, int (*f)[3],
                                            float (*t)[3]) {
  const float2 down = make_float2(0x1p-23f, 0x1p-23f), one = make_float2(-1.f, -1.f);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const float2 small = fma2(
        R.hf[3 * a], ql[0],
        fma2(R.hf[3 * a + 1], ql[1],
             fma2(R.hf[3 * a + 2], ql[2],
                  fma2(R.lo[3 * a], qh[0],
                       fma2(R.lo[3 * a + 1], qh[1], mul2(R.lo[3 * a + 2], qh[2]))))));
    float hi[2], lo[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      long long acc = centre;
      acc += (long long)R.hi[3 * a] * (long long)qi[u].x;
      acc += (long long)R.hi[3 * a + 1] * (long long)qi[u].y;
      acc += (long long)R.hi[3 * a + 2] * (long long)qi[u].z;
      f[u][a] = (int)(acc >> 32);
      const unsigned fw = (unsigned)(acc & 0xffffffffLL);
      hi[u] = __uint_as_float(0x3f800000u | (fw >> 9));
      lo[u] = __uint_as_float(0x3f800000u | ((fw & 511u) << 14));
    }
    const float2 fr = add2(add2(make_float2(hi[0], hi[1]), one),
                           fma2(add2(make_float2(lo[0], lo[1]), one), down, small));
    t[0][a] = fr.x;
    t[1][a] = fr.y;
  }
  const float least = fminf(fminf(fminf(t[0][0], t[0][1]), fminf(t[0][2], t[1][0])),
                            fminf(t[1][1], t[1][2]));
  const float most = fmaxf(fmaxf(fmaxf(t[0][0], t[0][1]), fmaxf(t[0][2], t[1][0])),
                           fmaxf(t[1][1], t[1][2]));
  if (least < 0.f || most >= 1.f) {
#pragma unroll
    for (int u = 0; u < 2; u++)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        if (t[u][a] < 0.f) {
          f[u][a] -= 1;
          t[u][a] += 1.f;
        } else if (t[u][a] >= 1.f) {
          f[u][a] += 1;
          t[u][a] -= 1.f;
        }
      }
  }
}

// x to the nearest multiple of 1 / scale (a power of two; ties to even), |x scale|
// below 2^22: by adding and taking away 1.5 2^23 (rintf is a conversion instruction)
__device__ __forceinline__ float round_to(float x, float scale) {
  return ((fmaf(x, scale, 12582912.f)) - 12582912.f) * (1.0f / scale);
}

template <bool INTERIOR>
__device__ __forceinline__ float trilinear_fx(const float* __restrict__ grid, int N, const int* f,
                                              const float* t) {
  const float wx[2] = {1.f - t[0], t[0]}, wy[2] = {1.f - t[1], t[1]}, wz[2] = {1.f - t[2], t[2]};
  float W = 0.f;
  if (INTERIOR) {
    const int nn = N * N;
    const float* g = grid + (f[0] * nn + f[1] * N + f[2]);
#pragma unroll
    for (int cx = 0; cx < 2; cx++)
#pragma unroll
      for (int cy = 0; cy < 2; cy++) {
        const float wxy = wx[cx] * wy[cy];
        const float* gr = g + cx * nn + cy * N;
        W = fmaf(wxy * wz[0], __ldg(gr), W);
        W = fmaf(wxy * wz[1], __ldg(gr + 1), W);
      }
    return W;
  }
  const int64_t nn = (int64_t)N * N;
#pragma unroll
  for (int c = 0; c < 8; c++) {
    const int x = f[0] + ((c >> 2) & 1), y = f[1] + ((c >> 1) & 1), z = f[2] + (c & 1);
    if (x < 0 || y < 0 || z < 0 || x >= N || y >= N || z >= N) continue;
    W = fmaf(wx[(c >> 2) & 1] * wy[(c >> 1) & 1] * wz[c & 1],
             __ldg(grid + (int64_t)x * nn + (int64_t)y * N + z), W);
  }
  return W;
}

// values of two elements of a split L (old planes, DELTA)
template <int PREC>
__device__ __forceinline__ float2 read_pair(const void* L, int64_t o, int64_t ps) {
  const uint16_t* b = (const uint16_t*)L;
  auto val = [&](int64_t oo) -> float2 {
    const uint32_t u = *reinterpret_cast<const uint32_t*>(b + oo);
    if (PREC == EMC_PREC_FP16_SPLIT)
      return make_float2(fp16_val((uint16_t)(u & 0xffffu)), fp16_val((uint16_t)(u >> 16)));
    return make_float2(bf16_val((uint16_t)(u & 0xffffu)), bf16_val((uint16_t)(u >> 16)));
  };
  float2 v = val(o);
  const int np = PREC == EMC_PREC_BF16_SPLIT ? 3 : 2;
  for (int q = 1; q < np; q++) {
    const float2 w = val(o + q * ps);
    v.x += w.x;  // planes of one element: their sum rounds at most twice
    v.y += w.y;
  }
  return v;
}

template <int PREC>
__device__ __forceinline__ uint16_t round_up_operand(float x) {
  if (PREC == EMC_PREC_FP16_SPLIT) {
    __half h = __float2half_ru(x);
    return *reinterpret_cast<uint16_t*>(&h);
  }
  __nv_bfloat16 b = __float2bfloat16_ru(x);
  return *reinterpret_cast<uint16_t*>(&b);
}

// What the expansion writes, beside the precisions' layouts of log W:
//  kOutGauss: s W as three FP16 planes (Gaussian model: no floor and no logarithm,
//    s = 2^e = gsc->x), hi integral (rint below 2048, else the FP16 rounding, itself
//    integral there), mid = fp16(s W - hi), lo = fp16(s W - hi - mid), the
//    representation error below 2^-23 s^-1 W units; the row sums are of W^2;
//  kOutW: W itself in FP32 (the Poisson-fluence model, whose split needs the row sum first),
//    its upper 16 bits in plane 0 and its lower ones in plane 1, and the slices' row sums
//    in plane 2, each at its row and slice (flu_split_kernel replaces all three in place).
constexpr int kOutGauss = 4, kOutW = 5;

// The rises dp and falls dm of a thread's two pixels over a tile's rows, gathered over the
// cluster's CTAs by its first one, into rows t, ntp + t and 2 ntp + t of D,
// rounded up to the operand type. rises: shared, one entry per thread.
template <int PREC>
__device__ __forceinline__ void write_increments(float (&dp)[2], float (&dm)[2], float4* rises,
                                                 bool inside, int64_t t, int64_t i0,
                                                 int64_t ld_pix, int64_t ntp,
                                                 uint16_t* __restrict__ D) {
  cg::cluster_group cluster = cg::this_cluster();
  rises[threadIdx.x] = make_float4(dp[0], dp[1], dm[0], dm[1]);
  cluster.sync();
  if (cluster.block_rank() == 0 && inside) {
    for (unsigned q = 1; q < cluster.num_blocks(); q++) {
      const float4 o = cluster.map_shared_rank(rises, q)[threadIdx.x];
      dp[0] = fmaxf(dp[0], o.x);
      dp[1] = fmaxf(dp[1], o.y);
      dm[0] = fmaxf(dm[0], o.z);
      dm[1] = fmaxf(dm[1], o.w);
    }
    float a[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      // the sum of the planes rounded at most twice: 2^-23 |d| covers it
      dp[u] += 2.0f * 1.1920929e-7f * fabsf(dp[u]);
      dm[u] += 2.0f * 1.1920929e-7f * fabsf(dm[u]);
      // bound of both rounded magnitudes (BF16 rounding up: at most 2^-7 relative)
      a[u] = fmaxf(fabsf(dp[u]), fabsf(dm[u])) * 1.0078125f;
    }
    const uint16_t p0 = round_up_operand<PREC>(dp[0]), p1 = round_up_operand<PREC>(dp[1]);
    const uint16_t m0 = round_up_operand<PREC>(dm[0]), m1 = round_up_operand<PREC>(dm[1]);
    const uint16_t a0 = round_up_operand<PREC>(a[0]), a1 = round_up_operand<PREC>(a[1]);
    *reinterpret_cast<uint32_t*>(D + t * ld_pix + i0) = (uint32_t)p0 | ((uint32_t)p1 << 16);
    *reinterpret_cast<uint32_t*>(D + (ntp + t) * ld_pix + i0) = (uint32_t)m0 | ((uint32_t)m1 << 16);
    *reinterpret_cast<uint32_t*>(D + (2 * ntp + t) * ld_pix + i0) =
        (uint32_t)a0 | ((uint32_t)a1 << 16);
  }
  cluster.sync();  // no CTA leaves while its rises may be read
}

// Two neighbouring elements of a 16-bit plane, in one access where WHOLE (the plane is
// 4-byte aligned; a caller's L of the Gaussian and Poisson-fluence models need not be. A
// flag in place of the template costs those 3 and 5%).
template <bool WHOLE>
__device__ __forceinline__ void put_pair(uint16_t* p, uint32_t v) {
  if (WHOLE) {
    *reinterpret_cast<uint32_t*>(p) = v;
  } else {
    p[0] = (uint16_t)v;
    p[1] = (uint16_t)(v >> 16);
  }
}
template <bool WHOLE>
__device__ __forceinline__ uint32_t get_pair(const uint16_t* p) {
  return WHOLE ? __ldcs(reinterpret_cast<const uint32_t*>(p)) : p[0] | (uint32_t)p[1] << 16;
}

// Eight bytes at a place of a 16-bit plane that need not be aligned to them.
__device__ __forceinline__ void put_bytes8(uint16_t* p, unsigned long long v) {
  if (((uintptr_t)p & 7) == 0) {
    *reinterpret_cast<unsigned long long*>(p) = v;
    return;
  }
#pragma unroll
  for (int k = 0; k < 4; k++) p[k] = (uint16_t)(v >> (16 * k));
}
__device__ __forceinline__ unsigned long long get_bytes8(const uint16_t* p) {
  if (((uintptr_t)p & 7) == 0) return *reinterpret_cast<const unsigned long long*>(p);
  unsigned long long v = 0;
#pragma unroll
  for (int k = 0; k < 4; k++) v |= (unsigned long long)p[k] << (16 * k);
  return v;
}

// s W as three FP16 planes (kOutGauss)
struct GaussSplit {
  uint16_t h, m, l;
};
__device__ __forceinline__ GaussSplit gauss_split(float x) {
  GaussSplit o;
  const float hi = x < 2048.f ? round_to(x, 1.f) : fp16_val(fp16_bits(x));
  const float r = x - hi;  // exact
  o.h = fp16_bits(hi);
  o.m = fp16_bits(r);
  o.l = fp16_bits(r - fp16_val(o.m));
  return o;
}

// RPC rotations of a tile per CTA; with DELTA the tile's 128 / RPC CTAs are a
// cluster, whose first one gathers the others' rises and falls.
template <int PREC, bool INTERIOR, bool DELTA, int RPC, bool WHOLE = true>
__global__ void __launch_bounds__(kTThreads, 6)
    expand_tile_kernel(const int4* __restrict__ qi_g, const float4* __restrict__ qlo_g,
                       int64_t ld_pix, int N, const float* __restrict__ grid,
                       const float4* __restrict__ g4,
                       const RotFX* __restrict__ rot, int64_t nrot, int64_t rows, float w_floor,
                       void* __restrict__ Lbase, int64_t ps, double* __restrict__ partial,
                       const void* __restrict__ Lold, uint16_t* __restrict__ D, int64_t ntp,
                       unsigned slices, const float4* __restrict__ gsc, int32_t* status) {
  static_assert(!DELTA || PREC == EMC_PREC_BF16_SPLIT || PREC == EMC_PREC_FP16_SPLIT,
                "increments: the contexts that prune");
  __shared__ RowFX R[RPC];
  __shared__ float2 rsum[kTThreads / 32][RPC];
  // eight rows of every lane's pair, rows padded to 33 so that the transposed
  // reads hit 16 distinct bank pairs per half warp
  __shared__ float2 park[kTThreads / 32][8 * 33];
  __shared__ float4 rises[DELTA ? kTThreads : 1];
  // a tile's CTAs are neighbours, then the slices, then the tiles
  constexpr unsigned kPer = kTRows / RPC;
  const unsigned slice = blockIdx.x / kPer % slices;
  const int64_t t = blockIdx.x / kPer / slices;
  const int64_t r0 = t * kTRows + blockIdx.x % kPer * RPC;
  const int nr = (int)max((int64_t)0, min((int64_t)RPC, nrot - r0));  // valid rows
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int x = threadIdx.x; x < RPC * 9; x += kTThreads) {
    const int r = x / 9, e = x % 9;
    int h = 0;
    float l = 0.f;
    if (r < nr) {
      h = rot[r0 + r].hi[e];
      l = rot[r0 + r].lo[e];
    }
    const float hf = (float)h * 0x1p-20f;
    R[r].hi[e] = h;
    R[r].hf[e] = make_float2(hf, hf);
    R[r].lo[e] = make_float2(l, l);
  }
  const int64_t i0 = (int64_t)slice * kTPix + 2 * threadIdx.x;
  const bool inside = i0 < ld_pix;  // ld_pix is even: both pixels or neither
  int4 qi[2];
  float2 qh[3], ql[3];
  {
    float4 l[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      qi[u] = inside ? qi_g[i0 + u] : make_int4(0, 0, 0, 0);
      l[u] = inside ? qlo_g[i0 + u] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    qh[0] = make_float2((float)qi[0].x * 0x1p-12f, (float)qi[1].x * 0x1p-12f);
    qh[1] = make_float2((float)qi[0].y * 0x1p-12f, (float)qi[1].y * 0x1p-12f);
    qh[2] = make_float2((float)qi[0].z * 0x1p-12f, (float)qi[1].z * 0x1p-12f);
    ql[0] = make_float2(l[0].x, l[1].x);
    ql[1] = make_float2(l[0].y, l[1].y);
    ql[2] = make_float2(l[0].z, l[1].z);
  }
  const long long centre = ((long long)(N >> 1) << 32) + ((N & 1) ? (1LL << 31) : 0LL);
  __syncthreads();
  float dp[2] = {-INFINITY, -INFINITY}, dm[2] = {-INFINITY, -INFINITY};
  int bad = 0, nonfinite = 0;
  const float gs = PREC == kOutGauss ? gsc->x : 1.f;
  // Row r + 1's grid points are formed and its voxels asked for before row r's
  // values are used: the gathers' latency is what the loop would wait for.
  float tt[2][3];
  Cell cell[2];
  auto fetch = [&](int r) {
    int f[2][3];
    rotate_pair(R[r], qi, qh, ql, centre, f, tt);
#pragma unroll
    for (int u = 0; u < 2; u++) {
      if (INTERIOR && g4)  // padding pixels and rows read the centre
        cell[u] = load_cell(g4, (f[u][0] * N + f[u][1]) * N + f[u][2]);
      else
        cell[u].a.x = r < nr && qi[u].w != 0 ? trilinear_fx<INTERIOR>(grid, N, f[u], tt[u]) : 0.f;
    }
  };
  fetch(0);
  for (int r = 0; r < RPC; r++) {
    const int64_t row = r0 + r;
    const bool vrow = r < nr;
    float W2[2];
#pragma unroll
    for (int u = 0; u < 2; u++)
      W2[u] = INTERIOR && g4 ? cell_value(cell[u], tt[u]) : cell[u].a.x;
    if (r + 1 < RPC) fetch(r + 1);
    float L[2] = {0.f, 0.f};
    float ws[2] = {0.f, 0.f}, we[2] = {0.f, 0.f};  // (kOutGauss: W^2 as ws + we)
#pragma unroll
    for (int u = 0; u < 2; u++) {
      if (vrow && qi[u].w != 0) {  // w: 1 pixel, 2 duplicate column, 0 padding / ones
        nonfinite |= !(fabsf(W2[u]) <= 3.4e38f);  // a NaN or infinite voxel of the model
        const float W = fmaxf(W2[u], w_floor);
        // duplicate columns repeat a pixel: not summed
        if (qi[u].w == 1) {
          ws[u] = PREC == kOutGauss ? W * W : W;
          if (PREC == kOutGauss) we[u] = fmaf(W, W, -ws[u]);
        }
        L[u] = PREC == kOutGauss ? W * gs : (PREC == kOutW ? W : logf(W));
      }
    }
    const f2 pair = two_sum(ws[0], ws[1]);  // row sum of the pair as s + se
    const float s = pair.h, se = PREC == kOutGauss ? pair.l + (we[0] + we[1]) : pair.l;
    if (inside && row < rows) {
      const int64_t o = row * ld_pix + i0;
      // DELTA: the change of the represented value (the planes' sum) of each element
      if (PREC == kOutGauss) {
        uint16_t h[2], m[2], l[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const GaussSplit g = gauss_split(L[u]);
          h[u] = g.h;
          m[u] = g.m;
          l[u] = g.l;
        }
        uint16_t* Lb = (uint16_t*)Lbase + o;
        put_pair<WHOLE>(Lb, (uint32_t)h[0] | ((uint32_t)h[1] << 16));
        put_pair<WHOLE>(Lb + ps, (uint32_t)m[0] | ((uint32_t)m[1] << 16));
        put_pair<WHOLE>(Lb + 2 * ps, (uint32_t)l[0] | ((uint32_t)l[1] << 16));
      } else if (PREC == kOutW) {
        const uint32_t u0 = __float_as_uint(L[0]), u1 = __float_as_uint(L[1]);
        uint16_t* Lb = (uint16_t*)Lbase + o;
        put_pair<WHOLE>(Lb, __byte_perm(u0, u1, 0x7632));
        put_pair<WHOLE>(Lb + ps, __byte_perm(u0, u1, 0x5410));
      } else if (PREC == EMC_PREC_FP32) {
        *reinterpret_cast<float2*>((float*)Lbase + o) = make_float2(L[0], L[1]);
      } else if (PREC == EMC_PREC_BF16) {
        const uint16_t b0 = bf16_bits(L[0]), b1 = bf16_bits(L[1]);
        *reinterpret_cast<uint32_t*>((uint16_t*)Lbase + o) = (uint32_t)b0 | ((uint32_t)b1 << 16);
      } else if (PREC == EMC_PREC_FP16_SPLIT) {
        uint16_t h[2], rr[2];
        float v[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          float hi = round_to(L[u], kHi16Scale);
          if (vrow && qi[u].w != 0 && (hi < kHiMin || hi > kHi16Max)) bad = 1;
          hi = fminf(fmaxf(hi, kHiMin), kHi16Max);
          h[u] = fp16_bits(hi);
          rr[u] = fp16_bits(L[u] - hi);
          v[u] = hi + fp16_val(rr[u]);
        }
        uint16_t* Lb = (uint16_t*)Lbase + o;
        *reinterpret_cast<uint32_t*>(Lb) = (uint32_t)h[0] | ((uint32_t)h[1] << 16);
        *reinterpret_cast<uint32_t*>(Lb + ps) = (uint32_t)rr[0] | ((uint32_t)rr[1] << 16);
        if (DELTA && vrow) {
          const float2 old = read_pair<PREC>(Lold, o, ps);
          const float d0 = v[0] - old.x, d1 = v[1] - old.y;
          dp[0] = fmaxf(dp[0], d0); dm[0] = fmaxf(dm[0], -d0);
          dp[1] = fmaxf(dp[1], d1); dm[1] = fmaxf(dm[1], -d1);
        }
      } else {
        // three-term split: hi on the 1/8 grid, residual r = mid + lo
        uint16_t h[2], m[2], l[2];
        float v[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          float hi = round_to(L[u], kHiScale);
          if (vrow && qi[u].w != 0 && (hi < kHiMin || hi > kHiMax)) bad = 1;
          hi = fminf(fmaxf(hi, kHiMin), kHiMax);
          const float r = L[u] - hi;  // exact
          m[u] = bf16_bits(r);
          l[u] = bf16_bits(r - bf16_val(m[u]));
          h[u] = bf16_bits(hi);
          v[u] = (hi + bf16_val(m[u])) + bf16_val(l[u]);
        }
        uint16_t* Lb = (uint16_t*)Lbase + o;
        *reinterpret_cast<uint32_t*>(Lb) = (uint32_t)h[0] | ((uint32_t)h[1] << 16);
        *reinterpret_cast<uint32_t*>(Lb + ps) = (uint32_t)m[0] | ((uint32_t)m[1] << 16);
        *reinterpret_cast<uint32_t*>(Lb + 2 * ps) = (uint32_t)l[0] | ((uint32_t)l[1] << 16);
        if (DELTA && vrow) {
          const float2 old = read_pair<PREC>(Lold, o, ps);
          const float d0 = v[0] - old.x, d1 = v[1] - old.y;
          dp[0] = fmaxf(dp[0], d0); dm[0] = fmaxf(dm[0], -d0);
          dp[1] = fmaxf(dp[1], d1); dm[1] = fmaxf(dm[1], -d1);
        }
      }
    }
    // row sums: park the pair; every eighth row, lane l sums eight lanes'
    // pairs of row l mod 8, and the lanes l, l ^ 8, l ^ 16, l ^ 24 combine
    float2* pk = park[warp];
    pk[(r & 7) * 33 + lane] = make_float2(s, se);
    if ((r & 7) == 7) {
      __syncwarp();
      const float2* src = pk + (lane & 7) * 33 + (lane >> 3) * 8;
      float a = 0.f, ae = 0.f;
#pragma unroll
      for (int m = 0; m < 8; m++) {
        const float2 v = src[m];
        const f2 z = two_sum(a, v.x);
        a = z.h;
        ae += v.y + z.l;
      }
#pragma unroll
      for (int off = 8; off <= 16; off <<= 1) {
        const float ao = __shfl_xor_sync(0xffffffffu, a, off);
        const float eo = __shfl_xor_sync(0xffffffffu, ae, off);
        const f2 z = two_sum(a, ao);
        a = z.h;
        ae += eo + z.l;
      }
      if (lane < 8) rsum[warp][r - 7 + lane] = make_float2(a, ae);
      __syncwarp();
    }
  }
  if (nonfinite) set_status(status, EMC_ERR_NUMERIC);
  if (bad) set_status(status, EMC_ERR_UNSUPPORTED);
  __syncthreads();
  if (threadIdx.x < RPC) {
    float s = 0.f, se = 0.f;
    if ((int)threadIdx.x < nr)
      for (int w = 0; w < kTThreads / 32; w++) {
        const float2 v = rsum[w][threadIdx.x];
        const f2 a = two_sum(s, v.x);
        s = a.h;
        se += v.y + a.l;
      }
    const double sum = f32_to_f64(s) + f32_to_f64(se);
    if (PREC == kOutW)
      put_bytes8((uint16_t*)Lbase + 2 * ps + (r0 + threadIdx.x) * ld_pix + (int64_t)slice * kTPix,
                 (unsigned long long)__double_as_longlong(sum));
    else
      partial[(int64_t)slice * rows + r0 + threadIdx.x] = sum;
  }
  if constexpr (DELTA)
    write_increments<PREC>(dp, dm, rises, inside, t, i0, ld_pix, ntp, D);
}

// bias_j = log w_j - scale (sum of the slices' partial sums, in slice order); with
// the last iteration's bias, the tile's largest rise and fall of it into
// bpm[t], bpm[nt + t] (rounded up). One CTA of 128 threads per row tile.
__global__ void __launch_bounds__(kTRows)
    expand_bias_kernel(const double* __restrict__ partial, int n_slices, int64_t rows,
                       const double* __restrict__ logw, int64_t nrot, double scale,
                       double* __restrict__ bias, const double* __restrict__ bias_old, float* __restrict__ bpm, int64_t nt) {
  __shared__ double rp[kTRows], rm[kTRows];
  const int64_t row = (int64_t)blockIdx.x * kTRows + threadIdx.x;
  double s = 0.0;
  for (int c = 0; c < n_slices; c++) s += partial[(int64_t)c * rows + row];
  const bool v = row < nrot;
  const double b = v ? logw[row] - s * scale : -INFINITY;
  bias[row] = b;
  if (!bias_old) return;
  const double d = v ? b - bias_old[row] : 0.0;
  rp[threadIdx.x] = v ? d : -INFINITY;
  rm[threadIdx.x] = v ? -d : -INFINITY;
  __syncthreads();
  for (int w = kTRows / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      rp[threadIdx.x] = fmax(rp[threadIdx.x], rp[threadIdx.x + w]);
      rm[threadIdx.x] = fmax(rm[threadIdx.x], rm[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    bpm[blockIdx.x] = __double2float_ru(rp[0]);
    bpm[nt + blockIdx.x] = __double2float_ru(rm[0]);
  }
}

// Poisson-fluence model: L_ij = log(W_ij / B_j) + c with B_j = sum_i W_ij,
// so that sum_i K_ik L_ij = sum_i K_ik log W_ij - N_k log B_j + c N_k, the
// scores of the maximum-likelihood fluence phi_jk = N_k / B_j up to the
// per-frame shift c N_k (removed in FP64 by the log-sum-exp merge). B_j is
// needed before the first L is written, so the expansion writes W in FP32
// (kOutW) first. a_j = c - log B_j is carried as ah (1/8 grid) + al: x + ah is
// formed with its exact rounding error e (two-sum), hi is the 1/8-grid rounding
// of the whole x + ah + e + al, and the rest r = ((x + ah - hi) + e) + al goes
// to mid + lo. No per-rotation rounding of a_j enters the contraction (it would
// be multiplied by N_k), and the rest stays centred on zero: were al left in
// every rest, the mid/lo accumulator would grow to N_k al and round at that
// size on every K step.
//
// c - log B as ah (1/8 grid) + al
__device__ __forceinline__ float2 flu_shift_split(double c, double B, bool valid) {
  const double aj = valid ? c - log(B) : 0.0;
  const float ah = (float)(rint(aj * kHiScale) / kHiScale);
  return make_float2(ah, (float)(aj - (double)ah));
}

// Per row: bias = log w_j (-inf on padding rows), B_j (0) into Bsum and Bctx, and
// (ah, al) over the row's partial sums (low: plane 2), one copy for each slice.
__global__ void __launch_bounds__(kTRows)
    flu_bias_kernel(uint16_t* __restrict__ low, int64_t ld_pix, int n_slices,
                    const double* __restrict__ logw, int64_t nrot, double c,
                    double* __restrict__ bias, double* __restrict__ Bsum,
                    double* __restrict__ Bctx, float* __restrict__ bpm, int64_t nt) {
  const int64_t row = (int64_t)blockIdx.x * kTRows + threadIdx.x;
  uint16_t* own = low + row * ld_pix;
  double B = 0.0;
  // (a sum's sector is its own: sixteen loads in flight)
  for (int q0 = 0; q0 < n_slices; q0 += 16) {
    unsigned long long part[16];
#pragma unroll
    for (int u = 0; u < 16; u++)
      part[u] = q0 + u < n_slices ? get_bytes8(own + (int64_t)(q0 + u) * kTPix) : 0ull;
#pragma unroll
    for (int u = 0; u < 16; u++) B += __longlong_as_double((long long)part[u]);
  }
  const bool v = row < nrot;
  const float2 as = flu_shift_split(c, B, v);
  const unsigned long long a =
      (unsigned long long)__float_as_uint(as.y) << 32 | __float_as_uint(as.x);
  for (int q = 0; q < n_slices; q++) put_bytes8(own + (int64_t)q * kTPix, a);
  bias[row] = v ? logw[row] : -INFINITY;
  Bsum[row] = v ? B : 0.0;
  Bctx[row] = v ? B : 0.0;
  if (bpm && threadIdx.x == 0) bpm[blockIdx.x] = bpm[nt + blockIdx.x] = 0.f;  // log w stays
}

struct FluSplit {
  uint16_t h, m, l;
  bool bad;
};
__device__ __forceinline__ FluSplit flu_split(float W, bool used, float ah, float al) {
  FluSplit o;
  float hi = 0.f, rest = 0.f;
  o.bad = false;
  if (used) {
    const float x = logf(W);
    const float s = x + ah;  // two-sum: s + e = x + ah exactly
    const float bb = s - x;
    const float e = (x - (s - bb)) + (ah - bb);
    hi = round_to(s + (e + al), kHiScale);
    o.bad = hi < kHiMin || hi > kHiMax;
    hi = fminf(fmaxf(hi, kHiMin), kHiMax);
    rest = ((s - hi) + e) + al;
  }
  o.h = bf16_bits(hi);
  o.m = bf16_bits(rest);
  o.l = bf16_bits(rest - bf16_val(o.m));
  return o;
}

// W to the three BF16 planes of L in place, and with DELTA the increments from the last
// iteration's planes (as expand_tile_kernel; the CTAs of a tile are a cluster).
// Bound by memory and the latency of its short rows: 4 B of W and 6 B of planes read, 6 B
// written per element, 3.9 TB/s with eight rows' loads in flight (one by one: 3.3).
// 96^3, 25728 rows x 7168 columns: W 970 us + split 788 us; one CTA per rotation in
// double-float arithmetic and a pass of its own for the increments took 1790 + 474 us.
constexpr int kSplitRows = 32;
template <bool DELTA, bool WHOLE = true>
__global__ void __launch_bounds__(kTThreads)
    flu_split_kernel(const int4* __restrict__ qi_g, int64_t ld_pix, int64_t nrot,
                     uint16_t* __restrict__ Lbase, int64_t ps, const uint16_t* __restrict__ Lold,
                     uint16_t* __restrict__ D, int64_t ntp, unsigned slices, int32_t* status) {
  __shared__ float4 rises[DELTA ? kTThreads : 1];
  __shared__ float2 asplit[kSplitRows];
  constexpr unsigned kPer = kTRows / kSplitRows;
  const unsigned slice = blockIdx.x / kPer % slices;
  const int64_t t = blockIdx.x / kPer / slices;
  const int64_t r0 = t * kTRows + blockIdx.x % kPer * kSplitRows;
  const int64_t i0 = (int64_t)slice * kTPix + 2 * threadIdx.x;
  const bool inside = i0 < ld_pix;
  bool used[2];
#pragma unroll
  for (int u = 0; u < 2; u++) used[u] = inside && qi_g[i0 + u].w != 0;
  constexpr int kAhead = 8;  // rows whose loads are in flight together
  uint32_t wh[kAhead], wl[kAhead];  // W's upper and lower halves
  uint32_t old[DELTA ? kAhead : 1][3];
  auto load = [&](int rb) {
#pragma unroll
    for (int r = 0; r < kAhead; r++) {
      const int64_t o = (r0 + rb + r) * ld_pix + i0;
      wh[r] = get_pair<WHOLE>(Lbase + o);
      wl[r] = get_pair<WHOLE>(Lbase + o + ps);
      if (DELTA)
#pragma unroll
        for (int q = 0; q < 3; q++)
          old[r][q] = __ldcs(reinterpret_cast<const uint32_t*>(Lold + o + q * ps));
    }
  };
  unsigned long long a = 0;
  if (threadIdx.x < kSplitRows)  // this slice's copy, before it is written over
    a = get_bytes8(Lbase + 2 * ps + (r0 + threadIdx.x) * ld_pix + (int64_t)slice * kTPix);
  if (inside) load(0);
  if (threadIdx.x < kSplitRows)
    asplit[threadIdx.x] =
        make_float2(__uint_as_float((uint32_t)a), __uint_as_float((uint32_t)(a >> 32)));
  __syncthreads();
  float dp[2] = {-INFINITY, -INFINITY}, dm[2] = {-INFINITY, -INFINITY};
  int bad = 0;
  if (inside) {
#pragma unroll 1
    for (int rb = 0; rb < kSplitRows; rb += kAhead) {
      if (rb > 0) load(rb);
#pragma unroll
      for (int r = 0; r < kAhead; r++) {
        const int64_t row = r0 + rb + r, o = row * ld_pix + i0;
        const bool vrow = row < nrot;
        const float2 aj = asplit[rb + r];
        const float ah = aj.x, al = aj.y;
        uint16_t h[2], m[2], l[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const FluSplit f =
              flu_split(__uint_as_float(__byte_perm(wl[r], wh[r], u ? 0x7632 : 0x5410)),
                        vrow && used[u], ah, al);
          h[u] = f.h;
          m[u] = f.m;
          l[u] = f.l;
          bad |= f.bad;
        }
        uint16_t* Lb = Lbase + o;
        put_pair<WHOLE>(Lb, (uint32_t)h[0] | ((uint32_t)h[1] << 16));
        put_pair<WHOLE>(Lb + ps, (uint32_t)m[0] | ((uint32_t)m[1] << 16));
        put_pair<WHOLE>(Lb + 2 * ps, (uint32_t)l[0] | ((uint32_t)l[1] << 16));
        if (DELTA && vrow) {
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const int sh = 16 * u;
            // the difference of each plane is exact in FP32; their sum rounds at most twice
            float d = bf16_val(h[u]) - bf16_val((uint16_t)(old[r][0] >> sh));
            d += bf16_val(m[u]) - bf16_val((uint16_t)(old[r][1] >> sh));
            d += bf16_val(l[u]) - bf16_val((uint16_t)(old[r][2] >> sh));
            dp[u] = fmaxf(dp[u], d);
            dm[u] = fmaxf(dm[u], -d);
          }
        }
      }
    }
  }
  if (bad) set_status(status, EMC_ERR_UNSUPPORTED);
  if constexpr (DELTA)
    write_increments<EMC_PREC_BF16_SPLIT>(dp, dm, rises, inside, t, i0, ld_pix, ntp, D);
}

// The whole Poisson-fluence expansion of small problems in one launch, and the
// Gaussian one (OUT: kOutW, kOutGauss), a CTA of TH threads per rotation, with W
// in shared memory: the tile kernels' launches leave most SMs idle there and each
// waits for the one before. TH / 128 slices of 256 pixels at a time; the sums in
// the order of the other form, so the bits are the same whichever runs. Bound by the
// latency of a slice's chain of loads: 384 threads where the SMs hold all rows' CTAs at
// once, 128 (ten CTAs an SM) where they do not (row_threads).
constexpr int kRowSlices = 40;  // 40 KB of W
template <int TH>
constexpr int row_ctas() {  // an SM
  return TH == 128 ? 10 : 3;
}
template <int OUT, int TH, bool INTERIOR, bool WHOLE>
__global__ void __launch_bounds__(TH, row_ctas<TH>())
    expand_row_kernel(const int4* __restrict__ qi_g, const float4* __restrict__ qlo_g,
                      int64_t ld_pix, int N, const float* __restrict__ grid,
                      const float4* __restrict__ g4, const RotFX* __restrict__ rot,
                      const double* __restrict__ logw, int64_t nrot, float w_floor, double c,
                      const float4* __restrict__ gsc, int slices, uint16_t* __restrict__ Lbase,
                      int64_t ps, double* __restrict__ bias, double* __restrict__ Bsum,
                      double* __restrict__ Bctx, int32_t* status) {
  extern __shared__ float2 wrow[];  // W of the row, a pixel pair an entry
  __shared__ RowFX R;
  __shared__ float2 rs[kRowSlices][kTThreads / 32];
  __shared__ double part[kRowSlices];
  __shared__ float2 as;
  const int64_t row = blockIdx.x;
  const bool valid = row < nrot;
  const int lane = threadIdx.x & 31, tt = threadIdx.x & (kTThreads - 1);
  if (threadIdx.x < 9) {
    const int e = threadIdx.x;
    const int h = valid ? rot[row].hi[e] : 0;
    const float l = valid ? rot[row].lo[e] : 0.f;
    const float hf = (float)h * 0x1p-20f;
    R.hi[e] = h;
    R.hf[e] = make_float2(hf, hf);
    R.lo[e] = make_float2(l, l);
  }
  const long long centre = ((long long)(N >> 1) << 32) + ((N & 1) ? (1LL << 31) : 0LL);
  __syncthreads();
  const float gs = OUT == kOutGauss ? gsc->x : 1.f;
  uint16_t* Lrow = Lbase + row * ld_pix;
  int nonfinite = 0;
  for (int sl = threadIdx.x / kTThreads; valid && sl < slices; sl += TH / kTThreads) {
    const int64_t i0 = (int64_t)sl * kTPix + 2 * tt;
    const bool inside = i0 < ld_pix;
    int4 qi[2];
    float4 q[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      qi[u] = inside ? qi_g[i0 + u] : make_int4(0, 0, 0, 0);
      q[u] = inside ? qlo_g[i0 + u] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float2 qh[3] = {make_float2((float)qi[0].x * 0x1p-12f, (float)qi[1].x * 0x1p-12f),
                          make_float2((float)qi[0].y * 0x1p-12f, (float)qi[1].y * 0x1p-12f),
                          make_float2((float)qi[0].z * 0x1p-12f, (float)qi[1].z * 0x1p-12f)};
    const float2 ql[3] = {make_float2(q[0].x, q[1].x), make_float2(q[0].y, q[1].y),
                          make_float2(q[0].z, q[1].z)};
    int f[2][3];
    float t[2][3], L[2], ws[2], we[2] = {0.f, 0.f};
    rotate_pair(R, qi, qh, ql, centre, f, t);
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const bool used = qi[u].w != 0;
      float W = 0.f;
      if (INTERIOR && g4)
        W = cell_value(load_cell(g4, (f[u][0] * N + f[u][1]) * N + f[u][2]), t[u]);
      else if (used)
        W = trilinear_fx<INTERIOR>(grid, N, f[u], t[u]);
      nonfinite |= used && !(fabsf(W) <= 3.4e38f);
      W = fmaxf(W, w_floor);
      ws[u] = used && qi[u].w == 1 ? (OUT == kOutGauss ? W * W : W) : 0.f;
      if (OUT == kOutGauss && used && qi[u].w == 1) we[u] = fmaf(W, W, -ws[u]);
      L[u] = used ? W * gs : 0.f;
    }
    if (OUT == kOutW && inside) wrow[i0 / 2] = make_float2(L[0], L[1]);
    if (OUT == kOutGauss && inside) {
      const GaussSplit x = gauss_split(L[0]), y = gauss_split(L[1]);
      put_pair<WHOLE>(Lrow + i0, (uint32_t)x.h | ((uint32_t)y.h << 16));
      put_pair<WHOLE>(Lrow + i0 + ps, (uint32_t)x.m | ((uint32_t)y.m << 16));
      put_pair<WHOLE>(Lrow + i0 + 2 * ps, (uint32_t)x.l | ((uint32_t)y.l << 16));
    }
    f2 pair = two_sum(ws[0], ws[1]);
    if (OUT == kOutGauss) pair.l += we[0] + we[1];
    float a = 0.f, ae = 0.f;
#pragma unroll
    for (int m = 0; m < 8; m++) {  // eight lanes' pairs, then the four sums of them
      const float x = __shfl_sync(0xffffffffu, pair.h, (lane & 24) + m);
      const float y = __shfl_sync(0xffffffffu, pair.l, (lane & 24) + m);
      const f2 z = two_sum(a, x);
      a = z.h;
      ae += y + z.l;
    }
#pragma unroll
    for (int off = 8; off <= 16; off <<= 1) {
      const float ao = __shfl_xor_sync(0xffffffffu, a, off);
      const float eo = __shfl_xor_sync(0xffffffffu, ae, off);
      const f2 z = two_sum(a, ao);
      a = z.h;
      ae += eo + z.l;
    }
    if (lane == 0) rs[sl][tt >> 5] = make_float2(a, ae);
  }
  __syncthreads();
  if ((int)threadIdx.x < slices) {
    float s = 0.f, se = 0.f;
    for (int w = 0; valid && w < kTThreads / 32; w++) {
      const float2 v = rs[threadIdx.x][w];
      const f2 a = two_sum(s, v.x);
      s = a.h;
      se += v.y + a.l;
    }
    part[threadIdx.x] = f32_to_f64(s) + f32_to_f64(se);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double B = 0.0;
    for (int q = 0; q < slices; q++) B += part[q];
    if (OUT == kOutGauss) {  // c: 1 / 2 sigma^2
      bias[row] = valid ? logw[row] - B * c : -INFINITY;
    } else {
      as = flu_shift_split(c, B, valid);
      bias[row] = valid ? logw[row] : -INFINITY;
      Bsum[row] = valid ? B : 0.0;
      Bctx[row] = valid ? B : 0.0;
    }
  }
  if (OUT == kOutGauss) {
    if (!valid)  // (a padding row: the loop above left it)
      for (int64_t i0 = 2 * threadIdx.x; i0 < ld_pix; i0 += 2 * TH)
        for (int q = 0; q < 3; q++) put_pair<WHOLE>(Lrow + i0 + q * ps, 0u);
    if (nonfinite) set_status(status, EMC_ERR_NUMERIC);
    return;
  }
  __syncthreads();
  const float ah = as.x, al = as.y;
  int bad = 0;
  for (int64_t i0 = 2 * threadIdx.x; i0 < ld_pix; i0 += 2 * TH) {
    const float2 W = valid ? wrow[i0 / 2] : make_float2(0.f, 0.f);
    const FluSplit x = flu_split(W.x, valid && qi_g[i0].w != 0, ah, al);
    const FluSplit y = flu_split(W.y, valid && qi_g[i0 + 1].w != 0, ah, al);
    bad |= x.bad || y.bad;
    uint16_t* Lb = Lrow + i0;
    put_pair<WHOLE>(Lb, (uint32_t)x.h | ((uint32_t)y.h << 16));
    put_pair<WHOLE>(Lb + ps, (uint32_t)x.m | ((uint32_t)y.m << 16));
    put_pair<WHOLE>(Lb + 2 * ps, (uint32_t)x.l | ((uint32_t)y.l << 16));
  }
  if (nonfinite) set_status(status, EMC_ERR_NUMERIC);
  if (bad) set_status(status, EMC_ERR_UNSUPPORTED);
}

// the grid in the cell layout of load_cell
__global__ void grid_cells_kernel(const float* __restrict__ g, int N, float4* __restrict__ g4) {
  const int64_t n3 = (int64_t)N * N * N;
  const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n3) return;
  const int z = (int)(l % N), y = (int)((l / N) % N);
  const bool zi = z + 1 < N, yi = y + 1 < N;
  const int64_t m = l + (int64_t)N * N;
  const bool xi = m < n3;
  g4[2 * l] = make_float4(g[l], zi ? g[l + 1] : 0.f, yi ? g[l + N] : 0.f,
                          (zi && yi) ? g[l + N + 1] : 0.f);
  g4[2 * l + 1] = make_float4(xi ? g[m] : 0.f, xi && zi ? g[m + 1] : 0.f,
                              xi && yi ? g[m + N] : 0.f, (xi && zi && yi) ? g[m + N + 1] : 0.f);
}

// fixed-point pixel geometry from the double-float one
__global__ void fixed_geometry_kernel(const float4* __restrict__ qh, const float4* __restrict__ ql,
                                      int64_t ld_pix, int4* __restrict__ qi,
                                      float4* __restrict__ qlo, float4* __restrict__ qf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ld_pix) return;
  const float4 a = qh[i], b = ql[i];
  const double q[3] = {(double)a.x + (double)b.x, (double)a.y + (double)b.y,
                       (double)a.z + (double)b.z};
  int h[3];
  float l[3];
  for (int c = 0; c < 3; c++) {
    const double r = rint(q[c] * 4096.0);
    h[c] = (int)r;
    l[c] = (float)(q[c] - r / 4096.0);
  }
  qi[i] = make_int4(h[0], h[1], h[2], (int)a.w);
  qlo[i] = make_float4(l[0], l[1], l[2], 0.f);
  if (qf) qf[i] = make_float4((float)h[0] * 0x1p-12f, (float)h[1] * 0x1p-12f,
                              (float)h[2] * 0x1p-12f, 0.f);
}

}  // namespace

int64_t expand_tile_slices(int64_t ld_pix) { return (ld_pix + kTPix - 1) / kTPix; }

cudaError_t launch_grid_cells(const float* grid, int N, float4* g4, cudaStream_t s) {
  const int64_t n3 = (int64_t)N * N * N;
  grid_cells_kernel<<<(unsigned)((n3 + 255) / 256), 256, 0, s>>>(grid, N, g4);
  return cudaGetLastError();
}

cudaError_t launch_fixed_geometry(const float4* qh, const float4* ql, int64_t ld_pix, int4* qi,
                                  float4* qlo, float4* qf, cudaStream_t s) {
  fixed_geometry_kernel<<<(unsigned)((ld_pix + 255) / 256), 256, 0, s>>>(qh, ql, ld_pix, qi, qlo,
                                                                        qf);
  return cudaGetLastError();
}

namespace {

// The expansion of rows (a multiple of 128) rotations in the layout `out` (a
// precision, kOutGauss or kOutW), and the slices' partial row sums.
cudaError_t launch_tiles(const Geom& g, const float* grid, const float4* g4, const RotFX* rot,
                         int64_t nrot, int64_t rows, int out, float w_floor, Planes L,
                         double* partial, const void* Lold, uint16_t* D, int64_t ntp,
                         const float4* gsc, int32_t* status, cudaStream_t s) {
  const int64_t nt = rows / kTRows;
  const int64_t ns = expand_tile_slices(g.ld_pix);
  const bool delta = Lold != nullptr;
  // 32 rotations a CTA (a quarter tile: small CTAs, so that the last wave of the
  // grid leaves few SMs idle), 16 where those would not give every SM its six
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool whole = ((uintptr_t)L.base & 3) == 0 || (out != kOutGauss && out != kOutW);
  const int rpc = ns * nt * 4 < 6 * (int64_t)sms || !whole ? 16 : 32;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)(ns * nt * (kTRows / rpc)));
  lc.blockDim = dim3(kTThreads);
  lc.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)(kTRows / rpc);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  lc.attrs = &at;
  lc.numAttrs = delta ? 1 : 0;
  cudaError_t e = cudaSuccess;
#define EMC_TILE_R(P, I, DL, ...)                                                              \
  e = cudaLaunchKernelEx(&lc, expand_tile_kernel<P, I, DL, __VA_ARGS__>, g.qi, g.qlo, g.ld_pix, g.N,    \
                         grid, g4, rot, nrot, rows, w_floor, L.base, L.plane_stride, partial,  \
                         Lold, D, ntp, (unsigned)ns, gsc, status)
#define EMC_TILE(P, I, DL)                   \
  do {                                       \
    if (rpc == 16) EMC_TILE_R(P, I, DL, 16); \
    else EMC_TILE_R(P, I, DL, 32);           \
  } while (0)
#define EMC_TILE_P(P)                          \
  if (g.interior) {                            \
    if (delta) EMC_TILE(P, true, true);        \
    else EMC_TILE(P, true, false);             \
  } else {                                     \
    if (delta) EMC_TILE(P, false, true);       \
    else EMC_TILE(P, false, false);            \
  }
#define EMC_TILE_O(P) /* no increments */      \
  do {                                         \
    if (g.interior) EMC_TILE(P, true, false);  \
    else EMC_TILE(P, false, false);            \
  } while (0);
#define EMC_TILE_L(P) /* any address of L */                     \
  if (whole) EMC_TILE_O(P)                                       \
  else if (g.interior) EMC_TILE_R(P, true, false, 16, false);    \
  else EMC_TILE_R(P, false, false, 16, false)
  switch (out) {
    case EMC_PREC_FP32: EMC_TILE_O(EMC_PREC_FP32); break;
    case EMC_PREC_BF16: EMC_TILE_O(EMC_PREC_BF16); break;
    case kOutGauss: EMC_TILE_L(kOutGauss); break;
    case kOutW: EMC_TILE_L(kOutW); break;
    case EMC_PREC_FP16_SPLIT: EMC_TILE_P(EMC_PREC_FP16_SPLIT); break;
    default: EMC_TILE_P(EMC_PREC_BF16_SPLIT); break;
  }
#undef EMC_TILE_L
#undef EMC_TILE_O
#undef EMC_TILE_P
#undef EMC_TILE
#undef EMC_TILE_R
  return e;
}

}  // namespace

cudaError_t launch_expand_tile(const Geom& g, const float* grid, const float4* g4,
                               const RotFX* rot,
                               const double* logw, int64_t nrot, int64_t rows, int precision,
                               float w_floor, Planes L, double* bias, double* partial,
                               const void* Lold, const double* bias_old, uint16_t* D, int64_t ntp,
                               float* bpm, int32_t* status, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  // increments: the split precisions (the contexts that prune)
  if (Lold && precision != EMC_PREC_BF16_SPLIT && precision != EMC_PREC_FP16_SPLIT)
    return cudaErrorInvalidValue;
  cudaError_t e = launch_tiles(g, grid, g4, rot, nrot, rows, precision, w_floor, L, partial, Lold,
                               D, ntp, nullptr, status, s);
  if (e != cudaSuccess) return e;
  const int64_t nt = rows / kTRows;
  expand_bias_kernel<<<(unsigned)nt, kTRows, 0, s>>>(
      partial, (int)expand_tile_slices(g.ld_pix), rows, logw, nrot, 1.0, bias,
      Lold ? bias_old : nullptr, bpm, nt);
  return cudaGetLastError();
}

namespace {

// Threads a rotation of the one-launch form, or 0 for the tile kernels. us of a call by the
// tile kernels, 384 and 128 threads a rotation (rows x columns):
//   512 x 832 39, 19, 21    512 x 3264 48, 31, 42     512 x 7296 73, 56, 89
//   1408 x 832 45, 38, 27   1408 x 3264 68, 74, 67    1408 x 7296 120, 138, 181
//   3328 x 832 56, 66, 48   3328 x 1856 81, 93, 82    10880 x 128 48, -, about 57
// (one CTA of 256 threads a rotation and a double-float grid point, before the tile kernels:
// 19, 36 and 66; 31, 66 and 132; 54 and 81)
int row_threads(int64_t rows, int64_t ns) {
  if (ns > kRowSlices) return 0;
  if (rows <= 512) return 384;
  return rows <= 4096 && rows * ns <= 16384 ? 128 : 0;
}

// The Gaussian model has one launch less to save (the scales come first in any form):
//   512 x 128 31, 21, 21   512 x 3264 44, 44, 49   128 x 9536 55, 60, 96
//   1408 x 832 36, 38, 33  3328 x 128 33, 40, 28   3328 x 832 46, 58, 48
// (before the tile kernels 21, 46 and 82; 34, 36 and 48)
int gauss_row_threads(int64_t rows, int64_t ns) {
  if (rows <= 512) return ns <= 16 ? 384 : 0;
  return rows <= 4096 && rows * ns <= 6144 ? 128 : 0;
}

template <int OUT>
cudaError_t launch_rows(int threads, const Geom& g, const float* grid, const float4* g4,
                        const RotFX* rot, const double* logw, int64_t nrot, int64_t rows,
                        float w_floor, double c, const float4* gsc, Planes L, double* bias,
                        double* Bsum, double* Bctx, int32_t* status, cudaStream_t s) {
  const bool whole = ((uintptr_t)L.base & 3) == 0;
  if (!whole) threads = 128;
  auto kern = threads == 384 ? (g.interior ? expand_row_kernel<OUT, 384, true, true>
                                           : expand_row_kernel<OUT, 384, false, true>)
              : whole        ? (g.interior ? expand_row_kernel<OUT, 128, true, true>
                                           : expand_row_kernel<OUT, 128, false, true>)
                             : (g.interior ? expand_row_kernel<OUT, 128, true, false>
                                           : expand_row_kernel<OUT, 128, false, false>);
  const size_t smem = OUT == kOutW ? sizeof(float) * (size_t)g.ld_pix : 0;
  kern<<<(unsigned)rows, threads, smem, s>>>(
      g.qi, g.qlo, g.ld_pix, g.N, grid, g4, rot, logw, nrot, w_floor, c, gsc,
      (int)expand_tile_slices(g.ld_pix), (uint16_t*)L.base, L.plane_stride, bias, Bsum, Bctx,
      status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_expand_gauss(const Geom& g, const float* grid, const float4* g4,
                                const RotFX* rot, const double* logw, int64_t nrot, int64_t rows,
                                Planes L, double* bias, double* partial, const float4* gsc,
                                double sigma, int32_t* status, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  const double inv = 1.0 / (2.0 * sigma * sigma);
  const int th = gauss_row_threads(rows, expand_tile_slices(g.ld_pix));
  if (th)
    return launch_rows<kOutGauss>(th, g, grid, g4, rot, logw, nrot, rows, 0.f, inv, gsc, L, bias,
                                  nullptr, nullptr, status, s);
  cudaError_t e = launch_tiles(g, grid, g4, rot, nrot, rows, kOutGauss, 0.f, L, partial, nullptr,
                               nullptr, 0, gsc, status, s);
  if (e != cudaSuccess) return e;
  expand_bias_kernel<<<(unsigned)(rows / kTRows), kTRows, 0, s>>>(
      partial, (int)expand_tile_slices(g.ld_pix), rows, logw, nrot, inv,
      bias, nullptr, nullptr, 0);
  return cudaGetLastError();
}

int expand_gauss_launches(int64_t rows, int64_t ld_pix) {
  return gauss_row_threads(rows, expand_tile_slices(ld_pix)) ? 1 : 2;
}

int expand_flu_launches(int64_t rows, int64_t ld_pix, bool delta) {
  return !delta && row_threads(rows, expand_tile_slices(ld_pix)) ? 1 : 3;
}

cudaError_t launch_expand_flu(const Geom& g, const float* grid, const float4* g4, const RotFX* rot,
                              const double* logw, int64_t nrot, int64_t rows, float w_floor,
                              double c, Planes L, double* bias, double* Bctx, const void* Lold,
                              uint16_t* D, int64_t ntp, float* bpm, int32_t* status,
                              cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  const int64_t ns = expand_tile_slices(g.ld_pix), nt = rows / kTRows;
  uint16_t* Lb = (uint16_t*)L.base;
  const int th = Lold ? 0 : row_threads(rows, ns);
  if (th)
    return launch_rows<kOutW>(th, g, grid, g4, rot, logw, nrot, rows, w_floor, c, nullptr, L, bias,
                              bias + rows, Bctx, status, s);
  cudaError_t e = launch_tiles(g, grid, g4, rot, nrot, rows, kOutW, w_floor, L, nullptr, nullptr,
                               nullptr, 0, nullptr, status, s);
  if (e != cudaSuccess) return e;
  flu_bias_kernel<<<(unsigned)nt, kTRows, 0, s>>>(Lb + 2 * L.plane_stride, g.ld_pix, (int)ns, logw,
                                                  nrot, c, bias, bias + rows, Bctx,
                                                  Lold ? bpm : nullptr, nt);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  constexpr int kPer = kTRows / kSplitRows;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)(ns * nt * kPer));
  lc.blockDim = dim3(kTThreads);
  lc.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kPer;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  lc.attrs = &at;
  lc.numAttrs = Lold ? 1 : 0;
  // (an iteration's L is aligned)
  auto split = Lold ? flu_split_kernel<true>
                    : (((uintptr_t)Lb & 3) == 0 ? flu_split_kernel<false>
                                                : flu_split_kernel<false, false>);
  return cudaLaunchKernelEx(&lc, split, g.qi, g.ld_pix, nrot, Lb, L.plane_stride,
                            (const uint16_t*)Lold, D, ntp, (unsigned)ns, status);
}

}  // namespace emc
