// simt.cu -- FP32 SIMT form of the Maximize step (precision EMC_PREC_FP32).
//
// Scores S_jk = sum_i K_ik log W_ij + bias_j (Eq. 2.3 plus the prior of
// Eq. 2.4) as a tiled FP32 FFMA contraction over pixels: 64 rotations x 128
// frames per CTA, 4 x 8 outputs per thread, 16-pixel smem stages. Dot products
// reach |S| ~ 1e4 while P needs S to ~1e-4, beyond what a chain of FP32 FMAs
// keeps. log W is therefore split while it is staged into shared memory:
// hi = log W rounded to the 1/8 grid and r = log W - hi (|r| <= 1/16, exact).
// Counts are integers, so every partial sum of K * hi is a multiple of 1/8
// below 2^21 and the FFMA chain of the hi accumulator never rounds; the r
// accumulator stays small (a random walk of size ~ sqrt(sum K^2) / 28), so its
// rounding is ~1e-5 absolute. The epilogue adds hi + r + bias in FP64.
//  pass 1 : per frame, per tile of 64 rotations, (max_j S_jk, sum_j exp(S_jk - max))
//  pass 2 : P_jk = exp(S_jk - lse_k) written as FP32 [rows][ld_data]
//  update : Num_ji = sum_k P_jk K_ki (Eq. 2.11), FP32 FFMA; the K column of
//           ones at i = n_pix yields den_j = sum_k P_jk.
#include "emc_common.cuh"
#include "emc_internal.h"

namespace emc {

constexpr int SB_M = 64, SB_N = 128, SB_K = 16, S_THREADS = 256;
constexpr int SA_LD = SB_M + 4, SBN_LD = SB_N + 4;
// Accumulators of 4 rows x 8 frames, two frames to a register pair: the packed
// FMA rounds each half as fmaf does and takes half the issue slots.
// A thread's frames are two runs of four, 64 apart, so that a quarter warp's
// 16-byte reads of the staged frames are contiguous (runs of eight cost twice the
// wavefronts, and they bound the kernel: 64^3, 3240 rotations x 2000 frames, pass 1
// 1650 -> 1330 us).
__device__ __forceinline__ int frame_of(int tx, int j) { return (j & 4) * 16 + tx * 4 + (j & 3); }
struct ScoreAcc {
  float2 hi2[4][4], r2[4][4];
  __device__ __forceinline__ float hi(int i, int j) const {
    return j & 1 ? hi2[i][j >> 1].y : hi2[i][j >> 1].x;
  }
  __device__ __forceinline__ float r(int i, int j) const {
    return j & 1 ? r2[i][j >> 1].y : r2[i][j >> 1].x;
  }
};

// Main loop shared by pass 1 and pass 2. Tile origin: rows r0, frames c0.
__device__ __forceinline__ void simt_scores_tile(const float* __restrict__ L, int64_t ld_pix,
                                                 const uint16_t* __restrict__ Kb, int64_t r0,
                                                 int64_t c0, float (*Ah)[SA_LD],
                                                 float (*Ar)[SA_LD], float (*Bs)[SBN_LD],
                                                 ScoreAcc& out) {
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) out.hi2[a][b] = out.r2[a][b] = make_float2(0.f, 0.f);
  const int ar = t >> 2, ac = (t & 3) * 4;  // A: row, pixel offset
  const int br = t >> 1, bc = (t & 1) * 8;  // B: frame, pixel offset
  const float* Ap = L + (r0 + ar) * ld_pix + ac;
  const uint16_t* Bp = Kb + (c0 + br) * ld_pix + bc;
  const int64_t ntiles = ld_pix / SB_K;
  float4 ra = *reinterpret_cast<const float4*>(Ap);
  uint4 rb = *reinterpret_cast<const uint4*>(Bp);
  for (int64_t kt = 0; kt < ntiles; kt++) {
    __syncthreads();
    const float av4[4] = {ra.x, ra.y, ra.z, ra.w};
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const float h = rintf(av4[c] * 8.f) * 0.125f;
      Ah[ac + c][ar] = h;
      Ar[ac + c][ar] = av4[c] - h;
    }
    const uint32_t w4[4] = {rb.x, rb.y, rb.z, rb.w};
#pragma unroll
    for (int c = 0; c < 4; c++) {
      Bs[bc + 2 * c][br] = __uint_as_float(w4[c] << 16);
      Bs[bc + 2 * c + 1][br] = __uint_as_float(w4[c] & 0xffff0000u);
    }
    __syncthreads();
    if (kt + 1 < ntiles) {
      ra = *reinterpret_cast<const float4*>(Ap + (kt + 1) * SB_K);
      rb = *reinterpret_cast<const uint4*>(Bp + (kt + 1) * SB_K);
    }
#pragma unroll
    for (int kk = 0; kk < SB_K; kk++) {
      float4 a = *reinterpret_cast<const float4*>(&Ah[kk][ty * 4]);
      float4 e = *reinterpret_cast<const float4*>(&Ar[kk][ty * 4]);
      float4 b0 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      float4 b1 = *reinterpret_cast<const float4*>(&Bs[kk][64 + tx * 4]);
      const float ah[4] = {a.x, a.y, a.z, a.w};
      const float aq[4] = {e.x, e.y, e.z, e.w};
      const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                            make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float2 h = make_float2(ah[i], ah[i]), q = make_float2(aq[i], aq[i]);
#pragma unroll
        for (int j = 0; j < 4; j++) {
          out.hi2[i][j] = fma2(h, bv[j], out.hi2[i][j]);
          out.r2[i][j] = fma2(q, bv[j], out.r2[i][j]);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(S_THREADS)
    simt_pass1_kernel(const float* __restrict__ L, int64_t ld_pix, const double* __restrict__ bias,
                      const uint16_t* __restrict__ Kb, int64_t ld_data,
                      double* __restrict__ part_m, float* __restrict__ part_s,
                      float* __restrict__ S, float* __restrict__ Sref, int64_t rows) {
  __shared__ __align__(16) float Ah[SB_K][SA_LD];
  __shared__ __align__(16) float Ar[SB_K][SA_LD];
  __shared__ __align__(16) float Bs[SB_K][SBN_LD];
  __shared__ double red[16][SB_N];
  const int64_t r0 = (int64_t)blockIdx.y * SB_M, c0 = (int64_t)blockIdx.x * SB_N;
  ScoreAcc sc;
  simt_scores_tile(L, ld_pix, Kb, r0, c0, Ah, Ar, Bs, sc);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  double b[4];
#pragma unroll
  for (int i = 0; i < 4; i++) b[i] = bias[r0 + ty * 4 + i];
  double x[4][8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    double m = -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      x[i][j] = ((double)sc.hi(i, j) + (double)sc.r(i, j)) + b[i];
      m = fmax(m, x[i][j]);
    }
    red[ty][frame_of(tx, j)] = m;
  }
  __syncthreads();
  double mcol[8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    double m = -INFINITY;
    for (int r = 0; r < 16; r++) m = fmax(m, red[r][frame_of(tx, j)]);
    mcol[j] = m;
  }
  __syncthreads();
  if (S) {
    // scores relative to the tile's column maximum rounded to the 1/64 grid
    float ref[8];
#pragma unroll
    for (int j = 0; j < 8; j++)
      ref[j] = mcol[j] == -INFINITY ? -3.0e38f : (float)(rint(mcol[j] * kGridD) / kGridD);
    // frame-major: 4 consecutive rows of one column per float4
#pragma unroll
    for (int j = 0; j < 8; j++) {
      float4 v;
      v.x = (float)(x[0][j] - (double)ref[j]);
      v.y = (float)(x[1][j] - (double)ref[j]);
      v.z = (float)(x[2][j] - (double)ref[j]);
      v.w = (float)(x[3][j] - (double)ref[j]);
      *reinterpret_cast<float4*>(S + (c0 + frame_of(tx, j)) * rows + r0 + ty * 4) = v;
    }
    if (ty == 0) {
#pragma unroll
      for (int j = 0; j < 8; j++) {
        Sref[(r0 / 32) * ld_data + c0 + frame_of(tx, j)] = ref[j];
        Sref[(r0 / 32 + 1) * ld_data + c0 + frame_of(tx, j)] = ref[j];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 8; j++) {
    float s = 0.f;
    if (mcol[j] != -INFINITY)
#pragma unroll
      for (int i = 0; i < 4; i++) s += expf((float)(x[i][j] - mcol[j]));
    red[ty][frame_of(tx, j)] = (double)s;
  }
  __syncthreads();
  // threads of the first rotation group write the tile's 8 columns each
  if (ty == 0) {
#pragma unroll
    for (int j = 0; j < 8; j++) {
      double s = 0.0;
      for (int r = 0; r < 16; r++) s += red[r][frame_of(tx, j)];
      int64_t col = c0 + frame_of(tx, j);
      part_m[(int64_t)blockIdx.y * ld_data + col] = mcol[j];
      part_s[(int64_t)blockIdx.y * ld_data + col] = (float)s;
    }
  }
}

__global__ void __launch_bounds__(S_THREADS)
    simt_normalize_kernel(const float* __restrict__ L, int64_t ld_pix,
                          const double* __restrict__ bias, int64_t nrot,
                          const uint16_t* __restrict__ Kb, int64_t ld_data, int64_t n_data,
                          const double* __restrict__ lse_m, const double* __restrict__ lse_s,
                          float* __restrict__ P) {
  __shared__ __align__(16) float Ah[SB_K][SA_LD];
  __shared__ __align__(16) float Ar[SB_K][SA_LD];
  __shared__ __align__(16) float Bs[SB_K][SBN_LD];
  const int64_t r0 = (int64_t)blockIdx.y * SB_M, c0 = (int64_t)blockIdx.x * SB_N;
  ScoreAcc sc;
  simt_scores_tile(L, ld_pix, Kb, r0, c0, Ah, Ar, Bs, sc);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  double lse[8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    int64_t col = c0 + frame_of(tx, j);
    lse[j] = col < n_data ? lse_m[col] + log(lse_s[col]) : INFINITY;
  }
#pragma unroll
  for (int i = 0; i < 4; i++) {
    int64_t row = r0 + ty * 4 + i;
    double b = bias[row];
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      double x = ((double)sc.hi(i, j) + (double)sc.r(i, j)) + b - lse[j];
      v[j] = (row < nrot && c0 + frame_of(tx, j) < n_data) ? expf((float)x) : 0.f;
    }
    float* dst = P + row * ld_data + c0 + tx * 4;
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(dst + 64) = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// Bit k % 32 of nz[r][k / 32]: some P of rows 64 r .. 64 r + 63 and frame k is not
// zero. A warp reads 128 frames of eight rows.
__global__ void __launch_bounds__(256)
    simt_nonzero_kernel(const float* __restrict__ P, int64_t ld_data, uint32_t* __restrict__ nz) {
  __shared__ uint32_t any[8][4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t k = (int64_t)blockIdx.x * 128 + 4 * lane;
  const float* p = P + ((int64_t)blockIdx.y * SB_M + w * 8) * ld_data + k;
  unsigned m = 0;
#pragma unroll
  for (int r = 0; r < 8; r++) {
    const float4 v = *reinterpret_cast<const float4*>(p + r * ld_data);
    m |= (v.x != 0.f ? 1u : 0u) | (v.y != 0.f ? 2u : 0u) | (v.z != 0.f ? 4u : 0u) |
         (v.w != 0.f ? 8u : 0u);
  }
  // lane l holds bits 4 l ..: eight lanes make a word
  m <<= 4 * (lane & 7);
  m |= __shfl_xor_sync(0xffffffffu, m, 1);
  m |= __shfl_xor_sync(0xffffffffu, m, 2);
  m |= __shfl_xor_sync(0xffffffffu, m, 4);
  if ((lane & 7) == 0) any[w][lane >> 3] = m;
  __syncthreads();
  if (threadIdx.x < 4) {
    uint32_t a = 0;
    for (int q = 0; q < 8; q++) a |= any[q][threadIdx.x];
    nz[(int64_t)blockIdx.y * (ld_data / 32) + blockIdx.x * 4 + threadIdx.x] = a;
  }
}

// Only the frames with a non-zero P in the tile's 64 rows are contracted, in
// order (most P underflow to exact zeros, which add nothing: 64^3, 3240 rotations x 2000
// frames, 1315 us over every frame, 107 us over these with their bits). nz: simt_nonzero_kernel's
// bits; ALL: every frame.
constexpr int kNzWords = 128;  // words of nz taken at a time: 4096 frames
template <bool ALL>
__global__ void __launch_bounds__(S_THREADS)
    simt_update_kernel(const float* __restrict__ P, int64_t ld_data,
                       const uint16_t* __restrict__ Kb, int64_t ld_pix, int64_t n_pix,
                       const uint32_t* __restrict__ nz, float* __restrict__ Num,
                       float* __restrict__ den) {
  __shared__ __align__(16) float As[SB_K][SA_LD];
  __shared__ __align__(16) float Bs[SB_K][SBN_LD];
  __shared__ uint16_t list[kNzWords * 32];
  __shared__ int wsum[4];
  const int64_t r0 = (int64_t)blockIdx.y * SB_M, c0 = (int64_t)blockIdx.x * SB_N;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4, lane = t & 31, wid = t >> 5;
  float2 acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = make_float2(0.f, 0.f);
  const int ar = t >> 2, ac = (t & 3) * 4;    // A = P: row, frame offset
  const int br = t >> 4, bc = (t & 15) * 8;   // B = K: frame, pixel offset
  const bool bval = c0 + bc < ld_pix;
  const int64_t words = ld_data / 32;
  if (!ALL) nz += blockIdx.y * words;
  for (int64_t w0 = 0; w0 < words; w0 += kNzWords) {
    // the frames of these words (offsets from 32 w0)
    uint32_t bits = t < kNzWords && w0 + t < words ? (ALL ? ~0u : nz[w0 + t]) : 0u;
    int inc = __popc(bits);
    const int own = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    __syncthreads();  // the last list is used up
    if (t < kNzWords && lane == 31) wsum[wid] = inc;
    __syncthreads();
    int at = inc - own, n = 0;
    for (int q = 0; q < 4; q++) {
      if (q < wid) at += wsum[q];
      n += wsum[q];
    }
    while (bits) {
      list[at++] = (uint16_t)(32 * t + __ffs(bits) - 1);
      bits &= bits - 1;
    }
    __syncthreads();
    const float* Ap = P + (r0 + ar) * ld_data + 32 * w0;
    const uint16_t* Bp = Kb + 32 * w0 * ld_pix + c0 + bc;
    float ra[4];
    uint4 rb;
    auto load = [&](int k0) {
#pragma unroll
      for (int c = 0; c < 4; c++) ra[c] = k0 + ac + c < n ? Ap[list[k0 + ac + c]] : 0.f;
      rb = bval && k0 + br < n ? *reinterpret_cast<const uint4*>(Bp + list[k0 + br] * ld_pix)
                               : make_uint4(0, 0, 0, 0);
    };
    load(0);
    for (int k0 = 0; k0 < n; k0 += SB_K) {
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 4; c++) As[ac + c][ar] = ra[c];
      const uint32_t w4[4] = {rb.x, rb.y, rb.z, rb.w};
#pragma unroll
      for (int c = 0; c < 4; c++) {
        Bs[br][bc + 2 * c] = __uint_as_float(w4[c] << 16);
        Bs[br][bc + 2 * c + 1] = __uint_as_float(w4[c] & 0xffff0000u);
      }
      __syncthreads();
      if (k0 + SB_K < n) load(k0 + SB_K);
#pragma unroll
      for (int kk = 0; kk < SB_K; kk++) {
        const float4 a = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
        const float4 b0 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
        const float4 b1 = *reinterpret_cast<const float4*>(&Bs[kk][64 + tx * 4]);
        const float av[4] = {a.x, a.y, a.z, a.w};
        const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                              make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int j = 0; j < 4; j++)
            acc[i][j] = fma2(make_float2(av[i], av[i]), bv[j], acc[i][j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++) {
    int64_t row = r0 + ty * 4 + i;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int64_t col = c0 + 64 * h + tx * 4;
      const float2 u = acc[i][2 * h], v = acc[i][2 * h + 1];
      if (col < ld_pix)
        *reinterpret_cast<float4*>(Num + row * ld_pix + col) = make_float4(u.x, u.y, v.x, v.y);
      if (col == n_pix) den[row] = u.x;
      if (col + 1 == n_pix) den[row] = u.y;
      if (col + 2 == n_pix) den[row] = v.x;
      if (col + 3 == n_pix) den[row] = v.y;
    }
  }
}

int64_t simt_pass1_tiles(int64_t rows) { return rows / SB_M; }

cudaError_t launch_simt_pass1(const float* L, int64_t ld_pix, const double* bias, int64_t rows,
                              const uint16_t* Kb, int64_t ld_data, int64_t n_data,
                              double* part_m, float* part_s, float* S, float* Sref,
                              cudaStream_t s) {
  (void)n_data;
  dim3 grd((unsigned)(ld_data / SB_N), (unsigned)(rows / SB_M));
  simt_pass1_kernel<<<grd, S_THREADS, 0, s>>>(L, ld_pix, bias, Kb, ld_data, part_m, part_s, S,
                                              Sref, rows);
  return cudaGetLastError();
}

cudaError_t launch_simt_normalize(const float* L, int64_t ld_pix, const double* bias, int64_t rows,
                                  int64_t nrot, const uint16_t* Kb, int64_t ld_data,
                                  int64_t n_data, const double* lse_m, const double* lse_s,
                                  float* P, cudaStream_t s) {
  dim3 grd((unsigned)(ld_data / SB_N), (unsigned)(rows / SB_M));
  simt_normalize_kernel<<<grd, S_THREADS, 0, s>>>(L, ld_pix, bias, nrot, Kb, ld_data, n_data,
                                                  lse_m, lse_s, P);
  return cudaGetLastError();
}

cudaError_t launch_simt_update(const float* P, int64_t ld_data, int64_t rows, const uint16_t* Kb,
                               int64_t ld_pix, int64_t n_pix, uint32_t* nz, float* Num,
                               float* den, cudaStream_t s) {
  if (nz) {
    simt_nonzero_kernel<<<dim3((unsigned)(ld_data / 128), (unsigned)(rows / SB_M)), 256, 0, s>>>(
        P, ld_data, nz);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  dim3 grd((unsigned)((ld_pix + SB_N - 1) / SB_N), (unsigned)(rows / SB_M));
  auto kern = nz ? simt_update_kernel<false> : simt_update_kernel<true>;
  kern<<<grd, S_THREADS, 0, s>>>(P, ld_data, Kb, ld_pix, n_pix, nz, Num, den);
  return cudaGetLastError();
}

}  // namespace emc
