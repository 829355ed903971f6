// learned.cu -- learned rotation proposal: binned frame features and a small
// MLP (512 -> 3 x 512 GELU -> one logit per rotation) with hand-written
// forward, backward and Adam kernels.
//
// The paper has no learned component; this is the workload's proposal stage:
// the network reads 32 radial x 16 angular bins of log(1 + mean count) of a
// frame and is trained on soft targets taken from dense EMC responsibilities
// (Eq. 2.4), so that the Maximize step can run over its top-M rotations only.
//
// Matrix products use BF16-rounded operands with FP32 accumulation ("BF16
// matmuls, FP32 master weights"). The output layer (512 x n_out, nearly all
// of the work) runs on the tensor cores: Z = H3 W4 and dW4 = (H3^T) dZ
// through the update form of the tcgen05 kernel (K-major A, MN-major B, FP32
// rows out), dH3 = dZ W4^T through its store form (both K-major), from BF16
// copies made by the kernels below, whenever the batch is a multiple of
// 128. The 512 x 512 layers and other batches use a tiled SIMT kernel that
// serves the three layouts (X W, dY W^T, X^T dY). Parameters live in one FP32
// array: W1[512][512] b1[512] W2 b2 W3 b3 W4[512][ld_out] b4[ld_out],
// ld_out = round_up(n_out, 64).
#include <algorithm>
#include <utility>

#include "emc_common.cuh"
#include "emc_internal.h"

namespace emc {

// ---------------------------------------------------------------- features --
// One CTA per frame: per-bin sums of the counts in shared memory, then
// log(1 + sum / pixels-in-bin); bins with no pixel give 0.
__global__ void features_kernel(const uint16_t* __restrict__ Kb, int kf16, int64_t ld_pix,
                                int64_t n_pix,
                                int64_t n_data, const int16_t* __restrict__ bin,
                                const float* __restrict__ inv_count, float* __restrict__ feat) {
  const int64_t k = blockIdx.x;
  __shared__ float acc[kFeat];
  for (int b = threadIdx.x; b < kFeat; b += blockDim.x) acc[b] = 0.f;
  __syncthreads();
  if (k < n_data)
    for (int64_t i = threadIdx.x; i < ld_pix; i += blockDim.x) {  // pixels + duplicate columns
      if (i == n_pix) continue;  // the column of ones
      const uint16_t u = Kb[k * ld_pix + i];
      const float c = kf16 ? fp16_val(u) : bf16_val(u);
      if (c != 0.f) atomicAdd(&acc[bin[i]], c);
    }
  __syncthreads();
  for (int b = threadIdx.x; b < kFeat; b += blockDim.x)
    feat[k * kFeat + b] = k < n_data ? log1pf(acc[b] * inv_count[b]) : 0.f;
}

cudaError_t launch_features(const uint16_t* Kb, int kf16, int64_t ld_pix, int64_t n_pix,
                            int64_t n_data, int64_t ld_data, const int16_t* bin,
                            const float* inv_count, float* feat, cudaStream_t s) {
  features_kernel<<<(unsigned)ld_data, 256, 0, s>>>(Kb, kf16, ld_pix, n_pix, n_data, bin,
                                                    inv_count, feat);
  return cudaGetLastError();
}

// -------------------------------------------------------------------- GEMM --
// C[M][N] = op(A) op(B); op(A)[m][k] = TA ? A[k*lda + m] : A[m*lda + k],
// op(B)[k][n] = TB ? B[n*ldb + k] : B[k*ldb + n]. EPI: 0 plain, 1 bias,
// 2 bias + GELU (the pre-activation goes to `pre`, GELU of it to C, and where
// given its BF16 copies to hb [M][ldc] and transposed to ht [N][M]),
// 3 times GELU'(pre) (the backward pass through the activation).
// BM rows a tile. A 512 x 512 x 512 layer is 32 x 64 tiles on 128 CTAs, one per SM, the next K
// block's loads in flight while this one is summed: 38 -> 22 us (64 x 64 tiles on
// 64 CTAs waited out every block's load latency). Batches that fill the SMs with 64 x 64 tiles
// twice over read less by those (16384 rows, forward: 1.19 ms by 32-row tiles, 0.87 so). Every
// element sums its products in order of k either way.
// (Rows of tiles go on in grid z: y holds 65535, 2.1 million rows of a batch.)
constexpr int G_BN = 64, G_THREADS = 256;

__device__ __forceinline__ float bf16_round(float x) { return bf16_val(bf16_bits(x)); }

__device__ __forceinline__ float gelu_f(float x) {
  return 0.5f * x * (1.f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) +
         x * __expf(-0.5f * x * x) * 0.39894228040143268f;
}

struct GemmEpi {
  const float* bias;
  float* pre;
  int64_t ldpre;
  uint16_t* hb;
  uint16_t* ht;
  float* bsum;  // column sums of op(B) in order of k, unrounded (EPI 0; bias gradients)
};

template <int G_BM, bool TA, bool TB, int EPI>
__global__ void __launch_bounds__(G_THREADS)
    mlp_gemm_kernel(int M, int N, int K, const float* __restrict__ A, int64_t lda,
                    const float* __restrict__ B, int64_t ldb, float* __restrict__ C, int64_t ldc,
                    const GemmEpi ep) {
  constexpr int G_BK = G_BM == 64 ? 16 : 32, TM = G_BM / 16;  // TM rows a thread
  __shared__ __align__(16) float As[G_BK][G_BM + 4];
  __shared__ __align__(16) float Bs[G_BK][G_BN + 4];
  constexpr int NA = G_BM * G_BK / G_THREADS, NB = G_BN * G_BK / G_THREADS;
  __shared__ float Bw[EPI == 0 ? G_BK : 1][G_BN];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * G_BM, n0 = blockIdx.x * G_BN;
  if (m0 >= M) return;
  const bool sums = EPI == 0 && ep.bsum && m0 == 0;
  float bs = 0.f;
  float ra[NA], rb[NB];
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NA; u++) {
      const int e = t + u * G_THREADS;
      const int gm = m0 + (TA ? e % G_BM : e / G_BK), gk = k0 + (TA ? e / G_BM : e % G_BK);
      ra[u] = gm < M && gk < K ? (TA ? A[(int64_t)gk * lda + gm] : A[(int64_t)gm * lda + gk]) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < NB; u++) {
      const int e = t + u * G_THREADS;
      const int gn = n0 + (TB ? e / G_BK : e % G_BN), gk = k0 + (TB ? e % G_BK : e / G_BN);
      rb[u] = gn < N && gk < K ? (TB ? B[(int64_t)gn * ldb + gk] : B[(int64_t)gk * ldb + gn]) : 0.f;
    }
  };
  float acc[TM][4] = {};
  load(0);
  for (int k0 = 0; k0 < K; k0 += G_BK) {
#pragma unroll
    for (int u = 0; u < NA; u++) {
      const int e = t + u * G_THREADS;
      As[TA ? e / G_BM : e % G_BK][TA ? e % G_BM : e / G_BK] = bf16_round(ra[u]);
    }
#pragma unroll
    for (int u = 0; u < NB; u++) {
      const int e = t + u * G_THREADS;
      Bs[TB ? e % G_BK : e / G_BN][TB ? e / G_BK : e % G_BN] = bf16_round(rb[u]);
      if (sums) Bw[TB ? e % G_BK : e / G_BN][TB ? e / G_BK : e % G_BN] = rb[u];
    }
    __syncthreads();
    if (k0 + G_BK < K) load(k0 + G_BK);
    if (sums && t < G_BN)
#pragma unroll 8
      for (int kk = 0; kk < G_BK; kk++) bs += Bw[kk][t];
#pragma unroll
    for (int kk = 0; kk < G_BK; kk++) {
      float a[TM];
      if (TM == 4) {
        const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * TM]);
        a[0] = a4.x;
        a[1] = a4.y;
        a[TM - 2] = a4.z;
        a[TM - 1] = a4.w;
      } else {
        const float2 a2 = *reinterpret_cast<const float2*>(&As[kk][ty * TM]);
        a[0] = a2.x;
        a[1] = a2.y;
      }
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (sums && t < G_BN && n0 + t < N) ep.bsum[n0 + t] = bs;
#pragma unroll
  for (int i = 0; i < TM; i++) {
    const int gm = m0 + ty * TM + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int gn = n0 + tx * 4 + j;
      if (gn >= N) continue;
      float v = acc[i][j];
      if (EPI == 1 || EPI == 2) v += ep.bias[gn];
      if (EPI == 2) {
        ep.pre[(int64_t)gm * ep.ldpre + gn] = v;
        v = gelu_f(v);
        if (ep.hb) {
          const uint16_t h = bf16_bits(v);
          ep.hb[(int64_t)gm * ldc + gn] = h;
          if (ep.ht) ep.ht[(int64_t)gn * M + gm] = h;
        }
      }
      if (EPI == 3) v *= gelu_grad_f(ep.pre[(int64_t)gm * ep.ldpre + gn]);
      C[(int64_t)gm * ldc + gn] = v;
    }
  }
}

int num_sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n;
}

// across x down blocks, the rows of blocks beyond 65535 in z
dim3 rows_grid(int64_t across, int64_t down) {
  const int64_t y = std::min<int64_t>(down, 65535);
  return dim3((unsigned)across, (unsigned)y, (unsigned)((down + y - 1) / y));
}

template <bool TA, bool TB, int EPI>
cudaError_t gemm(int M, int N, int K, const float* A, int64_t lda, const float* B, int64_t ldb,
                 float* C, int64_t ldc, const GemmEpi& ep, cudaStream_t s) {
  const int64_t across = ((int64_t)N + G_BN - 1) / G_BN;
  if (across * (((int64_t)M + 63) / 64) >= 2 * num_sms())
    mlp_gemm_kernel<64, TA, TB, EPI><<<rows_grid(across, ((int64_t)M + 63) / 64), G_THREADS, 0, s>>>(
        M, N, K, A, lda, B, ldb, C, ldc, ep);
  else
    mlp_gemm_kernel<32, TA, TB, EPI><<<rows_grid(across, ((int64_t)M + 31) / 32), G_THREADS, 0, s>>>(
        M, N, K, A, lda, B, ldb, C, ldc, ep);
  return cudaGetLastError();
}

// ------------------------------------------- BF16 operands for the tcgen05 --
// dst = bf16(src), four values a thread (V4: both 16- and 8-byte aligned, n a multiple of 4)
template <bool V4>
__global__ void to_bf16_kernel(const float* __restrict__ src, int64_t n, uint16_t* __restrict__ dst) {
  const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  if (V4) {
    const float4 v = *reinterpret_cast<const float4*>(src + i);
    *reinterpret_cast<ushort4*>(dst + i) =
        make_ushort4(bf16_bits(v.x), bf16_bits(v.y), bf16_bits(v.z), bf16_bits(v.w));
  } else {
    for (int64_t e = i; e < min(n, i + 4); e++) dst[e] = bf16_bits(src[e]);
  }
}

__global__ void add_bias_kernel(float* __restrict__ Z, int64_t ld, int64_t rows, int64_t cols,
                                const float* __restrict__ b) {
  const int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (c >= cols) return;
  const float v = b[c];
  const int64_t r0 = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * 8;
#pragma unroll
  for (int r = 0; r < 8; r++)
    if (r0 + r < rows) Z[(r0 + r) * ld + c] += v;
}

cudaError_t to_bf16(const float* src, int64_t n, uint16_t* dst, cudaStream_t s) {
  const unsigned blocks = (unsigned)((n / 4 + 256) / 256);
  if (((uintptr_t)src & 15) == 0 && ((uintptr_t)dst & 7) == 0 && n % 4 == 0)
    to_bf16_kernel<true><<<blocks, 256, 0, s>>>(src, n, dst);
  else
    to_bf16_kernel<false><<<blocks, 256, 0, s>>>(src, n, dst);
  return cudaGetLastError();
}

// C[M][N] (FP32, row stride N) = A[M][K] (BF16, K contiguous) B[K][N] (BF16, N
// contiguous) on the tensor cores; M multiple of 128, K and N multiples of 64
cudaError_t tc_gemm(const uint16_t* A, int64_t M, int64_t K, const uint16_t* B, int64_t N,
                    float* C, int32_t* status, cudaStream_t s) {
  Planes pa{const_cast<uint16_t*>(A), M * K, K};
  // few K blocks a tile: bound by its FP32 output, so whole-line stores
  return launch_tc_update(pa, EMC_PREC_BF16, M, B, K, N, INT64_MAX, C, nullptr, status, s,
                          nullptr, nullptr, TcCtl{}, true);
}

// ------------------------------------------------- loss and its gradient --
// Row b of z (n_out logits, stride ld; zb (may be NULL): a bias still to be added):
// lse[b] = log sum_j exp(z_j), mass[b] = sum_r p_r and loss
// += -sum_r p_r (z_{idx_r} - lse) / B. The sum is kept per thread as three FP32 words, each
// taking the exact rounding errors of the one before (what the third rounds is below 2^-64 of
// the sum; FP64 additions and conversions are rare on this part), merged in FP64.
__global__ void __launch_bounds__(512)
    softmax_lse_kernel(const float* __restrict__ z, int64_t ld, int n_out,
                       const float* __restrict__ zb, const int32_t* __restrict__ tidx,
                       const float* __restrict__ tprob, int R, int B, float* __restrict__ lse,
                       float* __restrict__ mass, double* loss) {
  const int64_t b = blockIdx.x;
  const float* row = z + b * ld;
  __shared__ float red[16];
  __shared__ double dred[16];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float M = -INFINITY;
#pragma unroll 8
  for (int j = threadIdx.x; j < n_out; j += 512) M = fmaxf(M, row[j] + (zb ? zb[j] : 0.f));
  for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  if (lane == 0) red[wid] = M;
  __syncthreads();
  M = red[0];
  for (int w = 1; w < 16; w++) M = fmaxf(M, red[w]);
  float s = 0.f, se = 0.f, st = 0.f;
#pragma unroll 8
  for (int j = threadIdx.x; j < n_out; j += 512) {
    const f2 a = two_sum(s, __expf((row[j] + (zb ? zb[j] : 0.f)) - M));
    const f2 b = two_sum(se, a.l);
    s = a.h;
    se = b.h;
    st += b.l;
  }
  double d = (double)s + ((double)se + (double)st);
  for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if (lane == 0) dred[wid] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 16; w++) t += dred[w];
    const float L = M + (float)log(t);
    double l = 0.0;
    float tm = 0.f;
    for (int r = 0; r < R; r++) {
      const float p = tprob[b * R + r];
      const int c = tidx[b * R + r];
      l -= (double)p * ((double)(row[c] + (zb ? zb[c] : 0.f)) - (double)L);
      tm += p;
    }
    lse[b] = L;
    mass[b] = tm;
    atomicAdd(loss, l / B);
  }
}

// (both softmax kernels: 512 x 50112 logits, 312 us with separate passes for the bias,
// the FP32 gradient, its BF16 copy and its column sums on top, 176 more; now 51 + 116 us)
// dL/dz = (softmax(z) sum_r p_r - onehot(p)) / B (zero beyond n_out) as BF16
// (dzb), or in FP32 over z itself (dzb NULL), and its column sums in row order
// (the bias gradient). A warp walks 32 columns of every row, 16 rows' loads in
// flight; the CTA first marks the rows that have a target among its 128 columns, and
// only those look their targets up. chunk: rows a CTA (grid y); several chunks leave their
// sums in db[chunk][ld], in row order each, for sum_chunks_kernel (3240 columns are 26 CTAs:
// 4096 rows with 64 targets took 2.85 ms in one chunk with the targets a row at a time, 0.30 ms
// so; 50100 columns 1.37 and 0.69 ms).
// MANY: rows' targets fall on a CTA's columns often. SPLIT: several chunks.
template <bool MANY, bool SPLIT>
__global__ void __launch_bounds__(128)
    softmax_grad_kernel(float* __restrict__ z, int64_t ld, int n_out,
                        const float* __restrict__ zb, const int32_t* __restrict__ tidx,
                        const float* __restrict__ tprob, int R, int B,
                        const float* __restrict__ lse, const float* __restrict__ mass, int chunk,
                        uint16_t* __restrict__ dzb, float* __restrict__ db) {
  constexpr int kRows = 16, kBatch = 512;
  __shared__ unsigned hits[kBatch / 32];
  const int lane = threadIdx.x & 31;
  const int cta0 = blockIdx.x * 128, c0 = cta0 + (threadIdx.x & 96), c = c0 + lane;
  const bool live = c < (int)ld, in = c < n_out;  // ld is a multiple of 64
  const float bias = zb && in ? zb[c] : 0.f;
  const float invB = 1.f / (float)B;
  float sum = 0.f;
  const int first = SPLIT ? blockIdx.y * chunk : 0, last = SPLIT ? min(B, first + chunk) : B;
  for (int b0 = first; b0 < last; b0 += kBatch) {
    const int b1 = min(last, b0 + kBatch);
    __syncthreads();
    if (threadIdx.x < kBatch / 32) hits[threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll 8
    for (int64_t e = (int64_t)b0 * R + threadIdx.x; e < (int64_t)b1 * R; e += 128) {
      const int q = tidx[e];
      if (q >= cta0 && q < cta0 + 128) {
        const int r = (int)(e / R) - b0;
        atomicOr(&hits[r >> 5], 1u << (r & 31));
      }
    }
    __syncthreads();
    if (!live) continue;  // whole warps
    float x[kRows];
    auto load = [&](int r0) {
#pragma unroll
      for (int u = 0; u < kRows; u++) x[u] = r0 + u < b1 ? z[(int64_t)(r0 + u) * ld + c] : 0.f;
    };
    load(b0);
    for (int r0 = b0; r0 < b1; r0 += kRows) {
      float v[kRows];
#pragma unroll
      for (int u = 0; u < kRows; u++) {
        const int r = min(r0 + u, b1 - 1);
        v[u] = in ? __expf((x[u] + bias) - lse[r]) * mass[r] * invB : 0.f;
      }
      if (r0 + kRows < b1) load(r0 + kRows);
      const unsigned h16 = hits[(r0 - b0) >> 5] >> ((r0 - b0) & 31) & 0xffffu;
      if (MANY && h16) {
        for (int t0 = 0; t0 < R; t0 += 32) {
          int q[kRows];  // the rows' targets together: one wait for 16 rows
#pragma unroll
          for (int u = 0; u < kRows; u++)
            q[u] = (h16 >> u & 1u) && t0 + lane < R ? tidx[(int64_t)(r0 + u) * R + t0 + lane] : -1;
#pragma unroll
          for (int u = 0; u < kRows; u++) {
            unsigned hit = __ballot_sync(0xffffffffu, q[u] >= c0 && q[u] < c0 + 32);
            while (hit) {
              const int w = __ffs(hit) - 1;
              hit &= hit - 1;
              if (__shfl_sync(0xffffffffu, q[u], w) == c)
                v[u] -= tprob[(int64_t)(r0 + u) * R + t0 + w] * invB;
            }
          }
        }
      } else if (h16) {
#pragma unroll
        for (int u = 0; u < kRows; u++) {
          if (!(h16 >> u & 1u)) continue;
          const int64_t e0 = (int64_t)(r0 + u) * R;
          for (int t0 = 0; t0 < R; t0 += 32) {
            const int q = t0 + lane < R ? tidx[e0 + t0 + lane] : -1;
            unsigned hit = __ballot_sync(0xffffffffu, q >= c0 && q < c0 + 32);
            while (hit) {
              const int w = __ffs(hit) - 1;
              hit &= hit - 1;
              if (__shfl_sync(0xffffffffu, q, w) == c) v[u] -= tprob[e0 + t0 + w] * invB;
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kRows; u++) {
        if (r0 + u >= b1) break;
        sum += v[u];
        if (dzb) dzb[(int64_t)(r0 + u) * ld + c] = bf16_bits(v[u]);
        else z[(int64_t)(r0 + u) * ld + c] = v[u];
      }
    }
  }
  if (in) db[(SPLIT ? (int64_t)blockIdx.y * ld : 0) + c] = sum;
}

// out[c] = the chunks' sums, in their order
__global__ void sum_chunks_kernel(const float* __restrict__ part, int64_t ld, int n, int chunks,
                                  float* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  float s = 0.f;
  for (int k = 0; k < chunks; k++) s += part[k * ld + c];
  out[c] = s;
}

// d = g * GELU'(a), elementwise
__global__ void gelu_backward_kernel(const float* __restrict__ g, const float* __restrict__ a,
                                     float* __restrict__ d, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = g[i] * gelu_grad_f(a[i]);
}

// Bound by its traffic (28 B a parameter): four parameters a thread (V4: every
// array 16-byte aligned), 26.5 M of them 150 -> 100 us (110 at the copy rate).
template <bool V4>
__global__ void __launch_bounds__(256)
    adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                float bc1, float bc2) {
  const int64_t i0 = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  auto step = [&](float gi, float& mi, float& vi, float& pi) {
    mi = b1 * mi + (1.f - b1) * gi;
    vi = b2 * vi + (1.f - b2) * gi * gi;
    pi -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  };
  if (V4 && i0 + 4 <= n) {
    const float4 g4 = __ldcs(reinterpret_cast<const float4*>(g + i0));
    float4 m4 = __ldcs(reinterpret_cast<const float4*>(m + i0));
    float4 v4 = __ldcs(reinterpret_cast<const float4*>(v + i0));
    float4 p4 = *reinterpret_cast<const float4*>(p + i0);
    step(g4.x, m4.x, v4.x, p4.x);
    step(g4.y, m4.y, v4.y, p4.y);
    step(g4.z, m4.z, v4.z, p4.z);
    step(g4.w, m4.w, v4.w, p4.w);
    __stcs(reinterpret_cast<float4*>(m + i0), m4);
    __stcs(reinterpret_cast<float4*>(v + i0), v4);
    *reinterpret_cast<float4*>(p + i0) = p4;
    return;
  }
  for (int64_t i = i0; i < min(n, i0 + 4); i++) {
    float mi = m[i], vi = v[i], pi = p[i];
    step(g[i], mi, vi, pi);
    m[i] = mi;
    v[i] = vi;
    p[i] = pi;
  }
}

// ------------------------------------------------------------ host side --
MlpLayout mlp_layout(int64_t n_out, int64_t B) {
  MlpLayout y;
  y.n_out = n_out;
  y.ld_out = (n_out + 63) / 64 * 64;
  const int64_t H = kFeat;
  int64_t o = 0;
  for (int l = 0; l < 3; l++) {
    y.W[l] = o;
    o += H * H;
    y.b[l] = o;
    o += H;
  }
  y.W[3] = o;
  o += H * y.ld_out;
  y.b[3] = o;
  o += y.ld_out;
  y.n_params = o;
  // work: pre-activations a[3], activations h[3], dh, da (each B x 512), z / dz (B x ld_out),
  // then the tensor-core path's BF16 copies: H3 [B][512], H3^T [512][B], dZ [B][ld_out],
  // W4 [512][ld_out], each from a 256-byte boundary
  y.B = B;
  auto up64 = [](int64_t n) { return (n + 63) / 64 * 64; };  // floats to 256 bytes
  y.work_floats = up64(8 * B * H + B * y.ld_out) + up64(B * H / 2) + up64(B * H / 2) +
                  up64(B * y.ld_out / 2) + up64(H * y.ld_out / 2);
  return y;
}

namespace {
struct Work {
  float* a[3];
  float* h[3];
  float* dh;
  float* da;
  float* z;
  uint16_t *h3b, *h3t, *dzb, *w4b;  // BF16 operands of the tensor-core products
};
Work carve(const MlpLayout& y, float* w) {
  Work k;
  const int64_t H = kFeat, BH = y.B * H;
  auto up64 = [](int64_t n) { return (n + 63) / 64 * 64; };
  for (int l = 0; l < 3; l++) k.a[l] = w + l * BH;
  for (int l = 0; l < 3; l++) k.h[l] = w + (3 + l) * BH;
  k.dh = w + 6 * BH;
  k.da = w + 7 * BH;
  k.z = w + 8 * BH;
  float* o = w + up64(8 * BH + y.B * y.ld_out);
  k.h3b = reinterpret_cast<uint16_t*>(o);
  o += up64(BH / 2);
  k.h3t = reinterpret_cast<uint16_t*>(o);
  o += up64(BH / 2);
  k.dzb = reinterpret_cast<uint16_t*>(o);
  o += up64(y.B * y.ld_out / 2);
  k.w4b = reinterpret_cast<uint16_t*>(o);
  return k;
}
bool tc_batch(int B) { return B >= 128 && B % 128 == 0; }
}  // namespace

// Forward into logits, without the output layer's bias where a batch goes by tensor cores.
// train: H3^T is then kept for the weight gradient.
static cudaError_t forward(const MlpLayout& y, const float* params, const float* X, int B,
                           float* work, float* logits, bool train, cudaStream_t s) {
  Work w = carve(y, work);
  const int H = kFeat;
  const bool tc = tc_batch(B);
  const float* in = X;
  cudaError_t e;
  for (int l = 0; l < 3; l++) {
    const bool last = tc && l == 2;
    e = gemm<false, false, 2>(B, H, H, in, H, params + y.W[l], H, w.h[l], H,
                              GemmEpi{params + y.b[l], w.a[l], H, last ? w.h3b : nullptr,
                                      last && train ? w.h3t : nullptr},
                              s);
    if (e != cudaSuccess) return e;
    in = w.h[l];
  }
  if (!tc)
    return gemm<false, false, 1>(B, (int)y.n_out, H, in, H, params + y.W[3], y.ld_out, logits,
                                 y.ld_out, GemmEpi{params + y.b[3]}, s);
  // output layer on the tensor cores: bf16(H3) bf16(W4), the bias to follow
  if ((e = to_bf16(params + y.W[3], (int64_t)H * y.ld_out, w.w4b, s)) != cudaSuccess) return e;
  return tc_gemm(w.h3b, B, H, w.w4b, y.ld_out, logits, nullptr, s);
}

cudaError_t mlp_forward(const MlpLayout& y, const float* params, const float* X, int B,
                        float* work, float* logits, cudaStream_t s) {
  cudaError_t e = forward(y, params, X, B, work, logits, false, s);
  if (e != cudaSuccess || !tc_batch(B)) return e;
  add_bias_kernel<<<rows_grid((y.n_out + 255) / 256, ((int64_t)B + 7) / 8), 256, 0, s>>>(
      logits, y.ld_out, B, y.n_out, params + y.b[3]);
  return cudaGetLastError();
}

cudaError_t mlp_train_step(const MlpLayout& y, float* params, float* grads, float* adam_m,
                           float* adam_v, int step, float lr, const float* X,
                           const int32_t* tidx, const float* tprob, int B, int R, float* work,
                           double* loss, cudaStream_t s) {
  Work w = carve(y, work);
  const int H = kFeat;
  const bool tc = tc_batch(B);
  const int64_t BH = (int64_t)B * H;
  cudaError_t e = forward(y, params, X, B, work, w.z, true, s);
  if (e != cudaSuccess) return e;
  float *lse = w.dh, *mass = w.dh + B;  // dh is written after the loss
  const float* zb = tc ? params + y.b[3] : nullptr;
  softmax_lse_kernel<<<B, 512, 0, s>>>(w.z, y.ld_out, (int)y.n_out, zb, tidx, tprob, R, B, lse,
                                       mass, loss);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // chunks of 512 rows where the columns leave SMs idle; their sums are kept in da, which is
  // written later: ceil(B / 512) ld_out values in B H, which fit from 256 H columns down (two chunks
  // of 513 rows are the tightest)
  const int64_t cols = (y.ld_out + 127) / 128;
  const int chunk = cols >= 4 * num_sms() || y.ld_out > 256 * H ? B : std::min(B, 512);
  const int chunks = (B + chunk - 1) / chunk;
  auto grad = (int64_t)R * 256 >= y.n_out ? softmax_grad_kernel<true, true>
              : chunks > 1                ? softmax_grad_kernel<false, true>
                                          : softmax_grad_kernel<false, false>;
  grad<<<dim3((unsigned)cols, (unsigned)chunks), 128, 0, s>>>(
      w.z, y.ld_out, (int)y.n_out, zb, tidx, tprob, R, B, lse, mass, chunk, tc ? w.dzb : nullptr,
      chunks > 1 ? w.da : grads + y.b[3]);
  if (chunks > 1)
    sum_chunks_kernel<<<(unsigned)((y.n_out + 255) / 256), 256, 0, s>>>(
        w.da, y.ld_out, (int)y.n_out, chunks, grads + y.b[3]);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // output layer: dW4 = h3^T dz, da3 = (dz W4^T) GELU'(a3)
  if (tc) {
    // on the tensor cores (the whole padded width: dZ is 0 beyond n_out)
    if ((e = tc_gemm(w.h3t, H, B, w.dzb, y.ld_out, grads + y.W[3], nullptr, s)) != cudaSuccess)
      return e;
    // narrow tiles while they fit the SMs at once, else 256 columns a tile (a tile's sum runs on one
    // SM, 225 and 270 us over 50112; B = 4096: 889 us narrow, 334 us so)
    const Planes dz{w.dzb, (int64_t)B * y.ld_out, y.ld_out};
    e = (B / 128) * (H / 32) <= num_sms()
            ? launch_tc_nt(w.dzb, w.w4b, B, H, y.ld_out, w.dh, nullptr, s)
            : launch_tc_store(dz, B, w.w4b, H, y.ld_out, w.dh, 0, nullptr, s);
    if (e != cudaSuccess) return e;
    gelu_backward_kernel<<<(unsigned)((BH + 255) / 256), 256, 0, s>>>(w.dh, w.a[2], w.da, BH);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else {
    e = gemm<true, false, 0>(H, (int)y.n_out, B, w.h[2], H, w.z, y.ld_out, grads + y.W[3],
                             y.ld_out, GemmEpi{}, s);
    if (e != cudaSuccess) return e;
    e = gemm<false, true, 3>(B, H, (int)y.n_out, w.z, y.ld_out, params + y.W[3], y.ld_out, w.da, H,
                             GemmEpi{nullptr, w.a[2], H}, s);
    if (e != cudaSuccess) return e;
  }
  // hidden layers: da and dh in turn hold dL/da of the layer
  float *g = w.da, *next = w.dh;
  for (int l = 2; l >= 0; l--) {
    const float* in = l == 0 ? X : w.h[l - 1];
    GemmEpi ep{};
    ep.bsum = grads + y.b[l];
    e = gemm<true, false, 0>(H, H, B, in, H, g, H, grads + y.W[l], H, ep, s);
    if (e != cudaSuccess) return e;
    if (l == 0) break;
    e = gemm<false, true, 3>(B, H, H, g, H, params + y.W[l], H, next, H,
                             GemmEpi{nullptr, w.a[l - 1], H}, s);
    if (e != cudaSuccess) return e;
    std::swap(g, next);
  }
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  const unsigned blocks = (unsigned)((y.n_params / 4 + 256) / 256);
  const bool v4 = (((uintptr_t)params | (uintptr_t)grads | (uintptr_t)adam_m | (uintptr_t)adam_v) &
                   15) == 0;
  auto adam = v4 ? adam_kernel<true> : adam_kernel<false>;
  adam<<<blocks, 256, 0, s>>>(params, grads, adam_m, adam_v, y.n_params, lr, b1, b2, 1e-8f, bc1,
                              bc2);
  return cudaGetLastError();
}

}  // namespace emc
