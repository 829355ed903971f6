// sparse.cu -- candidate selection and the Maximize step over candidate sets.
//
// Given M candidate rotations C_k per frame (from the learned proposal), the
// E- and M-steps (Eq. 2.4, 2.11) run over the pairs (j, k), j in C_k, only:
//   S_jk = sum_i K_ik log W_ij + bias_j,  lse_k = log sum_{j in C_k} exp S_jk,
//   P_jk = exp(S_jk - lse_k),  Num_j = sum_{k: j in C_k} P_jk K_k.
// The pairs are transposed once into a CSR list per rotation, so that both
// contractions read one log W row (staged in shared memory) and gather the
// frames' rows of K, which are 3x smaller than a split log W row and stay in L2
// at the 64^3 size. Scores use the dense forms' split of log W, its sums exact:
// as integers from a frame's non-zero list (sparse_rows_kernel), or hi on the 1/8
// grid and a small residual from its row (sparse_scores_kernel).
#include <limits.h>

#include <algorithm>

#include "emc_common.cuh"
#include "emc_internal.h"

namespace emc {

// ------------------------------------------------------------------- top-M --
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Block-wide exclusive prefix of a 0/1 flag (blockDim.x == 256); returns the
// prefix and writes the block total to *total.
__device__ __forceinline__ int block_prefix(int flag, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  const int in_warp = __popc(bal & ((1u << lane) - 1u));
  if (lane == 0) warp_tot[wid] = __popc(bal);
  __syncthreads();
  int before = 0, tot = 0;
  for (int w = 0; w < 8; w++) {
    if (w < wid) before += warp_tot[w];
    tot += warp_tot[w];
  }
  __syncthreads();
  *total = tot;
  return before + in_warp;
}

// Top M in one read of the row (M <= kTopHold), one CTA of 512 threads per row.
//  * A sample of 512 values, or groups of 8, spread over the row gives a threshold
//    that about 1.2 to 3 M of the row's values exceed (topm_rank). Each warp then reads a
//    contiguous sixteenth of the row, several loads in flight and no barrier, and
//    packs the values above the threshold into a list of its own, in index order.
//  * The M-th largest key T of the lists is built bit by bit from block-wide
//    counts of the keys in registers, which does not depend on how the keys are
//    spread (a histogram's atomics pile up on the few exponents logits share).
//  * A row that the sample misjudges (fewer than M values above the threshold, or a
//    full list; ordered or tied rows), a short row or a long list is streamed
//    instead: values enter a buffer of 8192 in order; when it is full, T of its entries
//    is found, the M that count stay, and from then on a value must exceed T to enter (an
//    equal one comes later in the order, so it loses every tie).
// Index order is kept throughout, so the last selection writes the result out.
// Bound by the one read: 2048 x 50100 logits, M = 512 took 701 us with five
// reads and histograms, 337 us streamed, 198 us so (61 us at the copy rate).
constexpr int kTopThreads = 512;
constexpr int kTopHold = 4096;   // longest list
constexpr int kTopCap = 8192;    // buffer entries: 16 per thread
constexpr int kTopChunk = 8 * kTopThreads;
constexpr int kTopPad = kTopCap + kTopCap / 16;  // entry e at e + e / 16: fewer bank conflicts
constexpr int kTopWarp = 256;    // entries of a warp's list
constexpr int kTopLists = 16 * kTopWarp;
static_assert(kTopHold + kTopChunk <= kTopCap, "a chunk fits after a selection");
constexpr size_t kTopSmem = 2 * sizeof(uint32_t) * kTopPad;
__device__ __forceinline__ int top_at(int e) { return e + (e >> 4); }

// Values a thread adds to the sample: eight, or one of a short row.
__host__ __device__ __forceinline__ int topm_share(int64_t n) { return n >= 4 * kTopChunk ? 8 : 1; }

// Rank in the sample that leaves at least M of n values above it but for a
// chance of about 1e-4 (four standard deviations of the sample's count more), or 0
// where the lists would be too full, or the row so short that one selection
// from all of it costs less.
int topm_rank(int64_t n, int M) {
  const double size = (double)topm_share(n) * kTopThreads, mean = (double)M * size / (double)n;
  const int r = (int)(mean + 4.0 * sqrt(mean) + 4.0);
  return n > kTopChunk && (double)r * n <= 2048.0 * size ? r : 0;
}

// block-wide sum; wt: one of two 16-entry buffers used in turn
__device__ __forceinline__ int top_sum(int v, int* wt) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  if (lane == 0) wt[wid] = v;
  __syncthreads();
  return __reduce_add_sync(0xffffffffu, lane < 16 ? wt[lane] : 0);
}

// block-wide exclusive prefix of v; *total: the sum
__device__ __forceinline__ int top_prefix(int v, int* wt, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) wt[wid] = inc;
  __syncthreads();
  const int w = lane < 16 ? wt[lane] : 0;
  *total = __reduce_add_sync(0xffffffffu, w);
  return inc - v + __reduce_add_sync(0xffffffffu, lane < wid ? w : 0);
}

// The M-th largest of the keys in the threads' registers (per of them each;
// unused ones are 0 and there are at least M others), down to bit `low`
// (bits below it 0: a lower bound). par: the buffer of wt that is next.
template <int MAXPER>
__device__ __forceinline__ uint32_t top_key(const uint32_t (&k)[MAXPER], int per, int M, int low,
                                            int* wt, int& par) {
  uint32_t T = 0;
  for (int bit = 31; bit >= low; bit--) {
    const uint32_t c = T | (1u << bit);  // > 0: unused keys do not count
    int g = 0;
#pragma unroll
    for (int i = 0; i < MAXPER; i++) {
      if (i >= per) break;
      g += k[i] >= c;
    }
    g = top_sum(g, wt + 16 * par);
    par ^= 1;
    if (g >= M) T = c;
    if (g == M) break;  // exactly the keys >= T
  }
  return T;
}

// T, the M-th largest of the buffer's cnt >= M keys (returned); the M entries
// that count stay, in index order: in the buffer, or (FINAL) in out, the larger
// ones first and then the first equal ones. s_min: a word of shared memory.
template <bool FINAL>
__device__ __forceinline__ uint32_t top_select(uint32_t* keys, int* idx, int cnt, int M, int* wt,
                                               int& par, uint32_t* s_min, int32_t* out) {
  const int per = (cnt + kTopThreads - 1) / kTopThreads;  // <= 16
  const int e0 = threadIdx.x * per, mine = min(max(cnt - e0, 0), per);
  if (threadIdx.x == 0) *s_min = 0xffffffffu;
  uint32_t k[16];
#pragma unroll
  for (int i = 0; i < 16; i++) k[i] = i < mine ? keys[top_at(e0 + i)] : 0u;
  uint32_t T = top_key(k, per, M, 0, wt, par);
  // where the bits ended early (exactly M keys >= T): the smallest of those
  uint32_t lo = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < 16; i++)
    if (i < mine && k[i] >= T) lo = min(lo, k[i]);
  lo = __reduce_min_sync(0xffffffffu, lo);
  if ((threadIdx.x & 31) == 0) atomicMin(s_min, lo);
  __syncthreads();
  T = *s_min;
  int gt = 0, eq = 0;
#pragma unroll
  for (int i = 0; i < 16; i++) {
    gt += i < mine && k[i] > T;
    eq += i < mine && k[i] == T;
  }
  int total;
  const int before = top_prefix(gt | (eq << 16), wt + 16 * par, &total);
  par ^= 1;
  const int need = M - (total & 0xffff);
  int ng = before & 0xffff, ne = before >> 16;
  if (FINAL) {
#pragma unroll
    for (int i = 0; i < 16; i++) {
      if (i >= mine) break;
      if (k[i] > T) {
        out[ng++] = idx[top_at(e0 + i)];
      } else if (k[i] == T) {
        if (ne < need) out[M - need + ne] = idx[top_at(e0 + i)];
        ne++;
      }
    }
  } else {
    int id[16];
#pragma unroll
    for (int i = 0; i < 16; i++) id[i] = i < mine ? idx[top_at(e0 + i)] : 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; i++) {
      if (i >= mine) break;
      const bool g = k[i] > T, q = k[i] == T;
      if (g || (q && ne < need)) {
        const int at = top_at(ng + min(ne, need));
        keys[at] = k[i];
        idx[at] = id[i];
      }
      ng += g;
      ne += q;
    }
    __syncthreads();
  }
  return T;
}

// VEC: rows start on 16-byte boundaries
template <bool VEC>
__device__ __forceinline__ void top_load8(const float* z, int64_t e, int n, float (&v)[8]) {
  if (VEC && e + 8 <= n) {
    const float4 a = *reinterpret_cast<const float4*>(z + e);
    const float4 b = *reinterpret_cast<const float4*>(z + e + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = e + i < n ? z[e + i] : 0.f;
  }
}

// the streamed form; returns the entries left in the buffer
template <bool VEC>
__device__ __noinline__ int top_stream(const float* z, int n, int M, uint32_t* keys, int* idx,
                                       int* wt, uint32_t* s_min) {
  int par = 0, cnt = 0;
  bool has = false;   // T bounds what may enter
  uint32_t T = 0;
  float v[8];
  top_load8<VEC>(z, 8 * threadIdx.x, n, v);
  for (int64_t base = 0; base < n; base += kTopChunk) {
    const int64_t e = base + 8 * threadIdx.x;
    uint32_t k[8];
#pragma unroll
    for (int i = 0; i < 8; i++) k[i] = order_key(v[i]);
    if (base + kTopChunk < n) top_load8<VEC>(z, e + kTopChunk, n, v);
    int at, total;
    unsigned enter;
    while (true) {
      enter = 0;
#pragma unroll
      for (int i = 0; i < 8; i++) enter |= (e + i < n && (!has || k[i] > T)) ? 1u << i : 0u;
      at = top_prefix(__popc(enter), wt + 16 * par, &total);
      par ^= 1;
      if (cnt + total <= kTopCap) break;
      T = top_select<false>(keys, idx, cnt, M, wt, par, s_min, nullptr);
      has = true;
      cnt = M;
    }
    at += cnt;
#pragma unroll
    for (int i = 0; i < 8; i++)
      if (enter & (1u << i)) {
        const int p = top_at(at++);
        keys[p] = k[i];
        idx[p] = (int)(e + i);
      }
    cnt += total;
  }
  __syncthreads();
  return cnt;
}

template <bool VEC>
__global__ void __launch_bounds__(kTopThreads, 2)
    topm_stream_kernel(const float* __restrict__ logits, int64_t ld, int n, int M, int rank,
                       int32_t* __restrict__ cand) {
  const float* z = logits + (int64_t)blockIdx.x * ld;
  extern __shared__ uint32_t top_smem[];
  uint32_t* keys = top_smem;
  int* idx = reinterpret_cast<int*>(top_smem + kTopPad);
  __shared__ int wt[32];
  __shared__ int lists[17];
  __shared__ uint32_t s_min;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int par = 0, cnt = 0;
  bool ok = false;
  if (rank > 0) {
    // the sample: a value every n / 512, or 8 from a multiple of 8 on
    const int share = topm_share(n);
    const int64_t at = (int64_t)threadIdx.x * (n - share) / (kTopThreads - 1);
    float v[8];
    if (share == 8)
      top_load8<VEC>(z, at & ~(int64_t)7, n, v);
    else
      v[0] = z[at];
    uint32_t k[8];
#pragma unroll
    for (int i = 0; i < 8; i++) k[i] = i < share ? order_key(v[i]) : 0u;
    const uint32_t T0 = top_key(k, share, rank, 16, wt, par);
    // the warp's sixteenth, 512 values a step (4 x 4 consecutive ones per lane)
    const int64_t seg = ((int64_t)(n + 15) / 16 + 3) & ~(int64_t)3;
    const int64_t b = wid * seg, end = min((int64_t)n, b + seg);
    uint32_t* lk = keys + wid * kTopWarp;
    int* li = idx + wid * kTopWarp;
    int len = 0;
    const unsigned below = (1u << lane) - 1u;
    for (int64_t e0 = b; e0 < end; e0 += 512) {
      float4 w[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t e = e0 + u * 128 + 4 * lane;
        if (VEC && e + 4 <= end) {
          w[u] = __ldcs(reinterpret_cast<const float4*>(z + e));
        } else {
          w[u].x = e < end ? z[e] : 0.f;
          w[u].y = e + 1 < end ? z[e + 1] : 0.f;
          w[u].z = e + 2 < end ? z[e + 2] : 0.f;
          w[u].w = e + 3 < end ? z[e + 3] : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t e = e0 + u * 128 + 4 * lane;
        const uint32_t kk[4] = {order_key(w[u].x), order_key(w[u].y), order_key(w[u].z),
                                order_key(w[u].w)};
        unsigned m = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) m |= (e + i < end && kk[i] >= T0) ? 1u << i : 0u;
        if (!__any_sync(0xffffffffu, m)) continue;
        int p = len, tot = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const unsigned bal = __ballot_sync(0xffffffffu, m & (1u << i));
          p += __popc(bal & below);
          tot += __popc(bal);
        }
#pragma unroll
        for (int i = 0; i < 4; i++)
          if (m & (1u << i)) {
            if (p < kTopWarp) {
              lk[p] = kk[i];
              li[p] = (int)(e + i);
            }
            p++;
          }
        len += tot;  // beyond kTopWarp: the row is streamed
      }
    }
    if (lane == 0) lists[wid] = len;
    __syncthreads();
    int start = 0, most = 0;
#pragma unroll
    for (int w = 0; w < 16; w++) {
      if (w < wid) start += lists[w];
      cnt += lists[w];
      most = max(most, lists[w]);
    }
    ok = most <= kTopWarp && cnt >= M;
    if (ok) {
      // the lists behind one another, above them in the same arrays
      uint32_t* ck = keys + kTopLists;
      int* ci = idx + kTopLists;
      __syncwarp();
      for (int t = lane; t < len; t += 32) {
        ck[top_at(start + t)] = lk[t];
        ci[top_at(start + t)] = li[t];
      }
      keys = ck;
      idx = ci;
    }
    __syncthreads();
  }
  if (!ok) {
    cnt = top_stream<VEC>(z, n, M, keys, idx, wt, &s_min);
    par = 0;
  }
  top_select<true>(keys, idx, cnt, M, wt, par, &s_min, cand + (int64_t)blockIdx.x * M);
}

// Longer lists, and many short rows. One CTA (256 threads) per row: radix selection
// of the M-th largest key over four 8-bit digits, then the keys above it in index order
// followed by the first equal keys in index order (ties towards the lower index).
__global__ void __launch_bounds__(256)
    topm_kernel(const float* __restrict__ logits, int64_t ld, int n, int M,
                int32_t* __restrict__ cand) {
  const float* z = logits + (int64_t)blockIdx.x * ld;
  int32_t* out = cand + (int64_t)blockIdx.x * M;
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_mask;
  __shared__ int s_need;
  __shared__ int warp_tot[8];
  if (threadIdx.x == 0) {
    s_prefix = 0;
    s_mask = 0;
    s_need = M;
  }
  for (int shift = 24; shift >= 0; shift -= 8) {
    hist[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t prefix = s_prefix, mask = s_mask;
    for (int j = threadIdx.x; j < n; j += 256) {
      const uint32_t k = order_key(z[j]);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int cum = 0;
      for (int b = 255; b >= 0; b--) {
        if (cum + (int)hist[b] >= s_need) {
          s_prefix = prefix | ((uint32_t)b << shift);
          s_need -= cum;
          break;
        }
        cum += (int)hist[b];
      }
      s_mask = mask | (255u << shift);
    }
    __syncthreads();
  }
  const uint32_t T = s_prefix;
  const int need = s_need;  // how many keys equal to T are taken
  int gt_before = 0, eq_before = 0;
  for (int base = 0; base < n; base += 256) {
    const int j = base + threadIdx.x;
    const uint32_t k = j < n ? order_key(z[j]) : 0u;
    const int gt = j < n && k > T, eq = j < n && k == T;
    int tgt, teq;
    const int pg = block_prefix(gt, warp_tot, &tgt);
    const int pe = block_prefix(eq, warp_tot, &teq);
    if (gt) out[gt_before + pg] = j;
    if (eq && eq_before + pe < need) out[(M - need) + eq_before + pe] = j;
    gt_before += tgt;
    eq_before += teq;
  }
}

cudaError_t launch_topm(const float* logits, int64_t B, int64_t n, int64_t ld, int M,
                        int32_t* cand, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  // Rows of up to four chunks that are streamed (no sample) are bound by the selection, two
  // CTAs an SM at a time; with more of them than five an SM the histograms' eight CTAs of
  // 256 threads finish earlier (2048 x 1380, M = 64: 59 and 46 us; 2048 x 9000, M = 4096:
  // 195 and 134; 800 x 1380, M = 64: 29 and 27; but 100 x 1380, M = 512: 11 and 25;
  // 2048 x 100, M = 100: 35 and 44; 2048 x 20000, M = 4096, ties: 240 and 292).
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool by_histograms =
      topm_rank(n, M) == 0 && n > 128 && n <= 4 * kTopChunk && B > 5 * sms;
  if (M <= kTopHold && !by_histograms) {
    const bool vec = ld % 4 == 0 && ((uintptr_t)logits & 15) == 0;
    auto kern = vec ? topm_stream_kernel<true> : topm_stream_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTopSmem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)B, kTopThreads, kTopSmem, s>>>(logits, ld, (int)n, M, topm_rank(n, M), cand);
    return cudaGetLastError();
  }
  topm_kernel<<<(unsigned)B, 256, 0, s>>>(logits, ld, (int)n, M, cand);
  return cudaGetLastError();
}

// ------------------------------------------------- training targets (top R) --
// Per frame (one thread, reading its frame-major scores sequentially): the R
// largest stored dense scores over rows [0, nrot) and their softmax
// (targets proportional to the dense responsibilities). iperm (may be NULL):
// the scores are in emc_iteration's internal frame order, frame k in column
// iperm[k]; live (may be NULL): only the row tiles t with
// live[t * (ld / 256) + column / 256] were contracted (the others hold no score).
__global__ void topr_columns_kernel(const float* __restrict__ S, int64_t ldS,
                                    const float* __restrict__ Sref, int64_t ld, int64_t nrot,
                                    int64_t n_data, int R, const int32_t* __restrict__ iperm,
                                    const uint8_t* __restrict__ live,
                                    int32_t* __restrict__ tidx, float* __restrict__ tprob) {
  const int64_t kk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (kk >= n_data) return;
  const int64_t k = iperm ? iperm[kk] : kk;  // the score column
  const uint8_t* lv = live ? live + (k >> 8) : nullptr;
  const int64_t nnt = ld >> 8;
  float val[kMaxTargets];
  int idx[kMaxTargets];
  for (int r = 0; r < R; r++) {
    val[r] = -INFINITY;
    idx[r] = 0;
  }
  int mpos = 0;
  float mval = -INFINITY;
  for (int64_t j = 0; j < nrot; j++) {
    if (lv && !lv[(j >> 7) * nnt]) {
      j |= 127;  // a tile not contracted: its scores underflow next to the frame's best
      continue;
    }
    const float v = S[k * ldS + j] + Sref[(j >> 5) * ld + k];
    if (v > mval) {
      val[mpos] = v;
      idx[mpos] = (int)j;
      mval = val[0];
      mpos = 0;
      for (int r = 1; r < R; r++)
        if (val[r] < mval) {
          mval = val[r];
          mpos = r;
        }
    }
  }
  float mx = -INFINITY;
  for (int r = 0; r < R; r++) mx = fmaxf(mx, val[r]);
  float sum = 0.f;
  for (int r = 0; r < R; r++) sum += __expf(val[r] - mx);
  for (int r = 0; r < R; r++) {
    tidx[kk * R + r] = idx[r];
    tprob[kk * R + r] = __expf(val[r] - mx) / sum;
  }
}

cudaError_t launch_topr_columns(const float* S, int64_t ldS, const float* Sref, int64_t ld,
                                int64_t nrot, int64_t n_data, int R, int32_t* tidx, float* tprob,
                                cudaStream_t s, const int32_t* iperm, const uint8_t* live) {
  if (R < 1 || R > kMaxTargets) return cudaErrorInvalidValue;
  topr_columns_kernel<<<(unsigned)((n_data + 127) / 128), 128, 0, s>>>(
      S, ldS, Sref, ld, nrot, n_data, R, iperm, live, tidx, tprob);
  return cudaGetLastError();
}

// --------------------------------------------------------- CSR by rotation --
// An index outside the sampling becomes -1: it is in no list, and its score stays -infinity.
__global__ void csr_count_kernel(int32_t* __restrict__ cand, int64_t n_pairs, int64_t n_rot,
                                 int32_t* __restrict__ cnt, int32_t* status) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_pairs) return;
  const int32_t j = cand[e];
  if (j < 0 || j >= n_rot) {
    set_status(status, EMC_ERR_ARG);
    cand[e] = -1;
    return;
  }
  atomicAdd(&cnt[j], 1);
}

// exclusive scan of cnt[0, n) into off[0, n] with one CTA of 1024 threads: four
// counts a thread and a block scan at a time (a thread's run of all its counts and a serial
// pass over the 1024 sums took 8 us for 26 counts, 14 us for 7840; now 3 and 8 us)
__global__ void __launch_bounds__(1024)
    csr_scan_kernel(const int32_t* __restrict__ cnt, int64_t n, int64_t* __restrict__ off) {
  __shared__ int64_t part[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t carry = 0;
  for (int64_t b = 0; b < n; b += 4096) {
    const int64_t i = b + 4 * threadIdx.x;
    int64_t v[4], own = 0;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      v[u] = i + u < n ? cnt[i + u] : 0;
      own += v[u];
    }
    int64_t inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    __syncthreads();  // part is free
    if (lane == 31) part[wid] = inc;
    __syncthreads();
    int64_t w = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    const int64_t before = __shfl_sync(0xffffffffu, w, wid > 0 ? wid - 1 : 0);
    int64_t acc = carry + (wid > 0 ? before : 0) + inc - own;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (i + u < n) off[i + u] = acc;
      acc += v[u];
    }
    carry += __shfl_sync(0xffffffffu, w, 31);
  }
  if (threadIdx.x == 0) off[n] = carry;
}

__global__ void csr_fill_kernel(const int32_t* __restrict__ cand, int64_t n_pairs, int M,
                                const int64_t* __restrict__ off, int32_t* __restrict__ cur,
                                int2* __restrict__ ent, double* __restrict__ Sc) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_pairs) return;
  const int32_t j = cand[e];
  if (j < 0) {
    Sc[e] = -INFINITY;
    return;
  }
  const int64_t pos = off[j] + atomicAdd(&cur[j], 1);
  ent[pos] = make_int2((int)(e / M), (int)(e % M));
}

// Candidate sets from two ranked lists per frame: the R entries of `first`
// (distinct; the dense E-step's top R), then the entries of `rest` (the
// network's top list) that are not among them, in order, until M are written.
// With M_rest >= M at most R entries of rest repeat first, so M are always
// found. One warp per frame; membership by broadcasting first's entries.
__global__ void merge_candidates_kernel(const int32_t* __restrict__ first, int R,
                                        const int32_t* __restrict__ rest, int M_rest,
                                        int64_t n, int M, int32_t* __restrict__ out) {
  const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (k >= n) return;
  const int32_t* f = first + k * R;
  const int32_t* r = rest + k * M_rest;
  int32_t* o = out + k * M;
  const int32_t f0 = lane < R ? f[lane] : -1;
  const int32_t f1 = lane + 32 < R ? f[lane + 32] : -1;
  const int nf = R < M ? R : M;
  for (int t = lane; t < nf; t += 32) o[t] = f[t];
  int filled = nf;
  for (int base = 0; base < M_rest && filled < M; base += 32) {
    const int32_t c = base + lane < M_rest ? r[base + lane] : -1;
    bool dup = c < 0;
    for (int t = 0; t < R; t++) {
      const int32_t v = __shfl_sync(0xffffffffu, t < 32 ? f0 : f1, t & 31);
      dup |= v == c;
    }
    const unsigned keep = __ballot_sync(0xffffffffu, !dup);
    const int pos = filled + __popc(keep & ((1u << lane) - 1u));
    if (!dup && pos < M) o[pos] = c;
    filled += __popc(keep);
  }
}

cudaError_t launch_merge_candidates(const int32_t* first, int R, const int32_t* rest, int M_rest,
                                    int64_t n, int M, int32_t* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  merge_candidates_kernel<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(first, R, rest, M_rest, n, M,
                                                                  out);
  return cudaGetLastError();
}

cudaError_t launch_scan_counts(const int32_t* cnt, int64_t n, int64_t* off, cudaStream_t s) {
  csr_scan_kernel<<<1, 1024, 0, s>>>(cnt, n, off);
  return cudaGetLastError();
}

cudaError_t launch_csr_build(int32_t* cand, int64_t n_data, int M, int64_t n_rot, int64_t rows,
                             int32_t* cnt, int64_t* off, int2* ent, double* Sc, int32_t* status,
                             cudaStream_t s) {
  const int64_t n_pairs = n_data * M;
  cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * rows, s);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((n_pairs + 255) / 256);
  csr_count_kernel<<<blocks, 256, 0, s>>>(cand, n_pairs, n_rot, cnt, status);
  csr_scan_kernel<<<1, 1024, 0, s>>>(cnt, rows, off);
  if ((e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * rows, s)) != cudaSuccess) return e;
  csr_fill_kernel<<<blocks, 256, 0, s>>>(cand, n_pairs, M, off, cnt, ent, Sc);
  return cudaGetLastError();
}

// ------------------------------------------------------ sparse contractions --
// two frame counts packed in 32 bits (BF16 or FP16 frames)
template <bool KF16>
__device__ __forceinline__ void unpack2(uint32_t w, float& lo, float& hi) {
  if (KF16) {
    lo = fp16_val((uint16_t)(w & 0xffffu));
    hi = fp16_val((uint16_t)(w >> 16));
  } else {
    lo = __uint_as_float(w << 16);
    hi = __uint_as_float(w & 0xffff0000u);
  }
}

// log W_ij as the contraction sees it, hi + rest with hi on the precision's grid (1/8; FP16
// split: 1/64).
template <int PREC>
__device__ __forceinline__ void row_parts(const void* __restrict__ L, int64_t plane_stride,
                                          int64_t o, float& h, float& r) {
  if (PREC == EMC_PREC_FP32) {
    const float x = reinterpret_cast<const float*>(L)[o];
    h = rintf(x * 8.f) * 0.125f;
    r = x - h;
  } else if (PREC == EMC_PREC_FP16_SPLIT) {
    const uint16_t* Lb = reinterpret_cast<const uint16_t*>(L) + o;
    h = fp16_val(Lb[0]);
    r = fp16_val(Lb[plane_stride]);
  } else {
    const uint16_t* Lb = reinterpret_cast<const uint16_t*>(L) + o;
    h = bf16_val(Lb[0]);
    if (PREC == EMC_PREC_BF16_SPLIT) {
      r = bf16_val(Lb[plane_stride]) + bf16_val(Lb[2 * plane_stride]);
    } else {
      r = h;
      h = rintf(h * 8.f) * 0.125f;
      r -= h;
    }
  }
}

// Scores from the frames' non-zero lists (a pixel and its count in 32 bits an entry). One CTA
// per rotation row, a warp per pair. log W_j is staged as integers in units of 2^-24 (hi
// exactly, the rest to 2^-25, below the split's own rounding), so the sums are integer and
// exact: nothing depends on their order or on the size of scores and bias.
//  * Lists of few entries on average: one gather an entry, of the 32-bit integer. A lane
//    finishes the pairs that the warp summed for it, 32 at a time: an FP64 instruction
//    takes a warp 16 cycles of its pipe however few lanes need it, and five a pair took as long
//    as a short list's gathers.
//  * Longer ones (lists_long): first the upper 16 bits alone, whose gathers meet half the bank
//    conflicts (neighbouring entries are near pixels), bound S_jk to N_k / 256. Only pairs that
//    may lie within 111 of their frame's best are then given the lower 16 bits' sum; the
//    others' P is 0 in FP32 and their share of the log-sum-exp below FP64's rounding.
// 64^3, 20000 frames of 710 entries x 512 candidates: two FP32 gathers an entry (seven shared-memory
// wavefronts) 5.25 ms, one integer gather 4.19, two stages 3.56; 32^3, 8000 x 512, 92 entries 1.08 ms,
// 0.49, 1.24.
// A row with a value beyond +-127.8 or not finite (no model's log W is, but FP32's of a
// zero floor) sums its parts in FP32 from memory, as such values always were.
constexpr float kFixUnits = 16777216.f;
constexpr size_t kSparseRowMax = 232448;  // a row of hi and rest in a CTA's shared memory

// hi + rest in units of 2^-24 (to integers by adding 1.5 2^23: the conversion runs on the
// FP64 pipe); beyond is set where they do not fit.
__device__ __forceinline__ int fixed_value(float h, float r, bool& beyond) {
  beyond |= !(fabsf(h) < 127.8f && fabsf(r) < 0.1f);
  const int hq = __float_as_int(fmaf(h, 64.f, 12582912.f)) - 0x4b400000;
  const int rq = __float_as_int(fmaf(r, kFixUnits, 12582912.f)) - 0x4b400000;
  return hq * (1 << 18) + rq;
}

// A row of L as integers, two pixels at a time: put(i / 2, values). By the CTA's 256 threads;
// returns, behind a barrier, whether a value lies beyond.
template <int PREC, class Put>
__device__ __forceinline__ bool stage_row(const void* __restrict__ L, int64_t plane_stride,
                                          int64_t row, int64_t ld_pix, Put put) {
  bool beyond = false;
  if (PREC == EMC_PREC_FP32 || ((uintptr_t)L & 3)) {
    for (int64_t i = 2 * threadIdx.x; i < ld_pix; i += 512) {
      float h[2], r[2];
#pragma unroll
      for (int u = 0; u < 2; u++) row_parts<PREC>(L, plane_stride, row + i + u, h[u], r[u]);
      put(i / 2, make_int2(fixed_value(h[0], r[0], beyond), fixed_value(h[1], r[1], beyond)));
    }
  } else {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint16_t*>(L) + row);
    const int64_t next = plane_stride / 2;  // planes are whole rows of 64
    for (int64_t i = threadIdx.x; i < ld_pix / 2; i += 256) {
      const uint32_t a = p[i];
      const uint32_t b = PREC == EMC_PREC_BF16 ? 0u : p[i + next];
      const uint32_t c = PREC == EMC_PREC_BF16_SPLIT ? p[i + 2 * next] : 0u;
      int q[2];
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const uint16_t x = (uint16_t)(a >> (16 * u)), y = (uint16_t)(b >> (16 * u));
        float h, r;
        if (PREC == EMC_PREC_FP16_SPLIT) {
          h = fp16_val(x);
          r = fp16_val(y);
        } else if (PREC == EMC_PREC_BF16_SPLIT) {
          h = bf16_val(x);
          r = bf16_val(y) + bf16_val((uint16_t)(c >> (16 * u)));
        } else {
          h = rintf(bf16_val(x) * 8.f) * 0.125f;
          r = bf16_val(x) - h;
        }
        q[u] = fixed_value(h, r, beyond);
      }
      put(i, make_int2(q[0], q[1]));
    }
  }
  return __syncthreads_or(beyond);
}

template <int PREC>
__device__ __forceinline__ double sum_parts(const void* __restrict__ L, int64_t plane_stride,
                                            int64_t row, const int64_t* __restrict__ koff,
                                            const uint32_t* __restrict__ kent) {
  float ah = 0.f, ar = 0.f;
  for (int64_t f = koff[0] + (threadIdx.x & 31); f < koff[1]; f += 32) {
    float h, r;
    row_parts<PREC>(L, plane_stride, row + (kent[f] & 0xffffu), h, r);
    ah = fmaf((float)(kent[f] >> 16), h, ah);
    ar = fmaf((float)(kent[f] >> 16), r, ar);
  }
  for (int o = 16; o; o >>= 1) {
    ah += __shfl_xor_sync(0xffffffffu, ah, o);
    ar += __shfl_xor_sync(0xffffffffu, ar, o);
  }
  return (double)ah + (double)ar;
}

// Whether the frames' lists take the two stages: the mean number of entries, from
// `least` on (0: never).
__device__ __forceinline__ bool lists_long(const int64_t* __restrict__ koff, int64_t n_data,
                                           int least) {
  return least > 0 && koff[n_data] >= least * n_data;
}

template <int PREC>
__device__ __forceinline__ void score_row(const void* __restrict__ L, int64_t plane_stride,
                                          int64_t ld_pix, const double* __restrict__ bias,
                                          int64_t j, int64_t e0, int64_t e1,
                                          const int2* __restrict__ ent, int M,
                                          const int64_t* __restrict__ koff,
                                          const uint32_t* __restrict__ kent, int2* Lq2,
                                          double* __restrict__ Sc) {
  const int* Lq = reinterpret_cast<const int*>(Lq2);
  const int lane = threadIdx.x & 31;
  const bool beyond = stage_row<PREC>(L, plane_stride, j * ld_pix, ld_pix,
                                      [&](int64_t i2, int2 q) { Lq2[i2] = q; });
  const double bj = bias[j];
  for (int64_t b = e0 + (threadIdx.x >> 5); b < e1; b += 256) {
    const bool on = b + 8 * lane < e1;  // the CTA's warps take the list's pairs in turn
    const int2 mine = on ? ent[b + 8 * lane] : make_int2(0, 0);
    const int pairs = (int)min((int64_t)32, (e1 - b + 7) / 8);
    double own = 0.0;
    if (!beyond) {
      long long sum = 0;
      for (int src = 0; src < pairs; src++) {
        const int k = __shfl_sync(0xffffffffu, mine.x, src);
        const int64_t f0 = koff[k];
        const int n = (int)(koff[k + 1] - f0);
        const uint32_t* list = kent + f0;
        long long acc = 0;
        for (int f = lane; f < n; f += 128) {
          uint32_t w[4];
#pragma unroll
          for (int u = 0; u < 4; u++) w[u] = f + 32 * u < n ? list[f + 32 * u] : 0u;
#pragma unroll
          for (int u = 0; u < 4; u++) acc += (long long)(int)(w[u] >> 16) * Lq[w[u] & 0xffffu];
        }
        // |acc| < 2^47 (N_k < 2^16): 24 bits and the rest, each summed in one instruction
        const unsigned low = __reduce_add_sync(0xffffffffu, (unsigned)(acc & 0xffffff));
        const int high = __reduce_add_sync(0xffffffffu, (int)(acc >> 24));
        if (lane == src) sum = ((long long)high << 24) + low;
      }
      own = (double)sum * (1.0 / kFixUnits);
    } else {
      for (int src = 0; src < pairs; src++) {
        const int k = __shfl_sync(0xffffffffu, mine.x, src);
        const double sum = sum_parts<PREC>(L, plane_stride, j * ld_pix, koff + k, kent);
        if (lane == src) own = sum;
      }
    }
    if (on) Sc[(int64_t)mine.x * M + mine.y] = own + bj;
  }
}

// Stage one: the sum of the upper 16 bits (units of 2^-8) into the place of the pair's P. With
// the bias, S_jk is within [0, N_k / 256) above it (S^u_jk). The choice compares these in
// units of 2^-18 as 64-bit integers (FP64 took 100 us of 3.6 ms), with the biases in
// `ubias` (|bias| by at most 2^43: beyond, rows go by that limit; one that is not finite
// keeps its pairs).
constexpr int kPairBeyond = INT_MIN, kPairLeft = INT_MIN + 1;  // to be scored; not to be
constexpr long long kBoundKeep = LLONG_MAX;
__device__ __forceinline__ long long bound_bias(double b) {
  const double x = b * 0x1p18;
  if (!isfinite(x)) return kBoundKeep;
  return __double2ll_rn(fmin(fmax(x, -0x1p61), 0x1p61));
}
template <int PREC>
__device__ __forceinline__ void bound_row(const void* __restrict__ L, int64_t plane_stride,
                                          int64_t ld_pix, const double* __restrict__ bias,
                                          int64_t j, int64_t e0, int64_t e1,
                                          const int2* __restrict__ ent, int M,
                                          const int64_t* __restrict__ koff,
                                          const uint32_t* __restrict__ kent, int2* Lq2,
                                          long long* __restrict__ ubias,
                                          int* __restrict__ upper) {
  const int16_t* Lu = reinterpret_cast<const int16_t*>(Lq2);
  if (threadIdx.x == 0) ubias[j] = bound_bias(bias[j]);
  const bool beyond =
      stage_row<PREC>(L, plane_stride, j * ld_pix, ld_pix, [&](int64_t i2, int2 q) {
        reinterpret_cast<unsigned*>(Lq2)[i2] = __byte_perm(q.x, q.y, 0x7632);
      });
  const int lane = threadIdx.x & 31;
  for (int64_t e = e0 + (threadIdx.x >> 5); e < e1; e += 8) {
    const int2 km = ent[e];
    const int64_t f0 = koff[km.x];
    const int n = (int)(koff[km.x + 1] - f0);
    const uint32_t* list = kent + f0;
    int sum = 0;  // below 65535 x 32743 < 2^31
    int f = lane;
    for (; f + 96 < n; f += 128) {
      uint32_t w[4];
#pragma unroll
      for (int u = 0; u < 4; u++) w[u] = list[f + 32 * u];
#pragma unroll
      for (int u = 0; u < 4; u++) sum += (int)(w[u] >> 16) * Lu[w[u] & 0xffffu];
    }
    for (; f < n; f += 32) {
      const uint32_t w = list[f];
      sum += (int)(w >> 16) * Lu[w & 0xffffu];
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) upper[(int64_t)km.x * M + km.y] = beyond ? kPairBeyond : sum;
  }
}

// A CTA per rotation row, in the form that the lists' length asks for. FORM: both in one launch,
// or one of them alone (a launch of 50100 CTAs that find nothing to do takes 33 us), where
// eight CTAs' 32-bit rows exceed an SM's shared memory and the 16-bit ones want less.
enum { kFormBoth = 0, kFormScore = 1, kFormBound = 2 };
template <int PREC, int FORM>
__global__ void __launch_bounds__(256, 8)
    sparse_rows_kernel(const void* __restrict__ L, int64_t plane_stride, int64_t ld_pix,
                       const double* __restrict__ bias, const int64_t* __restrict__ off,
                       const int2* __restrict__ ent, int M, const int64_t* __restrict__ koff,
                       const uint32_t* __restrict__ kent, int64_t n_data, int least,
                       long long* __restrict__ ubias, int* __restrict__ upper,
                       double* __restrict__ Sc) {
  const int64_t j = blockIdx.x;
  const int64_t e0 = off[j], e1 = off[j + 1];
  if (e0 == e1) return;
  extern __shared__ int2 Lq2[];
  const bool two = lists_long(koff, n_data, least);
  if (FORM != kFormScore && two)
    bound_row<PREC>(L, plane_stride, ld_pix, bias, j, e0, e1, ent, M, koff, kent, Lq2, ubias, upper);
  if (FORM != kFormBound && !two)
    score_row<PREC>(L, plane_stride, ld_pix, bias, j, e0, e1, ent, M, koff, kent, Lq2, Sc);
}

// One warp per frame: the pairs whose score is not needed are marked and get -infinity.
__global__ void __launch_bounds__(256)
    sparse_choose_kernel(const int64_t* __restrict__ koff, const uint32_t* __restrict__ kent,
                         int64_t n_data, int least, int M, const int32_t* __restrict__ cand,
                         const long long* __restrict__ ubias, int* __restrict__ upper,
                         double* __restrict__ Sc) {
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= n_data || !lists_long(koff, n_data, least)) return;
  int total = 0;  // N_k < 65536
  for (int64_t f = koff[k] + lane; f < koff[k + 1]; f += 32) total += (int)(kent[f] >> 16);
  total = __reduce_add_sync(0xffffffffu, total);
  int* u = upper + k * M;
  const int32_t* c = cand + k * M;
  auto bound = [&](int m) {  // S^u of pair m, or kBoundKeep; LLONG_MIN: no rotation
    if (c[m] < 0) return LLONG_MIN;
    const int x = u[m];
    const long long b = ubias[c[m]];
    return x == kPairBeyond || b == kBoundKeep ? kBoundKeep : b + ((long long)x << 10);
  };
  long long mx = LLONG_MIN;
#pragma unroll 4
  for (int m = lane; m < M; m += 32) {
    const long long x = bound(m);
    if (x != kBoundKeep) mx = max(mx, x);
  }
  for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  // N_k / 256 + 112, where 111 and the bias's rounding are enough
  const long long gap = 1024ll * total + (112ll << 18);
  const long long bottom = mx == LLONG_MIN ? mx + 1 : mx - gap;
#pragma unroll 4
  for (int m = lane; m < M; m += 32)
    if (bound(m) < bottom) {
      u[m] = kPairLeft;
      Sc[k * M + m] = -INFINITY;
    }
}

// Stage two: the lower 16 bits' sums of the needed pairs on top. The CTAs take rows in turn (a
// grid of the SMs' own number: where lists are short nothing is left to do).
template <int PREC>
__global__ void __launch_bounds__(256, 8)
    sparse_lower_kernel(const void* __restrict__ L, int64_t plane_stride, int64_t ld_pix,
                        int64_t rows, const double* __restrict__ bias,
                        const int64_t* __restrict__ off, const int2* __restrict__ ent, int M,
                        const int64_t* __restrict__ koff, const uint32_t* __restrict__ kent,
                        int64_t n_data, int least, const int* __restrict__ upper,
                        double* __restrict__ Sc) {
  if (!lists_long(koff, n_data, least)) return;
  extern __shared__ int2 Lq2[];
  const uint16_t* Ll = reinterpret_cast<const uint16_t*>(Lq2);
  const int lane = threadIdx.x & 31;
  for (int64_t j = blockIdx.x; j < rows; j += gridDim.x) {
    const int64_t e0 = off[j], e1 = off[j + 1];
    bool any = false;  // a row without a needed pair is passed over
    for (int64_t e = e0 + threadIdx.x; e < e1; e += 256) {
      const int2 km = ent[e];
      any |= upper[(int64_t)km.x * M + km.y] != kPairLeft;
    }
    if (!__syncthreads_or(any)) continue;
    const bool beyond =
        stage_row<PREC>(L, plane_stride, j * ld_pix, ld_pix, [&](int64_t i2, int2 q) {
          reinterpret_cast<unsigned*>(Lq2)[i2] = __byte_perm(q.x, q.y, 0x5410);
        });
    const double bj = bias[j];
    for (int64_t b = e0 + (threadIdx.x >> 5); b < e1; b += 256) {
      const int64_t e = b + 8 * lane;
      const int2 mine = e < e1 ? ent[e] : make_int2(0, 0);
      const int64_t at = (int64_t)mine.x * M + mine.y;
      const int up = e < e1 ? upper[at] : kPairLeft;
      const bool on = up != kPairLeft;
      unsigned todo = __ballot_sync(0xffffffffu, on);
      double parts = 0.0;
      unsigned low = 0;
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int k = __shfl_sync(0xffffffffu, mine.x, src);
        if (beyond) {
          const double x = sum_parts<PREC>(L, plane_stride, j * ld_pix, koff + k, kent);
          if (lane == src) parts = x;
          continue;
        }
        const int64_t f1 = koff[k + 1];
        unsigned sum = 0;  // below 65535 x 65535 < 2^32
        for (int64_t f = koff[k] + lane; f < f1; f += 32) {
          const uint32_t w = kent[f];
          sum += (w >> 16) * Ll[w & 0xffffu];
        }
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == src) low = sum;
      }
      if (on)
        Sc[at] = (beyond ? parts : (double)(((long long)up << 16) + low) * (1.0 / kFixUnits)) + bj;
    }
    __syncthreads();  // the row is staged anew
  }
}

// One CTA per rotation row: log W_j split into (hi on the 1/8 grid, rest) in
// shared memory; each warp takes pairs (frame, slot) of the row's list, two
// at a time, reading the frames' K rows 8 pixels (16 bytes) per lane.
template <int PREC>
__global__ void __launch_bounds__(256)
    sparse_scores_kernel(const void* __restrict__ L, int64_t plane_stride, int64_t ld_pix,
                         const double* __restrict__ bias, const uint16_t* __restrict__ Kb,
                         const int64_t* __restrict__ off, const int2* __restrict__ ent, int M,
                         double* __restrict__ Sc) {
  const int64_t j = blockIdx.x;
  const int64_t e0 = off[j], e1 = off[j + 1];
  if (e0 == e1) return;
  extern __shared__ float4 sm4[];
  float* Lh = reinterpret_cast<float*>(sm4);
  float* Lr = Lh + ld_pix;
  for (int64_t i = threadIdx.x; i < ld_pix; i += blockDim.x)
    row_parts<PREC>(L, plane_stride, j * ld_pix + i, Lh[i], Lr[i]);
  __syncthreads();
  const double bj = bias[j];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t n8 = ld_pix / 8;
  for (int64_t e = e0 + 2 * wid; e < e1; e += 2 * nw) {
    const bool two = e + 1 < e1;
    const int2 ka = ent[e];
    const int2 kb = two ? ent[e + 1] : ka;
    const uint4* Ka = reinterpret_cast<const uint4*>(Kb + (int64_t)ka.x * ld_pix);
    const uint4* Kc = reinterpret_cast<const uint4*>(Kb + (int64_t)kb.x * ld_pix);
    float ah = 0.f, ar = 0.f, bh = 0.f, br = 0.f;
    for (int64_t g = lane; g < n8; g += 32) {
      const uint4 wa = Ka[g], wb = Kc[g];
      const float4 h0 = reinterpret_cast<const float4*>(Lh)[2 * g];
      const float4 h1 = reinterpret_cast<const float4*>(Lh)[2 * g + 1];
      const float4 r0 = reinterpret_cast<const float4*>(Lr)[2 * g];
      const float4 r1 = reinterpret_cast<const float4*>(Lr)[2 * g + 1];
      const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
      const float rv[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
      const uint32_t ua[4] = {wa.x, wa.y, wa.z, wa.w}, ub[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int c = 0; c < 4; c++) {
        float a0, a1, b0, b1;
        unpack2<PREC == EMC_PREC_FP16_SPLIT>(ua[c], a0, a1);
        unpack2<PREC == EMC_PREC_FP16_SPLIT>(ub[c], b0, b1);
        ah = fmaf(a0, hv[2 * c], ah);
        ah = fmaf(a1, hv[2 * c + 1], ah);
        ar = fmaf(a0, rv[2 * c], ar);
        ar = fmaf(a1, rv[2 * c + 1], ar);
        bh = fmaf(b0, hv[2 * c], bh);
        bh = fmaf(b1, hv[2 * c + 1], bh);
        br = fmaf(b0, rv[2 * c], br);
        br = fmaf(b1, rv[2 * c + 1], br);
      }
    }
    for (int o = 16; o; o >>= 1) {
      ah += __shfl_xor_sync(0xffffffffu, ah, o);
      ar += __shfl_xor_sync(0xffffffffu, ar, o);
      bh += __shfl_xor_sync(0xffffffffu, bh, o);
      br += __shfl_xor_sync(0xffffffffu, br, o);
    }
    if (lane == 0) {
      Sc[(int64_t)ka.x * M + ka.y] = ((double)ah + (double)ar) + bj;
      if (two) Sc[(int64_t)kb.x * M + kb.y] = ((double)bh + (double)br) + bj;
    }
  }
}

// One warp per frame: lse over the frame's M candidates, P = exp(S - lse).
// shift (may be NULL): per-frame constant the scores carry (Poisson-fluence
// model), removed from the lse written out.
__global__ void sparse_lse_kernel(const double* __restrict__ Sc, int64_t n_data, int64_t ld_data,
                                  int M, float* __restrict__ Pc, double* __restrict__ lse_c,
                                  const double* __restrict__ shift, int32_t* status) {
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= ld_data) return;
  const double* s = Sc + k * M;
  float* p = Pc + k * M;
  if (k >= n_data) {
    for (int m = lane; m < M; m += 32) p[m] = 0.f;
    return;
  }
  double mx = -INFINITY;
  for (int m = lane; m < M; m += 32) mx = fmax(mx, s[m]);
  for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  double sum = 0.0;
  for (int m = lane; m < M; m += 32) sum += (double)__expf((float)(s[m] - mx));
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const double lse = mx + log(sum);
  if (!isfinite(lse)) set_status(status, EMC_ERR_NUMERIC);
  for (int m = lane; m < M; m += 32) p[m] = __expf((float)(s[m] - lse));
  if (lane == 0) lse_c[k] = lse - (shift ? shift[k] : 0.0);
}

// The pairs [s0, s0 + ns) of a row's list (ns <= kUpdSeg) with a non-zero weight, packed into
// (sk, sp) in list order; returns their number (the same in every thread) and
// adds the thread's share of the pairs' P to dsum. Most P of a candidate set
// underflow to exact zeros (64^3, 512 candidates: 1.6 of 512 are not), which
// add nothing to Num. Called by all 256 threads; sk and sp are free on entry.
constexpr int kUpdSeg = 1024;
struct UpdList {
  int k[kUpdSeg];
  float p[kUpdSeg];
  int warp_tot[8];
};
__device__ __forceinline__ int pack_pairs(UpdList& u, const int2* __restrict__ ent, int ns, int M,
                                          const float* __restrict__ Pc, bool flu, float Bj,
                                          const float* __restrict__ invn, float& dsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int n = 0;
  for (int t0 = 0; t0 < ns; t0 += 256) {
    const int t = t0 + threadIdx.x;
    int k = 0;
    float p = 0.f;
    if (t < ns) {
      const int2 km = ent[t];
      k = km.x;
      p = Pc[(int64_t)km.x * M + km.y];
      dsum += p;
      if (flu) p *= Bj * invn[k];
    }
    const unsigned keep = __ballot_sync(0xffffffffu, p != 0.f);  // a NaN is kept
    if (lane == 0) u.warp_tot[wid] = __popc(keep);
    __syncthreads();
    int at = n;
#pragma unroll
    for (int w = 0; w < 8; w++) {
      if (w < wid) at += u.warp_tot[w];
      n += u.warp_tot[w];
    }
    if (p != 0.f) {
      at += __popc(keep & ((1u << lane) - 1u));
      u.k[at] = k;
      u.p[at] = p;
    }
    __syncthreads();
  }
  return n;
}

// sum of v over the CTA's 256 threads, in thread 0
__device__ __forceinline__ float cta_sum(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float d = 0.f;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; w++) d += red[w];
  return d;
}

// One CTA per rotation row: Num_j = sum over the row's pairs with a non-zero
// weight of P_jk K_k; den_j = sum of the row's P_jk. Each thread owns 8
// consecutive pixels (one 16-byte load of a K row per pair), walking the packed
// pairs four at a time. Rows without pairs are zeroed. Poisson-fluence model
// (Bsum != NULL): the weights are P_jk B_j / N_k. vec: Num is 16-byte aligned.
template <bool KF16>
__global__ void __launch_bounds__(256)
    sparse_update_kernel(const uint16_t* __restrict__ Kb, int64_t ld_pix,
                         const int64_t* __restrict__ off, const int2* __restrict__ ent, int M,
                         const float* __restrict__ Pc, float* __restrict__ Num,
                         float* __restrict__ den, const double* __restrict__ Bsum,
                         const float* __restrict__ invn, bool vec) {
  const int64_t j = blockIdx.x;
  const int64_t e0 = off[j], e1 = off[j + 1];
  float* out = Num + j * ld_pix;
  __shared__ UpdList u;
  __shared__ float red[8];
  const bool flu = Bsum != nullptr;
  const float Bj = flu ? (float)Bsum[j] : 0.f;
  float dsum = 0.f;
  const int64_t n8 = ld_pix / 8;
  const bool one = e1 - e0 <= kUpdSeg;  // the list is packed once for every pixel
  int n = one ? pack_pairs(u, ent + e0, (int)(e1 - e0), M, Pc, flu, Bj, invn, dsum) : 0;
  for (int64_t g0 = 0; g0 < n8; g0 += 256) {
    const int64_t g = g0 + threadIdx.x;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int64_t s0 = e0; s0 < e1; s0 += kUpdSeg) {
      if (!one) {
        float again = 0.f;  // den counts every pair once, with the first pixels
        n = pack_pairs(u, ent + s0, (int)min((int64_t)kUpdSeg, e1 - s0), M, Pc, flu, Bj, invn,
                       g0 == 0 ? dsum : again);
      }
      if (g < n8) {
        for (int t = 0; t < n; t += 4) {
          uint4 w[4];
#pragma unroll
          for (int v = 0; v < 4; v++)
            if (t + v < n)
              w[v] = reinterpret_cast<const uint4*>(Kb + (int64_t)u.k[t + v] * ld_pix)[g];
#pragma unroll
          for (int v = 0; v < 4; v++) {
            if (t + v >= n) break;
            const float p = u.p[t + v];
            const uint32_t wv[4] = {w[v].x, w[v].y, w[v].z, w[v].w};
#pragma unroll
            for (int c = 0; c < 4; c++) {
              float k0, k1;
              unpack2<KF16>(wv[c], k0, k1);
              acc[2 * c] = fmaf(p, k0, acc[2 * c]);
              acc[2 * c + 1] = fmaf(p, k1, acc[2 * c + 1]);
            }
          }
        }
      }
      if (!one) __syncthreads();
    }
    if (g < n8 && vec) {
      float4* o4 = reinterpret_cast<float4*>(out + 8 * g);
      o4[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      o4[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    } else if (g < n8) {
#pragma unroll
      for (int c = 0; c < 8; c++) out[8 * g + c] = acc[c];
    }
  }
  const float d = cta_sum(dsum, red);
  if (threadIdx.x == 0) den[j] = d;
}

// The same from the frames' non-zero pixel lists: the row Num_j accumulates in
// shared memory (FP32 atomics; a frame's non-zero pixels are distinct), the
// packed pairs shared out over the CTA's warps (several warps to a pair when
// the row has fewer pairs than warps), then is written out whole; a row without
// non-zero weights is written as zeros straight away. 64^3, 20000 frames, 512 candidates:
// every pair's counts added 7.52 ms, the non-zero ones 0.43 ms, where
// the 0.57 GB of Num take 0.08 ms at the copy rate.
__global__ void __launch_bounds__(256)
    sparse_update_csr_kernel(const int64_t* __restrict__ koff, const uint32_t* __restrict__ kent,
                             int64_t ld_pix, const int64_t* __restrict__ off,
                             const int2* __restrict__ ent, int M, const float* __restrict__ Pc,
                             float* __restrict__ Num, float* __restrict__ den,
                             const double* __restrict__ Bsum, const float* __restrict__ invn,
                             bool vec) {
  const int64_t j = blockIdx.x;
  const int64_t e0 = off[j], e1 = off[j + 1];
  extern __shared__ float4 sm4u[];
  float* srow = reinterpret_cast<float*>(sm4u);
  __shared__ UpdList u;
  __shared__ float red[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float Bj = Bsum ? (float)Bsum[j] : 0.f;
  const int64_t n4 = ld_pix / 4;
  float dsum = 0.f;
  bool any = false;
  for (int64_t s0 = e0; s0 < e1; s0 += kUpdSeg) {
    const int n = pack_pairs(u, ent + s0, (int)min((int64_t)kUpdSeg, e1 - s0), M, Pc,
                             Bsum != nullptr, Bj, invn, dsum);
    if (n > 0 && !any) {
      for (int64_t i = threadIdx.x; i < n4; i += 256) sm4u[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
      any = true;
    }
    const int share = n >= 8 || n == 0 ? 1 : 8 / n;  // warps to a pair
    const int teams = 8 / share;
    if (wid < teams * share)
      for (int t = wid / share; t < n; t += teams) {
        const float p = u.p[t];
        const int64_t f1 = koff[u.k[t] + 1];
        for (int64_t f = koff[u.k[t]] + (wid % share) * 32 + lane; f < f1; f += 32 * share) {
          const uint32_t w = kent[f];
          atomicAdd(&srow[w & 0xffffu], p * (float)(w >> 16));
        }
      }
    __syncthreads();  // the list is repacked, or the row written, after this
  }
  float* row = Num + j * ld_pix;
  if (vec) {
    float4* out = reinterpret_cast<float4*>(row);
    for (int64_t i = threadIdx.x; i < n4; i += 256)
      out[i] = any ? sm4u[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    for (int64_t i = threadIdx.x; i < ld_pix; i += 256) row[i] = any ? srow[i] : 0.f;
  }
  const float d = cta_sum(dsum, red);
  if (threadIdx.x == 0) den[j] = d;
}

// 1 - sum_{j in C_k} P_jk of a dense E-step, from its stored scores (lse2 in
// the given frame order). iperm, live (may be NULL): scores in emc_iteration's
// internal order, and the row tiles contracted there (P = 0 in the others).
__global__ void missed_mass_kernel(const float* __restrict__ S, int64_t ldS,
                                   const float* __restrict__ Sref, int64_t ld_data, const float2* __restrict__ lse2,
                                   const int32_t* __restrict__ cand, int M, int64_t n_data,
                                   const int32_t* __restrict__ iperm,
                                   const uint8_t* __restrict__ live, float* __restrict__ missed) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_data) return;
  const int64_t c = iperm ? iperm[k] : k;  // the score column
  const uint8_t* lv = live ? live + (c >> 8) : nullptr;
  const int64_t nnt = ld_data >> 8;
  const float2 L = lse2[k];
  double sum = 0.0;
  for (int m = 0; m < M; m++) {
    const int64_t j = cand[k * M + m];
    if (j < 0) continue;
    if (lv && !lv[(j >> 7) * nnt]) continue;
    const float e = S[c * ldS + j] + ((Sref[(j >> 5) * ld_data + c] - L.x) - L.y);
    sum += (double)__expf(e);
  }
  missed[k] = (float)(1.0 - sum);
}

// Responsibilities of selected frames from stored scores (Eq. 2.4):
// P[f][j] = exp(S_jk - lse_k) for k = frames[f], read like missed_mass_kernel
// (frame-major scores relative to their 32-row group maxima; iperm/live: the
// internal order and contracted tiles of a pruned pass, skipped tiles give 0).
// Grid (ceil(nrot / 256), n): threads along rotations, coalesced in S and P.
__global__ void __launch_bounds__(256)
    responsibilities_kernel(const float* __restrict__ S, int64_t ldS,
                            const float* __restrict__ Sref, int64_t ld_data,
                            const float2* __restrict__ lse2, const int32_t* __restrict__ frames,
                            int64_t nrot, int64_t n_data, const int32_t* __restrict__ iperm,
                            const uint8_t* __restrict__ live, float* __restrict__ P,
                            int32_t* status) {
  const int64_t f = blockIdx.y;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t k = frames[f];
  if (k < 0 || k >= n_data) {
    if (j == 0) set_status(status, EMC_ERR_ARG);
    return;
  }
  if (j >= nrot) return;
  const int64_t c = iperm ? iperm[k] : k;
  float p = 0.f;
  if (!live || live[(j >> 7) * (ld_data >> 8) + (c >> 8)]) {
    const float2 L = lse2[k];
    p = __expf(S[c * ldS + j] + ((Sref[(j >> 5) * ld_data + c] - L.x) - L.y));
  }
  P[f * nrot + j] = p;
}

// lse[k] = m_k + log s_k
__global__ void lse_values_kernel(const double* __restrict__ m, const double* __restrict__ s,
                                  int64_t n, double* __restrict__ lse) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) lse[k] = m[k] + log(s[k]);
}

cudaError_t launch_responsibilities(const float* S, int64_t ldS, const float* Sref,
                                    int64_t ld_data, const float2* lse2, const int32_t* frames,
                                    int64_t n, int64_t nrot, int64_t n_data, float* P,
                                    int32_t* status, cudaStream_t s, const int32_t* iperm,
                                    const uint8_t* live) {
  if (n <= 0) return cudaSuccess;
  dim3 grd((unsigned)((nrot + 255) / 256), (unsigned)n);
  responsibilities_kernel<<<grd, 256, 0, s>>>(S, ldS, Sref, ld_data, lse2, frames, nrot, n_data,
                                              iperm, live, P, status);
  return cudaGetLastError();
}

cudaError_t launch_lse_values(const double* m, const double* sm, int64_t n, double* lse,
                              cudaStream_t s) {
  lse_values_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(m, sm, n, lse);
  return cudaGetLastError();
}

namespace {

// Mean entries of a list from which the two stages run (lists_long), or 0: never. us of a
// call by one gather an entry, and by two stages:
//   pairs a row, entries  204, 710     377, 397     158, 710   159, 266  158, 403  80, 403   80, 199
//                         4194, 3562   1164, 1018   246, 237   924, 897  178, 212  651, 685  428, 736
// Where a row has few pairs, the second launches gain nothing: 20, 710 310, 398; 35, 1527 392, 414.
int two_stages_from(int64_t n_data, int M, int64_t n_rot) {
  return n_data * M >= 64 * n_rot ? 384 : 0;
}

// the first stage of both forms in one launch: eight CTAs' 32-bit rows fit an SM
bool both_forms(size_t row) { return 8 * (row + 1024) <= 233472; }

template <int PREC>
cudaError_t sparse_scores(const Planes& L, int64_t rows, const double* bias, const uint16_t* Kb,
                          int64_t ld_pix, const int64_t* off, const int2* ent, int M,
                          const int64_t* koff, const uint32_t* kent, int64_t n_data,
                          const int32_t* cand, int64_t n_rot, long long* ubias, int* upper,
                          double* Sc, cudaStream_t s) {
  const size_t row = sizeof(float) * (size_t)ld_pix;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e;
  if (!kent) {
    e = cudaFuncSetAttribute(sparse_scores_kernel<PREC>, attr, (int)(2 * row));
    if (e != cudaSuccess) return e;
    sparse_scores_kernel<PREC><<<(unsigned)rows, 256, 2 * row, s>>>(
        L.base, L.plane_stride, ld_pix, bias, Kb, off, ent, M, Sc);
    return cudaGetLastError();
  }
  const int least = two_stages_from(n_data, M, n_rot);
  auto rows_kernel = [&](auto kern, size_t smem) {
    cudaError_t r = cudaFuncSetAttribute(kern, attr, (int)smem);
    if (r != cudaSuccess) return r;
    kern<<<(unsigned)rows, 256, smem, s>>>(L.base, L.plane_stride, ld_pix, bias, off, ent, M, koff,
                                           kent, n_data, least, ubias, upper, Sc);
    return cudaGetLastError();
  };
  if (least == 0) return rows_kernel(sparse_rows_kernel<PREC, kFormScore>, row);
  if ((e = cudaFuncSetAttribute(sparse_lower_kernel<PREC>, attr, (int)(row / 2))) != cudaSuccess)
    return e;
  if (both_forms(row)) {
    e = rows_kernel(sparse_rows_kernel<PREC, kFormBoth>, row);
  } else {
    e = rows_kernel(sparse_rows_kernel<PREC, kFormScore>, row);
    if (e == cudaSuccess) e = rows_kernel(sparse_rows_kernel<PREC, kFormBound>, row / 2);
  }
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  sparse_choose_kernel<<<(unsigned)((n_data * 32 + 255) / 256), 256, 0, s>>>(
      koff, kent, n_data, least, M, cand, ubias, upper, Sc);
  sparse_lower_kernel<PREC><<<(unsigned)std::min<int64_t>(rows, 8 * sms), 256, row / 2, s>>>(
      L.base, L.plane_stride, ld_pix, rows, bias, off, ent, M, koff, kent, n_data, least, upper,
      Sc);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sparse_scores(const Planes& L, int precision, int64_t rows, const double* bias,
                                 const uint16_t* Kb, int64_t ld_pix, const int64_t* off,
                                 const int2* ent, int M, const int64_t* koff,
                                 const uint32_t* kent, int64_t n_data, const int32_t* cand,
                                 int64_t n_rot, long long* ubias, int* upper, double* Sc,
                                 cudaStream_t s) {
  if (2 * sizeof(float) * (size_t)ld_pix > kSparseRowMax) return cudaErrorInvalidValue;
#define EMC_SPARSE_SCORES(P)                                                                    \
  return sparse_scores<P>(L, rows, bias, Kb, ld_pix, off, ent, M, koff, kent, n_data, cand, n_rot, \
                             ubias, upper, Sc, s)
  switch (precision) {
    case EMC_PREC_FP32: EMC_SPARSE_SCORES(EMC_PREC_FP32);
    case EMC_PREC_BF16: EMC_SPARSE_SCORES(EMC_PREC_BF16);
    case EMC_PREC_FP16_SPLIT: EMC_SPARSE_SCORES(EMC_PREC_FP16_SPLIT);
    default: EMC_SPARSE_SCORES(EMC_PREC_BF16_SPLIT);
  }
#undef EMC_SPARSE_SCORES
}

int sparse_score_launches(int64_t n_data, int M, int64_t n_rot, int64_t ld_pix, bool lists) {
  if (!lists || two_stages_from(n_data, M, n_rot) == 0) return 1;
  return both_forms(sizeof(float) * (size_t)ld_pix) ? 3 : 4;
}

cudaError_t launch_sparse_lse(const double* Sc, int64_t n_data, int64_t ld_data, int M, float* Pc,
                              double* lse_c, int32_t* status, cudaStream_t s,
                              const double* shift) {
  sparse_lse_kernel<<<(unsigned)((ld_data * 32 + 255) / 256), 256, 0, s>>>(Sc, n_data, ld_data, M,
                                                                          Pc, lse_c, shift, status);
  return cudaGetLastError();
}

cudaError_t launch_sparse_update(const uint16_t* Kb, int kf16, int64_t ld_pix,
                                 const int64_t* off, const int2* ent, int M, const float* Pc,
                                 int64_t rows, const int64_t* koff, const uint32_t* kent,
                                 float* Num, float* den, cudaStream_t s, const double* Bsum,
                                 const float* invn) {
  if (Bsum && !invn) return cudaErrorInvalidValue;
  const bool vec = ((uintptr_t)Num & 15) == 0;
  // the row of Num and the list share a CTA's 227 KB; between 56064 and 58048
  // pixels, where only the row fits, the frames' rows are read instead
  const size_t smem = sizeof(float) * (size_t)ld_pix;
  if (kent && (smem + sizeof(UpdList) + 256 <= 232448 || smem > 232192)) {
    cudaError_t e = cudaFuncSetAttribute(sparse_update_csr_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    sparse_update_csr_kernel<<<(unsigned)rows, 256, smem, s>>>(koff, kent, ld_pix, off, ent, M, Pc,
                                                               Num, den, Bsum, invn, vec);
    return cudaGetLastError();
  }
  if (kf16)
    sparse_update_kernel<true><<<(unsigned)rows, 256, 0, s>>>(Kb, ld_pix, off, ent, M, Pc,
                                                              Num, den, Bsum, invn, vec);
  else
    sparse_update_kernel<false><<<(unsigned)rows, 256, 0, s>>>(Kb, ld_pix, off, ent, M, Pc,
                                                               Num, den, Bsum, invn, vec);
  return cudaGetLastError();
}

cudaError_t launch_missed_mass(const float* S, int64_t ldS, const float* Sref, int64_t ld_data,
                               const float2* lse2, const int32_t* cand, int M, int64_t n_data,
                               float* missed, cudaStream_t s, const int32_t* iperm,
                               const uint8_t* live) {
  missed_mass_kernel<<<(unsigned)((n_data + 255) / 256), 256, 0, s>>>(
      S, ldS, Sref, ld_data, lse2, cand, M, n_data, iperm, live, missed);
  return cudaGetLastError();
}

}  // namespace emc
