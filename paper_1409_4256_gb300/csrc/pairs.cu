// pairs.cu -- the M-step's operand as short lists of pairs per rotation row.
//
// Frames' posteriors are sharp: of a row's responsibilities one or two are not
// exact zeros (64^3 workload: 26005 of 10^9 pairs over 20257 of 50100 rows). A
// row's numerators sum_k P_jk K_ik (Eq. 2.11) are then a sum of one or two
// frames, and rows without a pair need none: inside an iteration P itself is not
// written, and Num only for rows with mass. A row holds up to kRowPairs pairs; a
// 128-row tile with a longer row, or with more than kTilePairs in all (flat
// posteriors), keeps the tensor-core path over the planes of P, chosen on the
// device tile by tile (over). The pairs of a row are used in frame order, so results do
// not depend on the order in which they were found.
//
// A pair's weight is the value the planes would hold (BF16 hi + lo, or FP16 hi
// + lo of 2^14 P, summed in FP32), so both paths contract the same operand.
//
// Normalisation and update of an iteration: 64^3 (50100 x 20000) 179 + 214 us by planes,
// 65 + 83 us by pairs; 96^3, Poisson fluence (25680 x 10007) 212 + 765 and 177 +
// 132 us; 128^3 (204960 x 100000) 85.5 against 82.6 ms an iteration. emc_update, 64^3
// (10860 x 4999): 362 us contracting 217 MB of planes, of which 6144 elements are not zero; 80 us
// reading them once and writing Num.
// Summing the pairs inside the compression, without Num, took longer than
// writing it (96^3: compression 4.3 against 3.3 ms): it reads a frame's pixels in the
// order of its groups, two bytes at a time, once per pair.
#include "emc_common.cuh"
#include "emc_internal.h"
#include "row_pairs.cuh"

namespace emc {

namespace {

// Every non-zero element of the two planes of P into the rows' lists. Bound by
// the one read (217 MB: 38 us, 5.7 TB/s). A warp
// reads 256 frames of a row (16 bytes per lane and plane), a CTA 128 rows x 256
// frames; row tiles run fastest, so that the CTAs of a tile already found to be
// over leave at once, and a block with more than 512 pairs is given up. Padding frames
// (from n_data on) carry no counts: what a caller's P holds there adds nothing, to den neither.
template <bool F16>
__global__ void __launch_bounds__(256)
    pairs_from_planes_kernel(const uint16_t* __restrict__ P, int64_t plane, int64_t ld_data,
                             int64_t n_data, unsigned nmt, RowPairs rp) {
  const int64_t mt = blockIdx.x % nmt;
  if (__syncthreads_or(*reinterpret_cast<volatile uint8_t*>(rp.over + mt))) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)(blockIdx.x / nmt) * 256, k0 = c0 + 8 * lane;
  const uint16_t* base = P + (mt * 128 + warp) * ld_data + k0;
  const int used = (int)max((int64_t)0, min((int64_t)8, n_data - k0));
  const unsigned take = (1u << used) - 1u;  // the lane's frames that are no padding
  __shared__ BlockPairs<512> bp;
  block_pairs_clear(bp);
#pragma unroll 1
  for (int b = 0; b < 16; b += 4) {
    if (*reinterpret_cast<volatile int*>(&bp.n) > 512) break;
    uint4 h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {  // rows warp + 8 (b + u)
      const uint16_t* p = base + (int64_t)(8 * (b + u)) * ld_data;
      h[u] = __ldcs(reinterpret_cast<const uint4*>(p));
      l[u] = __ldcs(reinterpret_cast<const uint4*>(p + plane));
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const uint32_t hv[4] = {h[u].x, h[u].y, h[u].z, h[u].w};
      const uint32_t lv[4] = {l[u].x, l[u].y, l[u].z, l[u].w};
      // (a negative zero is listed with weight 0)
      int n = 0;
#pragma unroll
      for (int i = 0; i < 8; i++)
        n += (take >> i & 1u) != 0u && ((hv[i >> 1] | lv[i >> 1]) >> (16 * (i & 1)) & 0xffffu) != 0u;
      if (n == 0) continue;
      const int jj = warp + 8 * (b + u);
      int place, at = block_pairs_take(bp, jj, n, &place);
      if (at < 0) continue;
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const uint16_t hb = (uint16_t)(hv[i >> 1] >> (16 * (i & 1)));
        const uint16_t lb = (uint16_t)(lv[i >> 1] >> (16 * (i & 1)));
        if ((hb | lb) == 0 || !(take >> i & 1u)) continue;
        const float w = F16 ? (fp16_val(hb) + fp16_val(lb)) * (1.0f / kP16Scale)
                            : bf16_val(hb) + bf16_val(lb);
        block_pairs_put(bp, at++, jj, place++, 8 * lane + i, w, w);
      }
    }
  }
  block_pairs_flush(bp, rp, mt * 128, c0);
}

// A CTA per row tile: its counters cleared, and a look at eight of its rows in 256 frames. Where
// an eighth of those is not zero, the posterior is flat and the tile over, so that the search
// need not find it out block by block (64^3, 10860 x 4999 at 0.1 photons a pixel: 490 us with the search,
// 446 so, 423 contracted straight away; the clearing takes a launch in any case).
__global__ void __launch_bounds__(256)
    pairs_begin_kernel(const uint16_t* __restrict__ P, int64_t plane, int64_t ld_data,
                       RowPairs rp) {
  const int64_t mt = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t k0 = ld_data / 512 * 256 + 8 * lane;
  const uint16_t* p = P + (mt * 128 + 16 * warp) * ld_data + k0;
  const uint4 h = *reinterpret_cast<const uint4*>(p);
  const uint4 l = *reinterpret_cast<const uint4*>(p + plane);
  if (threadIdx.x < 128) rp.cnt[mt * 128 + threadIdx.x] = 0;
  const uint32_t v[4] = {h.x | l.x, h.y | l.y, h.z | l.z, h.w | l.w};
  int n = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) n += (v[i >> 1] >> (16 * (i & 1)) & 0xffffu) != 0u;
  __shared__ int sum[8];
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0) sum[warp] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) n += sum[w];
    rp.tile_n[mt] = 0;
    rp.over[mt] = n > 256 ? 1 : 0;
  }
}

// Row tiles that are over: their list, and their tiles of the update's output (codes
// mt * n_ntiles + nt).
__global__ void __launch_bounds__(1024)
    over_lists_kernel(const uint8_t* __restrict__ over, int nt, int n_ntiles,
                      int32_t* __restrict__ tiles, int32_t* __restrict__ codes,
                      int32_t* __restrict__ counts) {
  __shared__ int wsum[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int n = 0;
  for (int b = 0; b < nt; b += 1024) {
    const int t = b + threadIdx.x;
    const bool on = t < nt && over[t] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (lane == 0) wsum[wid] = __popc(m);
    __syncthreads();
    int at = n;
    for (int w = 0; w < 32; w++) {
      if (w < wid) at += wsum[w];
      n += wsum[w];
    }
    if (on) tiles[at + __popc(m & ((1u << lane) - 1u))] = t;
    __syncthreads();
  }
  __syncthreads();
  for (int c = threadIdx.x; c < n * n_ntiles; c += 1024) {
    // raster groups of 8 row tiles, as the update walks all tiles
    const int g = c / (8 * n_ntiles), rem = c % (8 * n_ntiles), in = min(8, n - 8 * g);
    codes[c] = tiles[8 * g + rem % in] * n_ntiles + rem / in;
  }
  if (threadIdx.x == 0) {
    counts[0] = n;
    counts[1] = n * n_ntiles;
  }
}

// every row tile of a list of (row tile, frame tile) codes is over
__global__ void mark_over_kernel(const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                                 int nnt, uint8_t* __restrict__ over) {
  const int n = *count;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
    over[list[t] / nnt] = 1;
}

// Num and den of the rows of tiles that are not over: a CTA per row, 8 pixels a
// thread, four frames in flight. Bound by writing Num (233 MB at the 64^3 workload in 83 us).
template <bool KF16>
__global__ void __launch_bounds__(128)
    update_pairs_kernel(RowPairs rp, const uint16_t* __restrict__ Kb, int64_t ld_pix, bool empty,
                        float* __restrict__ Num, float* __restrict__ den) {
  const int64_t row = blockIdx.x;
  if (rp.over[row >> 7]) return;
  __shared__ int raw[kRowPairs], sk[kRowPairs];
  __shared__ float sw[kRowPairs], sp[kRowPairs];
  const int n = rp.cnt[row];  // <= kRowPairs
  if (n == 0 && !empty) {
    if (den && threadIdx.x == 0) den[row] = 0.f;
    return;
  }
  if (n > 0) {  // the pairs in frame order
    const int64_t o = row * kRowPairs + threadIdx.x;
    const int k = threadIdx.x < n ? rp.k[o] : 0;
    if (threadIdx.x < n) raw[threadIdx.x] = k;
    __syncthreads();
    if (threadIdx.x < n) {
      int rank = 0;
      for (int i = 0; i < n; i++) rank += raw[i] < k;
      sk[rank] = k;
      sw[rank] = rp.w[o];
      sp[rank] = rp.p[o];
    }
    __syncthreads();
  }
  float d = 0.f;
  for (int i = 0; i < n; i++) d += sp[i];
  if (den && threadIdx.x == 0) den[row] = d;
  if (d == 0.f && !empty) return;
  float* out = Num + row * ld_pix;
  for (int64_t g = threadIdx.x; g < ld_pix / 8; g += 128) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = 0; i < n; i += 4) {
      uint4 q[4];
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (i + u < n)
          q[u] = reinterpret_cast<const uint4*>(Kb + (int64_t)sk[i + u] * ld_pix)[g];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if (i + u >= n) break;
        const uint32_t qv[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
        const float w = sw[i + u];
#pragma unroll
        for (int c = 0; c < 8; c++) {
          const uint16_t x = (uint16_t)(qv[c >> 1] >> (16 * (c & 1)));
          acc[c] = fmaf(w, KF16 ? fp16_val(x) : bf16_val(x), acc[c]);
        }
      }
    }
    float4* o = reinterpret_cast<float4*>(out + 8 * g);
    o[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    o[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
}

}  // namespace

cudaError_t launch_pairs_reset(const RowPairs& rp, int64_t rows, cudaStream_t s) {
  // cnt, tile_n and over lie one behind the other
  return cudaMemsetAsync(rp.cnt, 0, sizeof(int32_t) * rows + 5 * (rows / 128), s);
}

cudaError_t launch_pairs_begin(const uint16_t* P, int64_t plane, int64_t rows, int64_t ld_data,
                               const RowPairs& rp, cudaStream_t s) {
  pairs_begin_kernel<<<(unsigned)(rows / 128), 256, 0, s>>>(P, plane, ld_data, rp);
  return cudaGetLastError();
}

cudaError_t launch_pairs_from_planes(const uint16_t* P, int64_t plane, int64_t rows,
                                     int64_t ld_data, int64_t n_data, int f16, const RowPairs& rp,
                                     cudaStream_t s) {
  const unsigned nmt = (unsigned)(rows / 128);
  const int64_t grd = (int64_t)nmt * (ld_data / 256);
  if (grd > INT32_MAX) return cudaErrorInvalidValue;
  if (f16)
    pairs_from_planes_kernel<true><<<(unsigned)grd, 256, 0, s>>>(P, plane, ld_data, n_data, nmt, rp);
  else
    pairs_from_planes_kernel<false><<<(unsigned)grd, 256, 0, s>>>(P, plane, ld_data, n_data, nmt, rp);
  return cudaGetLastError();
}

cudaError_t launch_mark_over(const int32_t* list, const int32_t* count, int64_t nnt,
                             const RowPairs& rp, cudaStream_t s) {
  mark_over_kernel<<<64, 256, 0, s>>>(list, count, (int)nnt, rp.over);
  return cudaGetLastError();
}

cudaError_t launch_over_lists(const RowPairs& rp, int64_t rows, int n_ntiles, int32_t* tiles,
                              int32_t* codes, int32_t* counts, cudaStream_t s) {
  const int nt = (int)(rows / 128);
  over_lists_kernel<<<1, 1024, 0, s>>>(rp.over, nt, n_ntiles, tiles, codes, counts);
  return cudaGetLastError();
}

cudaError_t launch_update_pairs(const RowPairs& rp, int64_t rows, const uint16_t* Kb, int kf16,
                                int64_t ld_pix, bool empty, float* Num, float* den,
                                cudaStream_t s) {
  if (kf16)
    update_pairs_kernel<true><<<(unsigned)rows, 128, 0, s>>>(rp, Kb, ld_pix, empty, Num, den);
  else
    update_pairs_kernel<false><<<(unsigned)rows, 128, 0, s>>>(rp, Kb, ld_pix, empty, Num, den);
  return cudaGetLastError();
}

}  // namespace emc
