// row_pairs.cuh -- a block's non-zero pairs (128 rows x up to 256 frames) on their way to
// the rows' lists (RowPairs): collected in shared memory first, so that a block
// costs one global atomic per row in place of one per pair and a chain of them
// per thread. A block with more than CAP pairs shows a flat posterior: its row
// tile is marked over without listing them.
#pragma once
#include "emc_internal.h"

namespace emc {

template <int CAP>
struct BlockPairs {
  int n, row_n[128], row_at[128];
  int where[CAP];  // row << 24 | place among the row's << 12 | frame
  float w[CAP], p[CAP];
};

// by 256 threads; pairs may be added from here on
template <int CAP>
__device__ __forceinline__ void block_pairs_clear(BlockPairs<CAP>& bp) {
  if (threadIdx.x < 128) bp.row_n[threadIdx.x] = 0;
  if (threadIdx.x == 128) bp.n = 0;
  __syncthreads();
}

// the places of n pairs of row jj: the block's, or -1 where they are more than fit
template <int CAP>
__device__ __forceinline__ int block_pairs_take(BlockPairs<CAP>& bp, int jj, int n, int* place) {
  *place = atomicAdd(&bp.row_n[jj], n);
  const int at = atomicAdd(&bp.n, n);
  return at + n <= CAP ? at : -1;
}

template <int CAP>
__device__ __forceinline__ void block_pairs_put(BlockPairs<CAP>& bp, int at, int jj, int place,
                                                int frame, float w, float p) {
  bp.where[at] = jj << 24 | place << 12 | frame;
  bp.w[at] = w;
  bp.p[at] = p;
}

// into the lists of rows j0 .. of tile j0 / 128, frames from k0 on; by all 256 threads
template <int CAP>
__device__ __forceinline__ void block_pairs_flush(BlockPairs<CAP>& bp, const RowPairs& rp,
                                                  int64_t j0, int64_t k0) {
  const int tid = threadIdx.x;
  uint8_t* over = rp.over + (j0 >> 7);
  __syncthreads();
  const int total = bp.n;
  if (total == 0) return;
  if (total > CAP) {
    if (tid == 0) *over = 1;
    return;
  }
  if (tid == 128 && atomicAdd(rp.tile_n + (j0 >> 7), total) + total > kTilePairs) *over = 1;
  if (tid < 128 && bp.row_n[tid]) {
    const int at = atomicAdd(rp.cnt + j0 + tid, bp.row_n[tid]);
    if (at + bp.row_n[tid] > kRowPairs) *over = 1;
    bp.row_at[tid] = at;
  }
  __syncthreads();
  for (int i = tid; i < total; i += 256) {
    const int wh = bp.where[i], jj = wh >> 24;
    const int at = bp.row_at[jj] + (wh >> 12 & 4095);
    if (at < kRowPairs) {
      const int64_t o = (j0 + jj) * kRowPairs + at;
      rp.k[o] = (int32_t)(k0 + (wh & 4095));
      rp.w[o] = bp.w[i];
      rp.p[o] = bp.p[i];
    }
  }
}

}  // namespace emc
