// Block-wide exclusive scan for 256-thread blocks (stable compactions).
#pragma once

#include "gs2d_common.cuh"

namespace gs2d {

// Exclusive prefix of one value per thread over a 256-thread block (int, or
// uint32_t for sums modulo 2^32); *total receives the block sum.  s_w: shared
// scratch of 8 values.  Every thread of the block must call it.
template <typename T>
__device__ __forceinline__ T block_exscan256(T v, T* s_w, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T w = lane < 8 ? s_w[lane] : T(0);
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
      const T y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    if (lane < 8) s_w[lane] = w;
  }
  __syncthreads();
  const T pre = (warp ? s_w[warp - 1] : T(0)) + x - v;
  *total = s_w[7];
  __syncthreads();
  return pre;
}

// A 256-thread block's exclusive prefix of per-block counts and their total,
// summed by the block itself (for at most kSelfSumBlocks blocks: their counts
// are 16 KB from L2, ~1 us, where a scan launch costs 4-5 us), or read after
// a scan launch put the prefixes in blk and the total in *scanned_total.
// s: 16 ints; every thread calls it.
constexpr int kSelfSumBlocks = 4096;
__device__ __forceinline__ void block_base(const int32_t* __restrict__ blk, int nb,
                                           const int32_t* __restrict__ scanned_total, int* s,
                                           int* base, int* total) {
  if (scanned_total) {
    *base = blk[blockIdx.x];
    *total = *scanned_total;
    return;
  }
  int before = 0, all = 0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += 256) {
    const int v = blk[b];
    all += v;
    if (b < (int)blockIdx.x) before += v;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  all = __reduce_add_sync(0xffffffffu, all);
  if ((threadIdx.x & 31) == 0) {
    s[threadIdx.x >> 5] = before;
    s[8 + (threadIdx.x >> 5)] = all;
  }
  __syncthreads();
  before = all = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    before += s[w];
    all += s[8 + w];
  }
  *base = before;
  *total = all;
}

}  // namespace gs2d
