// Block-wide scan shared by the kernels that compact or lay out lists.
#pragma once
#include "twkv_dev.h"

namespace twkv {

// Exclusive scan of one value per thread over a CTA of 1024 threads; returns the thread's offset, *total = sum (valid for
// all threads).  s_warp: 32 ints of shared memory.
__device__ __forceinline__ int block_scan_excl(int x, int* s_warp, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  __syncthreads();                                         // s_warp may still be read from the previous call
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = s_warp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  *total = s_warp[31];
  return (warp ? s_warp[warp - 1] : 0) + incl - x;
}

}  // namespace twkv
