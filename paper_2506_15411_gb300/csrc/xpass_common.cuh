// xpass_common.cuh -- what the two forms of the x passes share: the (y, z) of a memory row and
// the residual reduction that ends the update pass.
#pragma once
#include "cbs_internal.h"
#include "fft_ip.cuh"

namespace cbs {

// (y, z) of memory row r of the y-blocked arrays: r = ((y / yblk) nz + z) yblk + y mod yblk
struct RowDecode {
  float inv_blk, inv_nz;
  int blk, nz;
  __device__ __forceinline__ void operator()(int r, int& y, int& z) const {
    const int t = ip_div(r, inv_blk), yi = r - t * blk;
    const int yb = ip_div(t, inv_nz);
    z = t - yb * nz;
    y = yb * blk + yi;
  }
};
__device__ __forceinline__ RowDecode row_decode(const IterArgs& a) {
  return RowDecode{1.0f / (float)a.yblk, 1.0f / (float)a.nz, a.yblk, a.nz};
}

// Where block b of a request's grid leaves its residual partial of the current iteration: the
// partials of kResidualSlots iterations are kept, and k_residuals sums each iteration's in a fixed
// order once per that many (or at the end of a block of iterations).  A last-block-done sum in the
// x pass itself would add two trips through memory to every iteration.
__device__ __forceinline__ double* residual_slot(const IterArgs& a, int seat, int b) {
  return a.partials + ((size_t)seat * kResidualSlots + a.slot % kResidualSlots) * a.grid_x + b;
}

// Block sum of the per-thread residual in FP64 (fixed order) into the block's slot.
__device__ __forceinline__ void residual_finish(float acc, const IterArgs& a, int seat, int b, double* wsum) {
  double d = (double)acc;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) d += __shfl_down_sync(0xffffffffu, d, off);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  if (lane == 0) wsum[wid] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double bs = 0.0;
    for (int w = 0; w < nw; ++w) bs += wsum[w];
    *residual_slot(a, seat, b) = bs;
  }
}

}  // namespace cbs
