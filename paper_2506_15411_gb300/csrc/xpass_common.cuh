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

// Block reduction of the per-thread residual in FP64, then a last-block-done pass that sums
// the per-block partials of the request in seat `seat` (blocks b = 0 .. G-1 of its grid) in a
// fixed order into its hist[slot] (deterministic).
__device__ __forceinline__ void residual_finish(float acc, const IterArgs& a, int seat, int b, int G, double* wsum,
                                                int* lastflag) {
  double* const part = a.partials + (size_t)seat * a.grid_x;
  unsigned* const counter = a.counter + seat;
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
    part[b] = bs;
    __threadfence();
    const unsigned prev = atomicAdd(counter, 1u);
    *lastflag = (prev == (unsigned)G - 1);
  }
  __syncthreads();
  if (!*lastflag) return;
  __threadfence();
  double s = 0.0;
  for (int i = threadIdx.x; i < G; i += blockDim.x) s += __ldcg(&part[i]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  __syncthreads();
  if (lane == 0) wsum[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double bs = 0.0;
    for (int w = 0; w < nw; ++w) bs += wsum[w];
    a.hist[(size_t)seat * a.hist_cap + a.slot] = bs;
    *counter = 0u;
  }
}

}  // namespace cbs
