// misc.cu -- set-up, adjoint-source and gradient kernels.
//
//   set-up:    k^2 = k_vac^2 (eps_r + i sigma(r)),  k0^2 = (min Re k^2 + max Re k^2)/2,
//              epsilon = max |k^2 - k0^2| (FP64 block reductions),  V = k^2 - k0^2 - i epsilon
//              (splitting of the scalar CBS, ref. [25] of arXiv 2506.15411)
//   adjoint:   point source conj(E(r0)) at r0 for the figure of merit |E(r0)|^2 (Fig. 2 caption)
//   gradient:  dL/d eps_r = 2 k_vac^2 Re[E_adj . E]  (one pass over both fields)
// All k^2 quantities are in units of 1/pitch^2 (kv2 = (k_vac pitch)^2).
#include <cfloat>
#include <cstdint>
#include "absorber.h"
#include "cbs_internal.h"
#include "tma.cuh"

namespace cbs {

namespace {

template <class T, class Op>
__device__ __forceinline__ T block_reduce(T v, Op op, T* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = op(v, __shfl_down_sync(0xffffffffu, v, off));
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < nw; ++w) v = op(v, sh[w]);
  __syncthreads();
  return v;   // valid in thread 0
}

// The block whose arrival is the last of the grid (all of its threads see the answer); the
// others' partial results are visible to it.  `count` returns to 0 for the next launch.
__device__ __forceinline__ bool last_block(unsigned* count) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(count, 1u) == gridDim.x - 1;
    if (last) *count = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last != 0;
}

// Extremes of eps and, in the last block, the splitting's k0^2 = kv2 (min + max) / 2.
__global__ void k_eps_minmax(const float* __restrict__ eps, size_t N, float* pmin, float* pmax, int* pbad,
                             double kv2, Splitting* sp) {
  __shared__ float sh[32];
  __shared__ int shi[32];
  float lo = FLT_MAX, hi = -FLT_MAX;
  int bad = 0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  auto take = [&](float e) {
    if (!isfinite(e)) bad = 1;
    lo = fminf(lo, e);
    hi = fmaxf(hi, e);
  };
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (; i + 7 * stride < N; i += 8 * stride) {   // eight loads in flight per thread
    float e[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) e[k] = eps[i + k * stride];
#pragma unroll
    for (int k = 0; k < 8; ++k) take(e[k]);
  }
  for (; i < N; i += stride) take(eps[i]);
  auto fold = [&] {
    lo = block_reduce(lo, [](float p, float q) { return fminf(p, q); }, sh);
    hi = block_reduce(hi, [](float p, float q) { return fmaxf(p, q); }, sh);
    bad = block_reduce(bad, [](int p, int q) { return p | q; }, shi);
  };
  fold();
  if (threadIdx.x == 0) {
    pmin[blockIdx.x] = lo;
    pmax[blockIdx.x] = hi;
    pbad[blockIdx.x] = bad;
  }
  if (!last_block(&sp->count)) return;
  lo = FLT_MAX;
  hi = -FLT_MAX;
  bad = 0;
  for (int k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
    lo = fminf(lo, __ldcg(&pmin[k]));
    hi = fmaxf(hi, __ldcg(&pmax[k]));
    bad |= __ldcg(&pbad[k]);
  }
  fold();
  if (threadIdx.x == 0) {
    sp->bad = bad;
    sp->k0sq = 0.5 * kv2 * ((double)lo + (double)hi);
  }
}

// The FP64 parts of the set-up kernels, as calls: inlined, the compiler computes them ahead of the
// branches that avoid them.
__device__ __noinline__ float real_v(float e, double kv2, double k0sq) { return (float)(kv2 * (double)e - k0sq); }
__device__ __noinline__ float imag_v(double s, double sy, double sz, int corner_max, double kv2, double eshift) {
  return (float)(kv2 * layer_combine(s, sy, sz, corner_max) - eshift);
}
__device__ __noinline__ double dev2(float e, double s, double sy, double sz, int corner_max, double kv2, double k0sq) {
  const double re = kv2 * (double)e - k0sq;
  const double im = kv2 * layer_combine(s, sy, sz, corner_max);
  return re * re + im * im;
}

constexpr int kRowChunk = 4;   // 32-voxel pieces of a row whose loads are issued together

// epsilon = max |k^2 - k0^2| in FP64, a warp per row.  FP64 is dear here (two lanes a cycle, even
// a comparison), so a voxel between the x layers (xlo <= x < xhi, where the x profile is 0) is
// taken in FP64 only if an upper bound in FP32 (the real part's error is far below 2^-20 of its
// terms, the imaginary part is the row's) exceeds the lane's maximum so far, and if it does not
// repeat the lane's last such voxel: the same result.  384 x 384 x 256 of two materials: 0.83 -> 0.19
// ms.  The whole of cbs_set_permittivity there 1.59 -> 0.41 ms, at 640 x 640 x 336 5.5 -> 0.9 ms, and
// at 64^3, where the host waited three times, 0.085 -> 0.058 ms.
__global__ void k_k2_maxdev(const float* __restrict__ eps, int nx, int ny, int nz, int xlo, int xhi,
                            const double* __restrict__ sx, const double* __restrict__ sy,
                            const double* __restrict__ sz, int corner_max, double kv2, double* part, Splitting* sp) {
  __shared__ double sh[32];
  const double k0sq = sp->k0sq;
  const float tau = 1.0f / (1 << 20);
  const float kv2f = (float)kv2, k0f = (float)k0sq;
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  double m = 0.0;
  float mf = -1.f;   // at most m; -1 while m is so small that a bound's squares may underflow
  float eh = 0.f;   // permittivity and row part of the lane's last voxel between the layers
  double imh = -1.0;
  for (int row = blockIdx.x * warps + (threadIdx.x >> 5); row < ny * nz; row += gridDim.x * warps) {
    const int z = row / ny;
    const double syr = sy[row - z * ny], szr = sz[z];
    const double im0 = kv2 * layer_combine(0.0, syr, szr, corner_max);
    const float imf = (float)im0, im2 = imf * imf * (1.f + 4.f * tau);
    bool below = im0 <= imh;   // a voxel of permittivity eh in this row adds nothing
    const float* const e0 = eps + (size_t)row * nx;
    for (int x0 = 0; x0 < nx; x0 += 32 * kRowChunk) {
      float e[kRowChunk];
#pragma unroll
      for (int k = 0; k < kRowChunk; ++k) e[k] = e0[min(x0 + 32 * k + lane, nx - 1)];   // (past the end: the last)
#pragma unroll
      for (int k = 0; k < kRowChunk; ++k) {
        const int x = min(x0 + 32 * k + lane, nx - 1);
        const bool inner = x >= xlo && x < xhi;
        const float t = kv2f * e[k];
        const float d = fabsf(t - k0f) + tau * (fabsf(t) + fabsf(k0f));
        const bool skip = inner && (fmaf(d, d, im2) * (1.f + tau) <= mf || (below && e[k] == eh));
        if (__any_sync(0xffffffffu, !skip)) {
          // squared: one square root per block, not per voxel
          m = fmax(m, dev2(e[k], inner ? 0.0 : sx[x], syr, szr, corner_max, kv2, k0sq));
          mf = __double2float_rd(m);
          if (mf < 1e-30f) mf = -1.f;
          if (inner) {
            eh = e[k];
            imh = im0;
            below = true;
          }
        }
      }
    }
  }
  m = block_reduce(m, [](double p, double q) { return fmax(p, q); }, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = sqrt(m);   // sqrt is monotonic: the same maximum
  if (!last_block(&sp->count)) return;
  m = 0.0;
  for (int k = threadIdx.x; k < gridDim.x; k += blockDim.x) m = fmax(m, __ldcg(&part[k]));
  m = block_reduce(m, [](double p, double q) { return fmax(p, q); }, sh);
  if (threadIdx.x == 0) sp->eps = m;
}

// V in the y-blocked layout of the iteration (row padding stays zero), a warp per row.  The
// imaginary part is the row's wherever the x profile is 0, and the real part is recomputed only
// where the permittivity changes from one 32-voxel piece to the next: FP64 for a small part of
// the voxels of a lens, the same values (384 x 384 x 256: 0.14 ms, 0.33 where every voxel differs).
// Without a valid splitting V is left as it was.
__global__ void k_build_v(const float* __restrict__ eps, int nx, int ny, int nz, int nxp, int yblk, int xlo, int xhi,
                          const double* __restrict__ sx, const double* __restrict__ sy,
                          const double* __restrict__ sz, int corner_max, double kv2, const Splitting* sp,
                          float2* __restrict__ V) {
  const double k0sq = sp->k0sq, eshift = sp->eps;
  if (sp->bad || !(eshift > 0.0) || !isfinite(eshift)) return;
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  float last = 0.f, re = real_v(last, kv2, k0sq);
  for (int row = blockIdx.x * warps + (threadIdx.x >> 5); row < ny * nz; row += gridDim.x * warps) {
    const int z = row / ny, y = row - z * ny;
    const double syr = sy[y], szr = sz[z];
    const float im0 = imag_v(0.0, syr, szr, corner_max, kv2, eshift);
    const float* const e0 = eps + (size_t)row * nx;
    float2* const v0 = V + wrow(y, z, nz, yblk) * nxp;
    for (int x0 = 0; x0 < nx; x0 += 32 * kRowChunk) {
      float e[kRowChunk];
#pragma unroll
      for (int k = 0; k < kRowChunk; ++k) e[k] = e0[min(x0 + 32 * k + lane, nx - 1)];
#pragma unroll
      for (int k = 0; k < kRowChunk; ++k) {
        const int x = x0 + 32 * k + lane;
        if (__any_sync(0xffffffffu, e[k] != last)) {
          last = e[k];
          re = real_v(e[k], kv2, k0sq);
        }
        const bool layer = x < nx && (x < xlo || x >= xhi);
        float im = im0;
        if (__any_sync(0xffffffffu, layer))
          if (layer) im = imag_v(sx[x], syr, szr, corner_max, kv2, eshift);
        if (x < nx) v0[x] = make_float2(re, im);
      }
    }
  }
}

// A field between the dense and the plan's layout, a warp per row; VEC: two values per access
// (even nx and a 16-byte aligned dense field).  48 bytes a voxel at the copy rate (384 x 384 x 256:
// 0.27 ms, 6.6 TB/s; one element a thread with its 64-bit divisions took 2.4 ms at 640 x 640 x 336).
template <bool VEC>
__global__ void k_field_layout(const float2* __restrict__ src, float2* __restrict__ dst, int to_dense, int nx, int ny,
                               int nz, int nxp, int yblk) {
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5, rows = ny * nz;
  for (int r = blockIdx.x * warps + (threadIdx.x >> 5); r < 3 * rows; r += gridDim.x * warps) {
    const int c = r / rows, row = r - c * rows, z = row / ny, y = row - z * ny;
    const size_t d = (size_t)r * nx, b = ((size_t)c * rows + wrow(y, z, nz, yblk)) * nxp;
    const float2* const s = src + (to_dense ? b : d);
    float2* const t = dst + (to_dense ? d : b);
    if constexpr (VEC) {
      const float4* const s4 = reinterpret_cast<const float4*>(s);
      float4* const t4 = reinterpret_cast<float4*>(t);
#pragma unroll 4
      for (int x = lane; x < nx / 2; x += 32) t4[x] = s4[x];
    } else {
#pragma unroll 4
      for (int x = lane; x < nx; x += 32) t[x] = s[x];
    }
  }
}

__global__ void k_adjoint_amp(const float2* __restrict__ E, size_t N, size_t idx, float scale,
                              float2* amp) {
  if (threadIdx.x < 3) {
    const float2 e = E[threadIdx.x * N + idx];
    amp[threadIdx.x] = make_float2(e.x * scale, -e.y * scale);
  }
}

// Two voxels per thread through 16-byte loads when N is even; scalar tail otherwise.
__global__ void k_gradient(const float2* __restrict__ E, const float2* __restrict__ Ea, size_t N,
                           float coef, float* __restrict__ g, int vec) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  if (vec) {
    const size_t M = N / 2;
    const float4* E4 = reinterpret_cast<const float4*>(E);
    const float4* A4 = reinterpret_cast<const float4*>(Ea);
    float2* g2 = reinterpret_cast<float2*>(g);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M; i += stride) {
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float4 e = __ldg(&E4[c * M + i]);
        const float4 a = __ldg(&A4[c * M + i]);
        s0 = fmaf(a.x, e.x, fmaf(-a.y, e.y, s0));
        s1 = fmaf(a.z, e.z, fmaf(-a.w, e.w, s1));
      }
      g2[i] = make_float2(coef * s0, coef * s1);
    }
  } else {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += stride) {
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 e = __ldg(&E[c * N + i]);
        const float2 a = __ldg(&Ea[c * N + i]);
        s = fmaf(a.x, e.x, fmaf(-a.y, e.y, s));
      }
      g[i] = coef * s;
    }
  }
}

__global__ void k_objective(const float2* __restrict__ E, size_t N, size_t idx, double* out) {
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int c = 0; c < 3; ++c) {
      const float2 e = E[c * N + idx];
      s += (double)e.x * e.x + (double)e.y * e.y;
    }
    *out = s;
  }
}

}  // namespace

cudaError_t launch_splitting(const float* eps, int nx, int ny, int nz, int xlo, int xhi, const double* sx, const double* sy,
                             const double* sz, int corner_max, double kv2, float* pmin, float* pmax, int* pbad,
                             double* part, int blocks, Splitting* sp, cudaStream_t s) {
  k_eps_minmax<<<blocks, 256, 0, s>>>(eps, (size_t)nx * ny * nz, pmin, pmax, pbad, kv2, sp);
  k_k2_maxdev<<<blocks, 256, 0, s>>>(eps, nx, ny, nz, xlo, xhi, sx, sy, sz, corner_max, kv2, part, sp);
  return cudaGetLastError();
}

cudaError_t launch_build_v(const float* eps, int nx, int ny, int nz, int nxp, int yblk, int xlo, int xhi, const double* sx,
                           const double* sy, const double* sz, int corner_max, double kv2, const Splitting* sp,
                           float2* V, cudaStream_t s) {
  k_build_v<<<152 * 8, 256, 0, s>>>(eps, nx, ny, nz, nxp, yblk, xlo, xhi, sx, sy, sz, corner_max, kv2, sp, V);
  return cudaGetLastError();
}

cudaError_t launch_field_layout(const float2* src, float2* dst, bool to_dense, int nx, int ny, int nz, int nxp,
                                int yblk, cudaStream_t s) {
  const float2* const dense = to_dense ? dst : src;
  if (nx % 2 == 0 && reinterpret_cast<uintptr_t>(dense) % 16 == 0)
    k_field_layout<true><<<152 * 8, 256, 0, s>>>(src, dst, to_dense ? 1 : 0, nx, ny, nz, nxp, yblk);
  else
    k_field_layout<false><<<152 * 8, 256, 0, s>>>(src, dst, to_dense ? 1 : 0, nx, ny, nz, nxp, yblk);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_amp(const float2* E, size_t N, int nx, int ny, int x, int y, int z,
                               float scale, float2* amp, cudaStream_t s) {
  const size_t idx = ((size_t)z * ny + y) * nx + x;
  k_adjoint_amp<<<1, 32, 0, s>>>(E, N, idx, scale, amp);
  return cudaGetLastError();
}

cudaError_t launch_gradient(const float2* E, const float2* Ea, size_t N, float coef, float* g,
                            cudaStream_t s) {
  const int vec = (N % 2 == 0) && ((reinterpret_cast<uintptr_t>(E) | reinterpret_cast<uintptr_t>(Ea)) % 16 == 0) &&
                  (reinterpret_cast<uintptr_t>(g) % 8 == 0);
  k_gradient<<<152 * 8, 256, 0, s>>>(E, Ea, N, coef, g, vec);
  return cudaGetLastError();
}

cudaError_t launch_objective(const float2* E, size_t N, int nx, int ny, int x, int y, int z,
                             double* out, cudaStream_t s) {
  const size_t idx = ((size_t)z * ny + y) * nx + x;
  k_objective<<<1, 32, 0, s>>>(E, N, idx, out);
  return cudaGetLastError();
}

// Self-test of the bounded waits: an mbarrier that nothing arrives at, waited on with the
// tile kernels' bounded wait (`limit` polls).  The wait must give up, the kernel record the
// timeout in *err and return -- the error path every tile kernel takes instead of hanging.
__global__ void k_wait_selftest(int* err, long long limit) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(&bar, 0, limit)) atomicExch(err, kErrTmaTimeout);
}

cudaError_t launch_wait_selftest(int* err, long long limit, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(err, limit);
  return cudaGetLastError();
}

}  // namespace cbs
