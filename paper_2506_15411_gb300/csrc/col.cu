// col.cu -- host side of the two-step column passes (colpass.cuh).
#include "colpass.cuh"

namespace cbs {

#define CBS_COL_PARTS(F) F(0) F(1) F(2) F(3) F(4) F(5) F(6) F(7) F(8) F(9) F(10) F(11) F(12) F(13) F(14) F(15)
#define CBS_COL_DECL(i) ColKernels col_kernels_##i(int n);
CBS_COL_PARTS(CBS_COL_DECL)

namespace {

ColKernels col_kernels(int n) {
#define CBS_COL_ENTRY(i) col_kernels_##i,
  static ColKernels (*const part[kColParts])(int) = {CBS_COL_PARTS(CBS_COL_ENTRY)};
  return part[n % kColParts](n);
}

size_t col_smem(const ColShape& sh, int ncomp, int twb, int pqb) {
  return (size_t)sh.sets * ncomp * sh.box * sh.nbox * sh.tx * sizeof(float2) + twb + pqb + 8 * (2 * sh.sets + 1) + 48;
}

}  // namespace

cudaError_t launch_col(const CUtensorMap& tm, const IterArgs& a, int kind, cudaStream_t s) {
  if (kind == colk::kZ)
    return launch_overlapped(col_kernels(a.nz).z, a.grid_z * a.nmem, a.zc.threads,
                             col_smem(a.zc, 3, a.twbz, a.pqbz), a.N <= kOverlapVoxels, s, tm, a);
  const ColKernels k = col_kernels(a.ny);
  return launch_overlapped(kind == colk::kYFwd ? k.yfwd : k.yinv, a.grid_y * a.nmem, a.yc.threads,
                           col_smem(a.yc, 1, a.twby, 0), a.N <= kOverlapVoxels, s, tm, a);
}

cudaError_t col_set_smem_limit(int n, bool z, int bytes) {
  const ColKernels k = col_kernels(n);
  if (z) return cudaFuncSetAttribute((const void*)k.z, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaError_t e = cudaFuncSetAttribute((const void*)k.yfwd, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)k.yinv, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

}  // namespace cbs
