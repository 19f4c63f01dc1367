// xrow.cu -- host side of the warp-per-row x passes (xrow.cuh).
#include "xrow.cuh"

namespace cbs {

#define CBS_ROW_PARTS(F) F(0) F(1) F(2) F(3) F(4) F(5) F(6) F(7) F(8) F(9) F(10) F(11) F(12) F(13) F(14) F(15)
#define CBS_ROW_DECL(i) RowKernel row_kernel_##i(int n);
CBS_ROW_PARTS(CBS_ROW_DECL)

namespace {

RowKernel row_kernel(int n) {
#define CBS_ROW_ENTRY(i) row_kernel_##i,
  static RowKernel (*const part[kRowParts])(int) = {CBS_ROW_PARTS(CBS_ROW_ENTRY)};
  return part[n % kRowParts](n);
}

}  // namespace

// S sets of rpb rows (W of three components at pitch ldw, E of three and V at pitch lde), the
// twiddles, 2 S + 1 mbarriers and the flags
size_t xrow_smem(const IterArgs& a) {
  const size_t sets = (size_t)a.xr.sets * a.xr.rpb * (3 * a.xr.ldw + 4 * a.xr.lde) * sizeof(float2) + a.twbx +
                      8 * (2 * a.xr.sets + 1) + 16;
  return std::max(sets, (size_t)xrow::kRowThreads * sizeof(float));   // (at the end: the threads' residuals)
}
int xrow_tiles(const IterArgs& a) { return (a.ny * a.nz + a.xr.rpb - 1) / a.xr.rpb; }

cudaError_t launch_xrow(const IterArgs& a, int mode, cudaStream_t s) {
  const int threads = 32 * (3 * a.xr.teams + 1);
  if (mode == 0)
    return launch_overlapped(row_kernel(a.nx), a.grid_x * a.nmem, threads, xrow_smem(a), a.N <= kOverlapVoxels, s, a, 0);
  row_kernel(a.nx)<<<a.grid_x * a.nmem, threads, xrow_smem(a), s>>>(a, mode);
  return cudaGetLastError();
}

cudaError_t xrow_set_smem_limit(int n, int bytes) {
  return cudaFuncSetAttribute((const void*)row_kernel(n), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace cbs
