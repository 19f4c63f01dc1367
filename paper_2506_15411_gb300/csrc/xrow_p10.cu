// xrow_p10.cu -- the warp-per-row x kernels of axis lengths n = 10 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(10)
}  // namespace cbs
