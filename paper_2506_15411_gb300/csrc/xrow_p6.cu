// xrow_p6.cu -- the warp-per-row x kernels of axis lengths n = 6 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(6)
}  // namespace cbs
