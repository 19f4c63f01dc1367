// xrow_p3.cu -- the warp-per-row x kernels of axis lengths n = 3 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(3)
}  // namespace cbs
