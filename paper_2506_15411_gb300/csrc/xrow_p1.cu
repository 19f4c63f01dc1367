// xrow_p1.cu -- the warp-per-row x kernels of axis lengths n = 1 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(1)
}  // namespace cbs
