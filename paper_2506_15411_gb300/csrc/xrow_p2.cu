// xrow_p2.cu -- the warp-per-row x kernels of axis lengths n = 2 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(2)
}  // namespace cbs
