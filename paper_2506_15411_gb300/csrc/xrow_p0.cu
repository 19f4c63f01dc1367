// xrow_p0.cu -- the warp-per-row x kernels of axis lengths n = 0 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(0)
}  // namespace cbs
