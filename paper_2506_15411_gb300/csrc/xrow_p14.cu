// xrow_p14.cu -- the warp-per-row x kernels of axis lengths n = 14 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(14)
}  // namespace cbs
