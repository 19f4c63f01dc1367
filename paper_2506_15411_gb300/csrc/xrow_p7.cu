// xrow_p7.cu -- the warp-per-row x kernels of axis lengths n = 7 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(7)
}  // namespace cbs
