// xrow_p8.cu -- the warp-per-row x kernels of axis lengths n = 8 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(8)
}  // namespace cbs
