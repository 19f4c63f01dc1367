// xrow_p12.cu -- the warp-per-row x kernels of axis lengths n = 12 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(12)
}  // namespace cbs
