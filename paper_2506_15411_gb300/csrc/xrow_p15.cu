// xrow_p15.cu -- the warp-per-row x kernels of axis lengths n = 15 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(15)
}  // namespace cbs
