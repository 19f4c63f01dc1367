// xrow_p9.cu -- the warp-per-row x kernels of axis lengths n = 9 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(9)
}  // namespace cbs
