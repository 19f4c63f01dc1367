// xrow_p5.cu -- the warp-per-row x kernels of axis lengths n = 5 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(5)
}  // namespace cbs
