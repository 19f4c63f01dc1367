// xrow_p13.cu -- the warp-per-row x kernels of axis lengths n = 13 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(13)
}  // namespace cbs
