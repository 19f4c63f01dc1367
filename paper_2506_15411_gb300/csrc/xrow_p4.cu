// xrow_p4.cu -- the warp-per-row x kernels of axis lengths n = 4 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(4)
}  // namespace cbs
