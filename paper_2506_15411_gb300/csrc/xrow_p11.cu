// xrow_p11.cu -- the warp-per-row x kernels of axis lengths n = 11 mod 16 (xrow.cuh).
#include "xrow.cuh"

namespace cbs {
CBS_ROW_PART(11)
}  // namespace cbs
