// col_p14.cu -- the two-step column kernels of axis lengths n = 14 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(14)
}  // namespace cbs
