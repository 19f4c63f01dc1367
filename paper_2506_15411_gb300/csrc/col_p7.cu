// col_p7.cu -- the two-step column kernels of axis lengths n = 7 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(7)
}  // namespace cbs
