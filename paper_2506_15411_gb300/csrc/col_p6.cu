// col_p6.cu -- the two-step column kernels of axis lengths n = 6 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(6)
}  // namespace cbs
