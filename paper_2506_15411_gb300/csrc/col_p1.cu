// col_p1.cu -- the two-step column kernels of axis lengths n = 1 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(1)
}  // namespace cbs
