// col_p2.cu -- the two-step column kernels of axis lengths n = 2 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(2)
}  // namespace cbs
