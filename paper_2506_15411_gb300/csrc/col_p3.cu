// col_p3.cu -- the two-step column kernels of axis lengths n = 3 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(3)
}  // namespace cbs
