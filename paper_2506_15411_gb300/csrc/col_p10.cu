// col_p10.cu -- the two-step column kernels of axis lengths n = 10 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(10)
}  // namespace cbs
