// col_p0.cu -- the two-step column kernels of axis lengths n = 0 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(0)
}  // namespace cbs
