// col_p9.cu -- the two-step column kernels of axis lengths n = 9 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(9)
}  // namespace cbs
