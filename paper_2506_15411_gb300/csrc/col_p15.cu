// col_p15.cu -- the two-step column kernels of axis lengths n = 15 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(15)
}  // namespace cbs
