// col_p8.cu -- the two-step column kernels of axis lengths n = 8 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(8)
}  // namespace cbs
