// col_p12.cu -- the two-step column kernels of axis lengths n = 12 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(12)
}  // namespace cbs
