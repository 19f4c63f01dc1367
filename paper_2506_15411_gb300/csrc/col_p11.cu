// col_p11.cu -- the two-step column kernels of axis lengths n = 11 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(11)
}  // namespace cbs
