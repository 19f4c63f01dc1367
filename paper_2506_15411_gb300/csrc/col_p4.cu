// col_p4.cu -- the two-step column kernels of axis lengths n = 4 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(4)
}  // namespace cbs
