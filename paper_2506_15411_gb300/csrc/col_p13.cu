// col_p13.cu -- the two-step column kernels of axis lengths n = 13 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(13)
}  // namespace cbs
