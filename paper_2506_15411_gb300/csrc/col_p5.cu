// col_p5.cu -- the two-step column kernels of axis lengths n = 5 mod 16 (colpass.cuh).
#include "colpass.cuh"

namespace cbs {
CBS_COL_PART(5)
}  // namespace cbs
