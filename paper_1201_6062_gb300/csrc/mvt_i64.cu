// Ring-fed block mat-vec kernels with FP64-accurate products in integer
// arithmetic (PolI64), one product per launch (every thread layout and ring
// depth).
#include "mvt.cuh"

namespace tdse {
const void *mvt_fn_i64_product(int idx, int rs) { return mvt_fn<PolI64, false>(idx, rs); }
}  // namespace tdse
