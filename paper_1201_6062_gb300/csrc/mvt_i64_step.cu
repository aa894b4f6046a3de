// Ring-fed block mat-vec kernels with FP64-accurate products in integer
// arithmetic (PolI64), all stages of a propagation per launch (persistent
// stepping; every thread layout and ring depth).
#include "mvt.cuh"

namespace tdse {
const void *mvt_fn_i64_step(int idx, int rs, int groups)
{
    if (groups == 2) {
        if (idx == 0) return mvt_fn_rs<PolI64, 128, 1, true, 2>(rs);
        if (idx == 1) return mvt_fn_rs<PolI64, 128, 2, true, 2>(rs);
        return nullptr;
    }
    return mvt_fn<PolI64, true>(idx, rs);
}
}  // namespace tdse
