// Digit-sliced batched products of FP64 contexts: 11 digits per operand (dig.cuh).
#include "dig.cuh"

namespace tdse {

const void *dig_fn11(int cg, int bn)
{
    if (cg == 1 && bn == 32) return (const void *)dig_kernel<11, 32, 1>;
    if (cg == 1 && bn == 64) return (const void *)dig_kernel<11, 64, 1>;
    if (cg == 2 && bn == 32) return (const void *)dig_kernel<11, 32, 2>;
    if (cg == 2 && bn == 64) return (const void *)dig_kernel<11, 64, 2>;
    return nullptr;
}

}  // namespace tdse
