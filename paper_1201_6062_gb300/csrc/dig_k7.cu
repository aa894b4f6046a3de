// Digit-sliced batched products of FP32 and float-float contexts: 7 digits per operand (dig.cuh).
#include "dig.cuh"

namespace tdse {

const void *dig_fn7(int cg, int bn)
{
    if (cg == 1 && bn == 32) return (const void *)dig_kernel<7, 32, 1>;
    if (cg == 1 && bn == 64) return (const void *)dig_kernel<7, 64, 1>;
    if (cg == 2 && bn == 32) return (const void *)dig_kernel<7, 32, 2>;
    if (cg == 2 && bn == 64) return (const void *)dig_kernel<7, 64, 2>;
    if (cg == 2 && bn == 128) return (const void *)dig_kernel<7, 128, 2>;
    return nullptr;
}

}  // namespace tdse
