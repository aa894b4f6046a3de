// Digit-sliced batched products of float-float contexts: 6 digits per operand (dig.cuh).
#include "dig.cuh"

namespace tdse {

const void *dig_fn6(int cg, int bn)
{
    if (cg == 1 && bn == 32) return (const void *)dig_kernel<6, 32, 1>;
    if (cg == 1 && bn == 64) return (const void *)dig_kernel<6, 64, 1>;
    if (cg == 2 && bn == 32) return (const void *)dig_kernel<6, 32, 2>;
    if (cg == 2 && bn == 64) return (const void *)dig_kernel<6, 64, 2>;
    if (cg == 2 && bn == 128) return (const void *)dig_kernel<6, 128, 2>;
    return nullptr;
}

}  // namespace tdse
