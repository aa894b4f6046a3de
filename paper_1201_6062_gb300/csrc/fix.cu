// Fixed-point copies of FP64 dipole blocks for the integer products (PolI64).
#include "kernels.h"

namespace tdse {

// One 32 x 32 tile per CTA, 32 x 8 threads.
__global__ void fix_maxima_kernel(const double *__restrict__ U, long long bstride, int ld, int n, int lmax, int *out)
{
    const int l = blockIdx.z, j = blockIdx.x * 32 + threadIdx.x;
    int cm = 0;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = blockIdx.y * 32 + r;
        int h = 0;
        if (i < n && j < n) h = __double2hiint(U[l * bstride + (long long)i * ld + j]) & 0x7fffffff;
        cm = max(cm, h);
        const int rm = __reduce_max_sync(0xffffffffu, h);
        if (threadIdx.x == 0 && i < n && rm > 0) atomicMax(out + (long long)l * n + i, rm);
    }
    if (j < n && cm > 0) atomicMax(out + (long long)(lmax + l) * n + j, cm);
}

cudaError_t launch_fix_maxima(const double *U, long long bstride, int ld, int n, int lmax, int *out, cudaStream_t s)
{
    const cudaError_t z = cudaMemsetAsync(out, 0, sizeof(int) * 2 * (size_t)lmax * n, s);
    if (z != cudaSuccess) return z;
    fix_maxima_kernel<<<dim3((n + 31) / 32, (n + 31) / 32, lmax), dim3(32, 8), 0, s>>>(U, bstride, ld, n, lmax, out);
    return cudaGetLastError();
}

// count elements of every block (the padding columns are zero and stay zero)
__global__ void __launch_bounds__(256)
fix_kernel(const double *__restrict__ U, long long bstride, long long count, const int *__restrict__ ue, int2 *out)
{
    const long long q = (long long)blockIdx.x * 256 + threadIdx.x;
    if (q >= count) return;
    const long long o = (long long)blockIdx.y * bstride + q;
    out[o] = PolI64::fix(U[o], ue[blockIdx.y]);
}

cudaError_t launch_fix(const double *U, long long bstride, long long count, int lmax, const int *ue, void *out, cudaStream_t s)
{
    fix_kernel<<<dim3((unsigned)((count + 255) / 256), lmax), 256, 0, s>>>(U, bstride, count, ue, reinterpret_cast<int2 *>(out));
    return cudaGetLastError();
}

}  // namespace tdse
