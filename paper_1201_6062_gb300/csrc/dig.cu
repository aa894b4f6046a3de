// Host side and digit conversions of the digit-sliced batched products (the
// GEMM is in dig.cuh).
#include "dig.cuh"

namespace tdse {

// Integers that hold S digits.
template <int S> using DigInt = typename std::conditional<(S > 7), __int128, long long>::type;
template <int S> using DigUint = typename std::conditional<(S > 7), unsigned __int128, unsigned long long>::type;

// |v| 2^(8S-1-e) rounded to the nearest integer, with the sign of v, for
// |v| < 2^e, from the bits of v: the FP64 pipe is 1/64 of the integer one on
// this GPU.
template <int S> __device__ __forceinline__ DigInt<S> dig_fixed(double v, int e)
{
    const long long bits = __double_as_longlong(v);
    const int E = (int)((bits >> 52) & 0x7ff);
    unsigned long long f = (unsigned long long)bits & 0xfffffffffffffULL;
    if (E) f |= 1ULL << 52;
    const int sh = max(E, 1) - 1075 + 8 * S - 1 - e;      // |v| = f 2^(max(E,1) - 1075)
    DigUint<S> m = f;
    if (sh >= 0) m <<= (sh < 8 * S - 54 ? sh : 8 * S - 54);      // (sh <= 8 S - 54 for |v| in range)
    else if (sh > -63) m = (f + (1ULL << (-sh - 1))) >> -sh;
    else m = 0;
    return bits < 0 ? -(DigInt<S>)m : (DigInt<S>)m;
}

// Digit s (0 the leading one) of q = sum_s d_s 256^(S-1-s), |d_s| <= 128.
template <int S> __device__ __forceinline__ void dig_split(DigInt<S> q, int d[S])
{
    DigUint<S> half = 0;
#pragma unroll
    for (int s = 1; s < S; ++s) half = (half << 8) | 0x80;
    const DigUint<S> u = (DigUint<S>)q + half;
#pragma unroll
    for (int s = 1; s < S; ++s) d[s] = (int)((unsigned)(u >> (8 * (S - 1 - s))) & 0xff) - 128;
    d[0] = (int)((DigInt<S>)u >> (8 * (S - 1)));
}

__device__ __forceinline__ unsigned dig_bf16x2(int a, int b)
{
    const __nv_bfloat162 p = __floats2bfloat162_rn((float)a, (float)b);
    return *reinterpret_cast<const unsigned *>(&p);
}

// ------------------------------------------------------------ dipole blocks --
template <int PREC> __device__ __forceinline__ double dig_u_at(const void *U, long long q)
{
    if constexpr (PREC == 0) return reinterpret_cast<const double *>(U)[q];
    else if constexpr (PREC == 1) return (double)reinterpret_cast<const float *>(U)[q];
    else {
        const float2 v = reinterpret_cast<const float2 *>(U)[q];
        return (double)v.x + (double)v.y;
    }
}

// High words of the row maxima (first half of eu) and column maxima (second
// half) of every block; one 32 x 32 tile per CTA, 32 x 8 threads.
template <int PREC>
__global__ void dig_umax_kernel(const void *U, long long bstride, int ld, int n, int lmax, int *eu)
{
    const int l = blockIdx.z, j = blockIdx.x * 32 + threadIdx.x;
    int cm = 0;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = blockIdx.y * 32 + r;
        int h = 0;
        if (i < n && j < n) h = __double2hiint(dig_u_at<PREC>(U, l * bstride + (long long)i * ld + j)) & 0x7fffffff;
        cm = max(cm, h);
        const int rm = __reduce_max_sync(0xffffffffu, h);
        if (threadIdx.x == 0 && i < n && rm > 0) atomicMax(eu + (long long)l * n + i, rm);
    }
    if (j < n && cm > 0) atomicMax(eu + (long long)(lmax + l) * n + j, cm);
}

// High words of maxima -> exponents (DIG_NONFINITE stays).
__global__ void dig_uexp_kernel(int *eu, long long count)
{
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < count) eu[q] = eu[q] >= DIG_NONFINITE ? DIG_NONFINITE : dig_exp(eu[q]);
}

// Digits of U_l (scaled per row) and of U_l^T (scaled per column of U_l), the
// latter transposed through shared memory; grid as dig_umax_kernel over ldb
// columns, so the padding is written (zero) too.
template <int PREC, int S>
__global__ void dig_u_kernel(const void *U, long long bstride, int ld, int n, int lmax, int ldb, const int *eu,
                             __nv_bfloat16 *out)
{
    __shared__ double tile[32][33];
    const int l = blockIdx.z;
    const long long plane = (long long)lmax * n * ldb;
    const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = i0 + r, j = j0 + threadIdx.x;
        tile[r][threadIdx.x] = (i < n && j < n) ? dig_u_at<PREC>(U, l * bstride + (long long)i * ld + j) : 0.0;
    }
    __syncthreads();
    for (int tr = 0; tr < 2; ++tr) {
        for (int r = threadIdx.y; r < 32; r += 8) {
            const int row = (tr ? j0 : i0) + r, col = (tr ? i0 : j0) + threadIdx.x;
            if (row >= n || col >= ldb) continue;
            const int e = eu[(long long)(tr * lmax + l) * n + row];
            const double v = tr ? tile[threadIdx.x][r] : tile[r][threadIdx.x];
            int d[S];
            if (e >= DIG_NONFINITE) {
#pragma unroll
                for (int s = 0; s < S; ++s) d[s] = 0;
            } else {
                dig_split<S>(dig_fixed<S>(v, e), d);
            }
            const long long o = ((long long)l * n + row) * ldb + col;
#pragma unroll
            for (int s = 0; s < S; ++s) out[(tr * S + s) * plane + o] = __float2bfloat16_rn((float)d[s]);
        }
    }
}

template <int PREC>
static cudaError_t dig_u_prec(const void *U, long long bstride, int ld, int n, int lmax, int ldb, int *eu,
                              __nv_bfloat16 *digits, cudaStream_t s)
{
    constexpr int S = dig_slices(PREC);
    const dim3 thr(32, 8), grid((ldb + 31) / 32, (n + 31) / 32, lmax);
    const cudaError_t z = cudaMemsetAsync(eu, 0, sizeof(int) * 2 * (size_t)lmax * n, s);
    if (z != cudaSuccess) return z;
    dig_umax_kernel<PREC><<<grid, thr, 0, s>>>(U, bstride, ld, n, lmax, eu);
    const long long cnt = 2LL * lmax * n;
    dig_uexp_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(eu, cnt);
    const dim3 g2((ldb + 31) / 32, (ldb + 31) / 32, lmax);
    dig_u_kernel<PREC, S><<<g2, thr, 0, s>>>(U, bstride, ld, n, lmax, ldb, eu, digits);
    return cudaGetLastError();
}

cudaError_t launch_dig_u(int prec, const void *U, long long bstride, int ld, int n, int lmax, int ldb, int *eu,
                         __nv_bfloat16 *digits, cudaStream_t s)
{
    if (lmax < 1) return cudaSuccess;
    switch (prec) {
    case 0: return dig_u_prec<0>(U, bstride, ld, n, lmax, ldb, eu, digits, s);
    case 1: return dig_u_prec<1>(U, bstride, ld, n, lmax, ldb, eu, digits, s);
    case 2: return dig_u_prec<2>(U, bstride, ld, n, lmax, ldb, eu, digits, s);
    }
    return cudaErrorInvalidValue;
}

// ----------------------------------------------------------------- states --
// grid (chunks of 1024 amplitudes of a block, lmax+1, B)
__global__ void __launch_bounds__(256) dig_max_kernel(const double2 *__restrict__ src, int n, int lmax, int B, int *xmax)
{
    const int l = blockIdx.y, b = blockIdx.z;
    const double2 *p = src + (long long)b * (lmax + 1) * n + (long long)l * n;
    int mr = 0, mi = 0;
    for (int i = blockIdx.x * 1024 + threadIdx.x; i < min(n, (int)blockIdx.x * 1024 + 1024); i += 256) {
        const double2 v = p[i];
        mr = max(mr, __double2hiint(v.x) & 0x7fffffff);
        mi = max(mi, __double2hiint(v.y) & 0x7fffffff);
    }
    mr = __reduce_max_sync(0xffffffffu, mr);
    mi = __reduce_max_sync(0xffffffffu, mi);
    if ((threadIdx.x & 31) == 0) {
        int *o = xmax + (long long)l * 2 * B + 2 * b;
        if (mr > 0) atomicMax(o, mr);
        if (mi > 0) atomicMax(o + 1, mi);
    }
}

cudaError_t launch_dig_max(const double2 *src, int n, int lmax, int B, int *xmax, cudaStream_t s)
{
    dig_max_kernel<<<dim3((n + 1023) / 1024, lmax + 1, B), 256, 0, s>>>(src, n, lmax, B, xmax);
    return cudaGetLastError();
}

// Four amplitudes per thread: 64 bytes in, 8 bytes per digit and plane out.
// Streaming bound: 16 bytes in and 4S bytes out per (pulse, amplitude).
template <int S>
__global__ void __launch_bounds__(128)
dig_x_kernel(const double2 *__restrict__ src, int n, int nb, int lmax, int B, const int *__restrict__ xmax,
             int *__restrict__ xmax_next, __nv_bfloat16 *__restrict__ out)
{
    const int l = blockIdx.y, b = blockIdx.z;
    pdl_launch_dependents();
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x < 2) xmax_next[(long long)l * 2 * B + 2 * b + threadIdx.x] = 0;
    const int i = (blockIdx.x * 128 + threadIdx.x) * 4;
    if (i >= n) return;
    const double2 *p = src + (long long)b * (lmax + 1) * n + (long long)l * n + i;
    double v[2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double2 w = i + q < n ? p[q] : make_double2(0.0, 0.0);
        v[0][q] = w.x;
        v[1][q] = w.y;
    }
    const long long plane = (long long)(lmax + 1) * nb;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
        const int h = xmax[(long long)l * 2 * B + 2 * b + part];
        int d[4][S];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (h >= DIG_NONFINITE) {
#pragma unroll
                for (int s = 0; s < S; ++s) d[q][s] = 0;
            } else {
                dig_split<S>(dig_fixed<S>(v[part][q], dig_exp(h)), d[q]);
            }
        }
        __nv_bfloat16 *o = out + (2LL * b + part) * plane + (long long)l * nb + i;   // (nb, i: multiples of 4)
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const uint2 w = make_uint2(dig_bf16x2(d[0][s], d[1][s]), dig_bf16x2(d[2][s], d[3][s]));
            *reinterpret_cast<uint2 *>(o + (long long)s * 2 * B * plane) = w;
        }
    }
}

cudaError_t launch_dig_x(int slices, const double2 *src, int n, int nb, int lmax, int B, const int *xmax, int *xmax_next,
                         __nv_bfloat16 *digits, cudaStream_t s)
{
    void *args[] = {(void *)&src, (void *)&n, (void *)&nb, (void *)&lmax, (void *)&B, (void *)&xmax, (void *)&xmax_next,
                    (void *)&digits};
    const void *fn = slices == 7 ? (const void *)dig_x_kernel<7> : (const void *)dig_x_kernel<11>;
    return launch_pdl(fn, dim3((n + 511) / 512, lmax + 1, B), dim3(128), 0, s, args);
}

// ----------------------------------------------------------------- launch --
static int dig_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms < 2 ? 2 : sms & ~1;
}

// The tile whose longest CTA (pair) is estimated to finish first.  CTA 0 has the
// longest share of the walk (dig_tile_of).  Cycles of a step (one digit pair of
// tiles, 64 columns): measured 500-530 at 32 planes, 510-600 at 64 and 620-840 at
// 128, 620 and 690 for single CTAs: the issue of the products and their loads
// more than the products themselves, except at 128.  The update of the last tile
// follows its products, some 1000 cycles a pulse.  Measured, us a stage at 32 /
// 64 / 128 planes: FP32, lmax=9, n=487, 100 pulses 155 / 133 / 124, lmax=20, n=200,
// 300 pulses 222 / 153 / 151, lmax=7, n=301, 24 pulses 55 / 61 / 68; float-float,
// lmax=15, n=1000, 256 pulses 1677 / 929 / 632; FP64, lmax=7, n=301, 24 pulses
// 107 / 137, lmax=15, n=1000, 64 pulses 1050 / 799; single CTAs, FP64, lmax=3, n=100,
// 200 pulses 65 / 90.
DigTile dig_tile(int slices, int n, int lmax, int B)
{
    const int cg = n > DBM ? 2 : 1, units = dig_sms() / cg, mt = (n + DBM * cg - 1) / (DBM * cg);
    long long steps = 0;                                 // digit pairs of tiles of a product
    for (int g = 0; g < dig_groups(slices); ++g) steps += (dig_top(slices, g) + 1) * (long long)((n + DBK - 1) / DBK);
    DigTile best{cg, 32};
    long long low = 0;
    for (int bn = 32; bn <= (cg == 2 && !dig_int(slices) ? 128 : 64); bn *= 2) {
        const long long per = (long long)mt * ((2LL * B + bn - 1) / bn), tiles = per * (lmax + 1);
        long long parts = 0;                             // products of CTA 0
        for (long long t = 0; t < tiles; t += units) parts += lmax > 1 && t < per * (lmax - 1) ? 2 : 1;
        const int step = cg == 1 ? (bn == 32 ? 620 : 690) : (bn == 32 ? 510 : (bn == 64 ? 570 : 700));
        const long long est = parts * steps * step + 500LL * bn;
        if (bn == 32 || est < low) {
            low = est;
            best.bn = bn;
        }
    }
    return best;
}

size_t dig_scratch_bytes(DigTile t) { return (size_t)dig_sms() * (t.bn / 2) * DBM * sizeof(float4); }

cudaError_t launch_dig(int slices, DigTile t, const DigMaps &m, const DigArgs &A, cudaStream_t stream)
{
    const void *fn = slices == 7 ? dig_fn7(t.cg, t.bn) : dig_fn11(t.cg, t.bn);
    if (!fn) return cudaErrorInvalidValue;
    const int smem = dig_smem(t.bn, t.cg);
    const cudaError_t e = ensure_dyn_smem(fn, smem);
    if (e != cudaSuccess) return e;
    const int rows = DBM * t.cg;
    const long long ctas = (long long)t.cg * ((A.n + rows - 1) / rows) * ((2 * A.B + t.bn - 1) / t.bn) * (A.lmax + 1);
    void *args[] = {(void *)&m, (void *)&A};
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)(ctas < dig_sms() ? ctas : dig_sms()));
    lc.blockDim = dim3(DIG_THREADS);
    lc.dynamicSmemBytes = (size_t)smem;
    lc.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)t.cg;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = t.cg > 1 ? 2 : 1;
    return cudaLaunchKernelExC(&lc, fn, args);
}

}  // namespace tdse
