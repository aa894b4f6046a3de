// Batched pulses with FP64-class or FP32-class products on the tensor cores
// (tcgen05, sm_103a), by splitting both operands into 8-bit digits.
//
// D_l = U_l X_{l+1} + U_{l-1}^T X_{l-1} (paper Sec. 4, block form of H C for
// all pulses at once).  Every row of a dipole block is scaled by a power of
// two and written as S balanced digits base 256, |d| <= 128,
//     u = 2^(eu-7) sum_s d_s 256^-s,
// every (block, pulse plane) of the state likewise (the error-free splitting
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).  A digit is an
// integer of 8 bits, exact in bf16, and a sum of 1024 products of digits is an
// integer of at most 2^24, exact in the FP32 accumulators of tcgen05.mma: the
// products carry no rounding at all.  Digit pairs (s, t) with s + t <= S - 1
// are multiplied, so what is left out is below S 2^-8S of max|u| max|x| per
// product, the maxima those of the row and of the (block, plane).
//
// The digits are fixed point, and a bound state has one amplitude near 1 and
// others of its block far below, which meet dipole elements that fall off: S is
// chosen so that the sum of such small terms keeps the digits that FP32 or FP64
// products would give it.  7 digits (FP32, float-float) carry terms down to
// 2^-29 of the largest at FP32's accuracy, 11 (FP64) down to 2^-31 at FP64's.
// Largest error of a component of D x over the sum of its own terms' magnitudes,
// the products these replace (FMA pipe, FP64 pipe) and these: hydrogen in a
// sphere of 100 a.u., n=301, 20 a.u. into a pulse, FP32 1.0e-6 and 4.6e-8,
// float-float 3.7e-7 and 1.2e-8, FP64 1.4e-15 and 1.7e-16; one amplitude of 1
// whose elements fall to 1e-7 and a tail of 1e-10, 1.7e-6 and 1.1e-7, 4.7e-7
// and 9.1e-8, 1.2e-15 and 1.7e-16 (with 4, 6 and 8 digits 1.3e-1, 1.0e-5, 1.2e-9).
//
// Pairs of one weight w = s + t share an accumulator.  Weights are taken two
// at a time (w and w - 1, group by group; S odd: weight 0 alone): step s = 0 .. w
// loads A_s and B_{w-s} and multiplies A_s B_{w-s} (weight w) and A_{s-1} B_{w-s}
// (w - 1), so each digit tile is loaded once per group and two steps are live at
// any time.  A group's accumulators are drained before 1024 products have been
// added: every 512 columns of K for w = 0, 320 for 2, 192, 128, 64, 64 for 4 .. 10.
// Two pairs of accumulators in tensor memory let the drain of one overlap the
// products of the next.
//
// Bound: the products, S (S + 1) / 2 bf16 MMAs per element.  CG = 2: a pair of
// CTAs (one TPC) shares a 256-row tile, each loading its own rows of A and half
// of B, which takes the operand traffic of an SM from 73 to 55 bytes per tensor
// cycle (L2) and from 128 to 96 (shared memory reads; 128 is what it delivers).
// CG = 1 serves blocks of at most 128 rows.
//
// Warps 0 and 3 stream the digit tiles with TMA, one thread of warp 1 issues the
// MMAs, two warpgroups drain the accumulators into per-thread running sums, and
// two more apply the FP64 stage update while they are at the next tile: the
// update is bound by the FP64 pipe (2 operations per cycle and SM; 8-10 per
// amplitude here), and run by the draining warps it stalled the products.
// Measured on GB300, one stage of 256 pulses, lmax=15, n=1000 (31 GFLOP of real
// products): float-float 3637 (FMA pipe, bgemm_df.cu) -> 632 us, FP32 945
// (batch.cu) -> 628 us; FP64, 24 pulses, lmax=7, n=301: 649 (pulse by pulse) ->
// 107 us.  28 products at the bf16 rate of 1927 TFLOP/s would take 455 us.  Of the
// way there (float-float, 6 digits): 128-row tiles of single CTAs updated by the
// draining warps 1305 us, pairs with updating warps 898, the whole-warp issue loop
// (elect_one) 603, states by bulk copies 560, eight updating warps 509.  What is
// left: a step (24 KB of operands a CTA) takes 620 cycles against 448 of products,
// 40 bytes a cycle and SM out of L2.
// All waits are bounded (sync.cuh).
#pragma once
#include <type_traits>

#include "dig.h"
#include "kernels.h"
#include "sync.cuh"
#include "tcgen.cuh"

namespace tdse {

constexpr int DBM = 128, DBK = 64;
constexpr int DA_BYTES = DBM * DBK * 2;                 // 16 KB
constexpr int DIG_DRAIN_WARPS = 8, DIG_UPD_WARPS = 8;
constexpr int DIG_THREADS = 128 + 32 * (DIG_DRAIN_WARPS + DIG_UPD_WARPS);   // warps 0..3: loads of A, MMA issue, state loads, loads of B
// Registers: launched with 96 per thread.  Where a draining thread holds 128
// words of running sums, the first warpgroup keeps 32, the draining ones take
// 160 each and the updating ones keep 64: 128 * (32 + 2 * 160 + 2 * 64) =
// 640 * 96; else 40, 144, 72.
constexpr int DIG_REGS_LAUNCH = 96;
__host__ __device__ constexpr bool dig_wide(int S, int bn) { return bn * (S > 7 ? 2 : 1) >= 128; }
__host__ __device__ constexpr int dig_regs_low(bool wide) { return wide ? 32 : 40; }
__host__ __device__ constexpr int dig_regs_drain(bool wide) { return wide ? 160 : 144; }
__host__ __device__ constexpr int dig_regs_upd(bool wide) { return wide ? 64 : 72; }
__host__ __device__ constexpr int dig_regs(bool wide) { return 128 * dig_regs_low(wide) + 32 * DIG_DRAIN_WARPS * dig_regs_drain(wide) + 32 * DIG_UPD_WARPS * dig_regs_upd(wide); }
static_assert(dig_regs(true) <= DIG_THREADS * DIG_REGS_LAUNCH && dig_regs(false) <= DIG_THREADS * DIG_REGS_LAUNCH, "register split");
constexpr uint64_t DIG_WAIT_NS = 2000000000ull;
constexpr int DIG_SUPER = 8;                            // K tiles (of 64) per round over the groups
constexpr int DIG_NONFINITE = 0x7ff00000;               // xmax / eu mark of a non-finite maximum

__host__ __device__ constexpr int dig_stage_bytes(int bn, int cg) { return DA_BYTES + bn / cg * DBK * 2; }
__host__ __device__ constexpr int dig_stages(int bn, int cg) { return 196608 / dig_stage_bytes(bn, cg); }
// Behind the operand ring: DIG_NSU slots of the states (c, x, acc) of one pulse and the tile's rows, which
// DIG_UPD_GROUPS groups of updating warps take in turn.  A wait by parity tells a phase from the one before
// only, so a waiter must have seen every phase of its barrier: with a multiple of the groups a slot stays
// with one group within a tile, and the next tile starts (d_full) when both have finished (d_empty).
constexpr int DIG_NSU = 4, DIG_SLOT = 3 * DBM * 16;
constexpr int DIG_UPD_GROUPS = 2;
static_assert(DIG_NSU % DIG_UPD_GROUPS == 0 && DIG_UPD_GROUPS == 2, "a state slot must not change hands within a tile");
__host__ __device__ constexpr int dig_smem(int bn, int cg)
{
    return dig_stages(bn, cg) * dig_stage_bytes(bn, cg) + DIG_NSU * DIG_SLOT + 1024;
}

// Weights are taken two at a time: group g has the pairs of weight dig_top(S, g) and of the one below
// (S odd: group 0 has weight 0 alone).
__host__ __device__ constexpr int dig_groups(int S) { return (S + 1) / 2; }
__host__ __device__ constexpr int dig_top(int S, int g) { return 2 * g + 1 - (S & 1); }
// K tiles the accumulators of top weight w take before a drain: (w+1) pairs times 64 per tile <= 1024 products.
__host__ __device__ constexpr int dig_chunk(int w) { return w == 0 ? 8 : 16 / (w + 1); }
__host__ __device__ constexpr bool dig_int(int S) { return S > 7; }      // FP64 contexts: integer sums

// Running sums of NC outputs of one thread, in units of 2^(eu+ex-14).
// FP32 / float-float contexts: a float-float pair, the three leading weights
// added exactly (TwoSum), the others in FP32.
template <int S, int NC> struct DigAcc {
    float h[NC], l[NC];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int j = 0; j < NC; ++j) { h[j] = 0.f; l[j] = 0.f; }
    }
    __device__ __forceinline__ void add(int j, float v)
    {
        const df s = df_two_sum(h[j], v);
        h[j] = s.h;
        l[j] = __fadd_rn(l[j], s.l);
    }
    // a sum of products of weight W
    template <int W> __device__ __forceinline__ void fold(int j, float v)
    {
        constexpr float unit = 1.0f / (1ULL << (8 * W));
        if constexpr (W == 0) add(j, v);
        else if constexpr (W <= 2) add(j, __fmul_rn(v, unit));
        else l[j] = __fmaf_rn(v, unit, l[j]);
    }
};

// FP64 contexts: weights 0..4 as an exact integer in units of the fourth, 5..9 as one in units of the ninth
// (|sum| < 2^59 and 2^61 for K <= 4096), into which the tenth is rounded.
template <int NC> struct DigAcc<11, NC> {
    long long a[NC], b[NC];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int j = 0; j < NC; ++j) { a[j] = 0; b[j] = 0; }
    }
    template <int W> __device__ __forceinline__ void fold(int j, float v)
    {
        if constexpr (W == 10) b[j] += (long long)__float2int_rn(__fmul_rn(v, 0x1p-8f));
        else if constexpr (W > 4) b[j] += (long long)__float2int_rn(v) << (8 * (9 - W));
        else a[j] += (long long)__float2int_rn(v) << (8 * (4 - W));
    }
    // The sum times 2^e, rounded to nearest, from the bits: in FP64, conversions, sum and scale held the pipe
    // 20000 cycles a product (a conversion or an addition takes 19 cycles a warp instruction).
    __device__ __forceinline__ double value(int j, int e) const
    {
        // a 2^40 + b in four words
        const long long c = b[j] >> 40;                                      // what b carries into a
        const unsigned long long lo = (unsigned long long)(b[j] - (c << 40)), hi = (unsigned long long)(a[j] + c);
        unsigned h = (unsigned)((long long)hi >> 56), m = (unsigned)(hi >> 24), l = (unsigned)(hi << 8) | (unsigned)(lo >> 32);
        unsigned t = (unsigned)lo;
        const unsigned neg = (unsigned)((int)h >> 31);                       // all ones if negative
        if (neg) {
            t = ~t + 1u;
            l = ~l + (t == 0u);
            m = ~m + (t == 0u && l == 0u);
            h = ~h + (t == 0u && l == 0u && m == 0u);
        }
        if ((h | m | l | t) == 0u) return 0.0;
        int x = 127 - 72 + e;                                                // weight of the leading bit of (h m l t)
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (h == 0u) { h = m; m = l; l = t; t = 0u; x -= 32; }
        const int z = __clz((int)h);
        h = __funnelshift_l(m, h, z);
        m = __funnelshift_l(l, m, z);
        l = __funnelshift_l(t, l, z);
        t <<= z;
        x -= z;                                                              // value = 1.x 2^x, leading bit at the top of h
        unsigned long long r = ((unsigned long long)h << 32) | m;
        const unsigned low = (unsigned)(r & 0x7ffu);
        r >>= 11;
        if (low > 0x400u || (low == 0x400u && ((l | t) != 0u || (r & 1u)))) ++r;
        if (x > -1000 && x < 1000)
            // (the leading bit of r adds 1 to the exponent field)
            return __longlong_as_double((long long)((r + ((unsigned long long)(x + 1022) << 52)) |
                                                    ((unsigned long long)(neg & 0x80000000u) << 32)));
        const double v = scalbn((double)r, x - 52);
        return neg ? -v : v;
    }
};

// Exponent of the power of two above a maximum with high word h.
__device__ __forceinline__ int dig_exp(int h) { return max(h >> 20, 1) - 1022; }

__device__ __forceinline__ float dig_pow2f(int e)       // 2^e for e <= 127, 0 below 2^-126
{
    return e < -126 ? 0.f : __int_as_float((e + 127) << 23);
}

// f 2^e for a float f that is zero or normal (a subnormal f counts as zero) and |e| < 800, from the bits of f.
__device__ __forceinline__ double dig_widen(float f, int e)
{
    const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
    const unsigned hi = (b & 0x80000000u) | ((m >> 3) + ((unsigned)(896 + e) << 20));
    return m < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

__device__ __forceinline__ double dig_join(float h, float l, int e)     // (h + l) 2^e
{
    if (e > -800 && e < 800) return dig_widen(h, e) + dig_widen(l, e);
    return scalbn((double)h + (double)l, e);
}

// Biased exponents (+ 2048) of a pulse's two columns in 16-bit halves, bit 15 of a half: not finite.
__device__ __forceinline__ int dig_pack(const int *m)
{
    const int2 h = *reinterpret_cast<const int2 *>(m);
    return (dig_exp(h.x) + 2048 + (h.x >= DIG_NONFINITE ? 0x8000 : 0)) |
           (int)((unsigned)(dig_exp(h.y) + 2048 + (h.y >= DIG_NONFINITE ? 0x8000 : 0)) << 16);
}

// The shift applied to the first product's sum, in exponents of the two products' units.
__device__ __forceinline__ int dig_shift(int e0, int e1) { return min(e0 - e1, 100); }

// One amplitude of a scratch tile: (re, im) of D x, as float-float sums in the
// product's unit (FP32 / float-float contexts) or as doubles (FP64 contexts).
union DigOut {
    float4 f;
    double2 d;
    __device__ DigOut() {}
};

// A stage's inputs of one (pulse, amplitude) and the update of batch.h's batch_update.
struct DigIn { double2 c, x, acc; };

__device__ __forceinline__ bool dig_first(const DigArgs &A) { return A.mode == EPI_RK4 ? A.stage == 0 : A.stage == 1; }

// The update's results: the next stage's input and the accumulator.  KIND is a
// template parameter because the compiler evaluates short alternatives of a
// uniform branch side by side, and every FP64 instruction holds the pipe for
// 16 cycles (measured 64 per warp instruction of one scheduler): the four
// alternatives together took 1150 cycles a pulse, one takes 600.
struct DigNext { double2 out, acc; };
enum { DIG_RK4_FIRST, DIG_RK4_MID, DIG_RK4_LAST, DIG_TAYLOR };

template <int KIND>
__device__ __forceinline__ DigNext dig_update(const DigArgs &A, double e, double f, double dr, double di, const DigIn &in)
{
    if (A.gauge) { const double t = dr; dr = -di; di = t; }
    const double hr = e * in.x.x + f * dr;
    const double hi = e * in.x.y + f * di;
    const double kr = hi, ki = -hr;
    DigNext r;
    if constexpr (KIND == DIG_RK4_FIRST || KIND == DIG_RK4_MID) {
        r.acc = KIND == DIG_RK4_FIRST ? make_double2(kr, ki) : make_double2(in.acc.x + 2.0 * kr, in.acc.y + 2.0 * ki);
        r.out = make_double2(in.c.x + A.step * kr, in.c.y + A.step * ki);
    } else if constexpr (KIND == DIG_RK4_LAST) {
        r.out = make_double2(in.c.x + A.step * (in.acc.x + kr), in.c.y + A.step * (in.acc.y + ki));
        r.acc = r.out;
    } else {
        const double2 T = make_double2(A.step * kr, A.step * ki);
        const double2 base = A.stage == 1 ? in.x : in.acc;
        r.acc = make_double2(base.x + T.x, base.y + T.y);
        r.out = A.stage < A.order ? T : r.acc;
    }
    return r;
}

// Tile t of the walk: interior blocks (two products) first, the end blocks
// (one product) last, so that the last round of tiles is the short ones.
__device__ __forceinline__ void dig_tile_of(int t, int per_block, int L, int &l, int &rem)
{
    const int q = t / per_block;
    rem = t % per_block;
    l = L == 1 ? 0 : (q < L - 2 ? q + 1 : (q == L - 2 ? 0 : L - 1));
}

template <int S, int BN, int CG>
__global__ void __launch_bounds__(DIG_THREADS, 1)
dig_kernel(const __grid_constant__ DigMaps M, const DigArgs A)
{
    constexpr int NG = dig_groups(S);
    constexpr int NC = BN / 2;                          // columns per draining thread
    static_assert(NG <= 6, "groups");
    constexpr int STAGE = dig_stage_bytes(BN, CG);
    constexpr int NST = dig_stages(BN, CG);

    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[NST];
    __shared__ __align__(8) uint64_t empty[NST];
    __shared__ __align__(8) uint64_t acc_full[2];
    __shared__ __align__(8) uint64_t acc_empty[2];
    __shared__ __align__(8) uint64_t d_full, d_empty;   // this CTA's scratch tile of D x
    __shared__ __align__(8) uint64_t st_full[DIG_NSU], st_empty[DIG_NSU];
    __shared__ __align__(8) uint64_t mma_drain;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ int issued[2], consumed;
    __shared__ int st_issued;
    unsigned char *slots = smem + (size_t)NST * STAGE;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp-uniform)
    const int rank = CG == 2 ? (int)cluster_rank() : 0;
    const int n = A.n, L = A.lmax + 1;
    const int nk = (n + DBK - 1) / DBK;
    const int mt = (n + DBM * CG - 1) / (DBM * CG);
    const int nt = (2 * A.B + BN - 1) / BN;
    const int ntiles = mt * nt * L;
    const int first = blockIdx.x / CG, stride = gridDim.x / CG;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&acc_full[a], 1);
            mbar_init(&acc_empty[a], CG * DIG_DRAIN_WARPS);
        }
        mbar_init(&d_full, DIG_DRAIN_WARPS);
        mbar_init(&d_empty, DIG_UPD_WARPS);
        for (int q = 0; q < DIG_NSU; ++q) {
            mbar_init(&st_full[q], 1);
            mbar_init(&st_empty[q], DIG_UPD_WARPS / DIG_UPD_GROUPS);
        }
        mbar_init(&mma_drain, 1);
        st_issued = 0;
        abort_flag = 0;
        issued[0] = issued[1] = 0;
        consumed = 0;
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc<CG>(&tmem_base, 4 * BN);
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_all();           // the peer's barriers are initialised
    tc_fence_after();
    volatile int *abort = &abort_flag;
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
    pdl_launch_dependents();
    pdl_wait();                                          // state digits and maxima come from the previous kernel

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(dig_regs_low(dig_wide(S, BN))));
        if (warp == 0 || warp == 3) {
            // ------- operand loads: warp 0 those of A (rows of U), warp 3 those of B (pulse planes)
            // Whole-warp loops with an elected issuer, as the products below: one
            // diverged lane loading both took 400 cycles a step.
            const bool isb = warp == 3;
            const CUtensorMap *tm = isb ? &M.X : &M.U;
            int s = 0, it = 0;
            uint32_t ph = 1;                             // parity of the slot's previous release
            bool ok = true;
            for (int t = first; t < ntiles && ok; t += stride) {
                int l, rem;
                dig_tile_of(t, mt * nt, L, l, rem);
                const int y = isb ? (rem % nt) * BN + rank * (BN / CG) : ((rem / nt) * CG + rank) * DBM;
                for (int part = 0; part < 2 && ok; ++part) {
                    if ((part == 0 && l >= A.lmax) || (part == 1 && l < 1)) continue;
                    const int za = part * S * A.lmax + (part == 0 ? l : l - 1), dz = isb ? -1 : A.lmax;
                    const int xcol = isb ? (part == 0 ? l + 1 : l - 1) * A.nb : 0;
                    for (int k0 = 0; k0 < nk && ok; k0 += DIG_SUPER)
                        for (int g = NG - 1; g >= 0 && ok; --g) {
                            const int k1 = min(k0 + DIG_SUPER, nk);
                            for (int kb = k0; kb < k1 && ok; ++kb) {
                                const int w = dig_top(S, g);
                                int z = isb ? w : za;                        // digit plane of step 0
                                for (int st = 0; st <= w; ++st, z += dz) {
                                    if (it >= NST) {
                                        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&empty[s], ph, abort, DIG_WAIT_NS)) != 0;
                                        if (!ok) break;
                                    }
                                    if (elect_one()) {
                                        unsigned char *p = smem + (size_t)s * STAGE + (isb ? DA_BYTES : 0);
                                        if (!isb && rank == 0) mbar_arrive_expect_tx(&full[s], CG * STAGE);
                                        if constexpr (CG == 2) tma_load_3d_pair(p, tm, xcol + kb * DBK, y, z, cluster_addr(&full[s], 0));
                                        else tma_load_3d(p, tm, xcol + kb * DBK, y, z, &full[s]);
                                    }
                                    __syncwarp();
                                    ++it;
                                    if (++s == NST) { s = 0; ph ^= 1; }
                                }
                            }
                        }
                }
            }
            if (lane == 0) issued[isb] = it;
        } else if (warp == 1 && rank == 0) {
            // ----------------------------------- MMA issuer (of the pair's even CTA)
            constexpr uint32_t idesc = idesc_bf16(DBM * CG, BN);
            auto mma = [](uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
                if constexpr (CG == 2) mma_bf16_pair(d, a, b, idesc, acc);
                else mma_bf16(d, a, b, idesc, acc);
            };
            auto commit = [](uint64_t *bar) {
                if constexpr (CG == 2) mma_commit_pair(bar);
                else mma_commit(bar);
            };
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, abort, DIG_WAIT_NS)) != 0;
            };
            const uint64_t d0 = desc_sw128(smem_u32(smem));
            int s = 0, j = 0, done = 0;                  // ring slot, accumulator pairs, stages
            uint32_t ph = 0;                             // the slot's phase
            bool ok = true;
            for (int t = first; t < ntiles && ok; t += stride) {
                int l, rem;
                dig_tile_of(t, mt * nt, L, l, rem);
                const int parts = (l < A.lmax ? 1 : 0) + (l >= 1 ? 1 : 0);
                for (int part = 0; part < parts && ok; ++part)
                    for (int k0 = 0; k0 < nk && ok; k0 += DIG_SUPER)
                        for (int g = NG - 1; g >= 0 && ok; --g) {
                            const int k1 = min(k0 + DIG_SUPER, nk), w = dig_top(S, g), chunk = dig_chunk(w);
                            for (int kc = k0; kc < k1 && ok; kc += chunk, ++j) {
                                const int ab = j & 1;
                                if (j >= 2 && !wait(&acc_empty[ab], (uint32_t)(((j >> 1) - 1) & 1))) { ok = false; break; }
                                tc_fence_after();
                                const uint32_t dodd = tmem + (uint32_t)(ab * 2 * BN), deven = dodd + BN;
                                const int ke = min(kc + chunk, k1);
                                for (int kb = kc; kb < ke && ok; ++kb) {
                                    uint64_t aprev = d0;
                                    int sprev = s;
                                    for (int st = 0; st <= w; ++st) {
                                        if (!wait(&full[s], ph)) { ok = false; break; }
                                        tc_fence_after();
                                        const uint64_t da = d0 + (uint64_t)(s * (STAGE >> 4)), db = da + (DA_BYTES >> 4);
                                        const uint32_t fresh = kb > kc ? 1u : 0u;
                                        if (elect_one()) {
#pragma unroll
                                            for (int kk = 0; kk < DBK / 16; ++kk)         // 16 bf16 = 32 bytes along K
                                                mma(dodd, da + 2 * kk, db + 2 * kk, kk > 0 || st > 0 ? 1u : fresh);
                                            if (st > 0) {
#pragma unroll
                                                for (int kk = 0; kk < DBK / 16; ++kk)
                                                    mma(deven, aprev + 2 * kk, db + 2 * kk, kk > 0 || st > 1 ? 1u : fresh);
                                                commit(&empty[sprev]);       // its A was last read here
                                            }
                                            if (st == w) commit(&empty[s]);
                                        }
                                        __syncwarp();
                                        aprev = da;
                                        sprev = s;
                                        ++done;
                                        if (++s == NST) { s = 0; ph ^= 1; }
                                    }
                                }
                                if (ok && elect_one()) commit(&acc_full[ab]);
                                __syncwarp();
                            }
                        }
            }
            if (lane == 0) consumed = done;
        } else if (warp == 2) {
            // ------------------------------------------ state loads for the update
            if (lane == 0) {
                const bool first_stage = dig_first(A);
                const bool need_c = A.mode == EPI_RK4 || first_stage;
                const uint64_t pol = l2_evict_first_policy();
                int it = 0;
                for (int t = first; t < ntiles && !*abort; t += stride) {
                    int l, rem;
                    dig_tile_of(t, mt * nt, L, l, rem);
                    const int i0 = ((rem / nt) * CG + rank) * DBM, b0 = (rem % nt) * (BN / 2);
                    const uint32_t bytes = (uint32_t)(min(DBM, n - i0) * 16);
                    if (i0 >= n) continue;
                    const int np = min(BN / 2, A.B - b0);
                    for (int p = 0; p < np; ++p, ++it) {
                        const int s = it % DIG_NSU;
                        if (it >= DIG_NSU && !mbar_wait_bounded(&st_empty[s], (uint32_t)((it / DIG_NSU - 1) & 1), abort, DIG_WAIT_NS))
                            break;
                        unsigned char *d = slots + s * DIG_SLOT;
                        const long long q = (long long)(b0 + p) * A.N + (long long)l * n + i0;
                        mbar_arrive_expect_tx(&st_full[s], ((need_c ? 1 : 0) + (first_stage ? 0 : 2)) * bytes);
                        if (need_c) bulk_g2s(d, A.c + q, bytes, &st_full[s], pol);
                        if (!first_stage) {
                            bulk_g2s(d + DBM * 16, A.x + q, bytes, &st_full[s], pol);
                            bulk_g2s(d + 2 * DBM * 16, A.acc + q, bytes, &st_full[s], pol);
                        }
                        st_issued = it + 1;
                    }
                }
            }
        }
    } else if (warp < 4 + DIG_DRAIN_WARPS) {
        // ------------------------------------------- draining warps 4..11
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(dig_regs_drain(dig_wide(S, BN))));
        const int quarter = warp & 3;                    // TMEM lanes this warp may read
        const int half = (warp - 4) >> 2;                // which half of the tile's columns
        const int ncol = 2 * A.B;
        DigOut *scr = reinterpret_cast<DigOut *>(A.scratch) + ((size_t)blockIdx.x * (BN / 2) + half * (NC / 2)) * DBM +
                      quarter * 32 + lane;               // [pulse][row]
        int j = 0, jt = 0;
        bool ok = true;
        for (int t = first; t < ntiles && ok; t += stride, ++jt) {
            int l, rem;
            dig_tile_of(t, mt * nt, L, l, rem);
            const int row = ((rem / nt) * CG + rank) * DBM + quarter * 32 + lane;
            const int c0 = (rem % nt) * BN + half * NC;
            const bool both = l >= 1 && l < A.lmax && row < n;
            DigAcc<S, NC> R;
            R.clear();
            const int eu0 = both ? A.eu[(long long)l * n + row] : 0;
            const int eu1 = both ? A.eu[(long long)(A.lmax + l - 1) * n + row] : 0;
            auto unit = [&](auto wc) {                   // drain one pair of accumulators of top weight W
                constexpr int W = decltype(wc)::value;
                const int ab = j & 1;
                bool have = mbar_wait_bounded(&acc_full[ab], (uint32_t)((j >> 1) & 1), abort, DIG_WAIT_NS);
                have = __all_sync(0xffffffffu, have);
                if (!have) { ok = false; return; }
                tc_fence_after();
                const uint32_t ta = tmem + (uint32_t)(ab * 2 * BN + half * NC) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
                for (int ch = 0; ch < NC / 8; ++ch) {
                    float vo[8], ve[8];
                    tmem_ld8x2(ta + (uint32_t)(ch * 8), ta + (uint32_t)(BN + ch * 8), vo, ve);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if constexpr (W > 2) {           // the smaller first
                            R.template fold<W>(ch * 8 + q, vo[q]);
                            R.template fold<W - 1>(ch * 8 + q, ve[q]);
                        } else {
                            R.template fold<W>(ch * 8 + q, vo[q]);
                            if constexpr (W > 0) R.template fold<W - 1>(ch * 8 + q, ve[q]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (CG == 2) mbar_arrive_cluster(cluster_addr(&acc_empty[ab], 0));
                    else mbar_arrive(&acc_empty[ab]);
                }
                ++j;
            };
            bool claimed = false;                        // the update has left the scratch tile
            auto claim = [&]() {
                if (!claimed && jt > 0)
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(&d_empty, (uint32_t)((jt - 1) & 1), abort, DIG_WAIT_NS));
                claimed = true;
            };
            for (int part = 0; part < 2 && ok; ++part) {
                if ((part == 0 && l >= A.lmax) || (part == 1 && l < 1)) continue;
                for (int k0 = 0; k0 < nk && ok; k0 += DIG_SUPER) {
                    const int k1 = min(k0 + DIG_SUPER, nk);
                    auto group = [&](auto gc) {
                        constexpr int G = decltype(gc)::value;
                        if constexpr (G < NG) {
                            constexpr int W = dig_top(S, G);
                            for (int kc = k0; kc < k1 && ok; kc += dig_chunk(W)) unit(std::integral_constant<int, W>{});
                        }
                    };
                    group(std::integral_constant<int, 5>{});
                    group(std::integral_constant<int, 4>{});
                    group(std::integral_constant<int, 3>{});
                    group(std::integral_constant<int, 2>{});
                    group(std::integral_constant<int, 1>{});
                    group(std::integral_constant<int, 0>{});
                }
                if (part == 0 && l >= 1 && ok) {
                    // the second product has other row and column exponents
                    const int *m0 = A.xmax + (long long)(l + 1) * ncol, *m1 = A.xmax + (long long)(l - 1) * ncol;
                    if constexpr (dig_int(S)) {
                        claim();
                        if (!ok) break;
#pragma unroll
                        for (int p = 0; p < NC / 2; ++p) {
                            const int col = c0 + 2 * p;
                            double2 v = make_double2(0.0, 0.0);
                            if (both && col < ncol)
                                v = make_double2(R.value(2 * p, eu0 + dig_exp(m0[col]) - 14),
                                                 R.value(2 * p + 1, eu0 + dig_exp(m0[col + 1]) - 14));
                            scr[p * DBM].d = v;
                        }
                        R.clear();
                    } else {
#pragma unroll
                        for (int q = 0; q < NC; ++q) {
                            // rescale the sum so far to the second product's unit (its value below 2^-100 of the
                            // other's unit is lost, far under the digits left out); velocity gauge: minus the second
                            int x = 0;
                            if (both && c0 + q < ncol) x = dig_shift(eu0 + dig_exp(m0[c0 + q]), eu1 + dig_exp(m1[c0 + q]));
                            const float sc = A.gauge ? -dig_pow2f(x) : dig_pow2f(x);
                            R.h[q] = __fmul_rn(R.h[q], sc);
                            R.l[q] = __fmul_rn(R.l[q], sc);
                        }
                    }
                }
            }
            if (!ok) break;
            claim();
            if (!ok) break;
#pragma unroll
            for (int p = 0; p < NC / 2; ++p) {
                if constexpr (dig_int(S)) {
                    const int col = c0 + 2 * p;
                    double2 v = make_double2(0.0, 0.0);
                    if (row < n && col < ncol) {
                        const int *m = A.xmax + (long long)(l >= 1 ? l - 1 : l + 1) * ncol + col;
                        const int e = (l >= 1 ? A.eu[(long long)(A.lmax + l - 1) * n + row] : A.eu[(long long)l * n + row]) - 14;
                        v = make_double2(R.value(2 * p, e + dig_exp(m[0])), R.value(2 * p + 1, e + dig_exp(m[1])));
                        if (l >= 1 && A.gauge) v = make_double2(-v.x, -v.y);
                        if (both) {
                            const double2 w = scr[p * DBM].d;
                            v = make_double2(v.x + w.x, v.y + w.y);
                        }
                    }
                    scr[p * DBM].d = v;
                } else {
                    scr[p * DBM].f = make_float4(R.h[2 * p], R.l[2 * p], R.h[2 * p + 1], R.l[2 * p + 1]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&d_full);
        }
    } else {
        // ------------------------------------------- updating warps 12..19
        // Two groups of four warps (128 rows) take the pulses in turn: a pulse is
        // a chain of some 1200 cycles besides the 640 its FP64 instructions hold
        // a scheduler's pipe, so one group alone leaves that pipe idle.  The states
        // of a pulse are staged in shared memory by warp 2 (a load takes some 3500
        // cycles behind the operand tiles), D x is read one pulse ahead.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(dig_regs_upd(dig_wide(S, BN))));
        const int grp = (warp - 4 - DIG_DRAIN_WARPS) >> 2;
        const int r0 = (warp & 3) * 32 + lane;
        const int ncol = 2 * A.B;
        const bool first_stage = dig_first(A);
        const bool last_stage = A.stage == (A.mode == EPI_RK4 ? 3 : A.order);
        const DigOut *scr = reinterpret_cast<const DigOut *>(A.scratch) + (size_t)blockIdx.x * (BN / 2) * DBM + r0;
        int jt = 0, it0 = 0;                             // tiles, state slots before this tile
        bool ok = true;
        for (int t = first; t < ntiles && ok; t += stride, ++jt) {
            int l, rem;
            dig_tile_of(t, mt * nt, L, l, rem);
            const int i0 = ((rem / nt) * CG + rank) * DBM, row = i0 + r0;
            const int b0 = (rem % nt) * (BN / 2);        // first pulse
            const int np = i0 < n ? min(BN / 2, A.B - b0) : 0;
            const bool valid = row < n;
            const bool up = l < A.lmax, dn = l >= 1;
            int eu0 = valid && up ? A.eu[(long long)l * n + row] : 0;
            int eu1 = valid && dn ? A.eu[(long long)(A.lmax + l - 1) * n + row] : 0;
            const int ubad = max(eu0, eu1) >= DIG_NONFINITE ? 0x80008000 : 0;
            const long long a = (long long)b0 * A.N + (long long)l * n + row;
            const double e = valid ? A.E[(long long)l * n + row] : 0.0;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&d_full, (uint32_t)(jt & 1), abort, DIG_WAIT_NS)) != 0;
            if (!ok) break;
            DigOut nx;
            nx.f = scr[grp * DBM].f;
            auto pulses = [&](auto kc) {
                constexpr int KIND = decltype(kc)::value;
#pragma unroll 1
                for (int p32 = 0; p32 < np && ok; p32 += 32) {
                    // pulse b0 + p32 + lane: field value, exponents of the columns of the two products (two 16-bit
                    // halves, bias 2048, bit 15: not finite); the maxima of column lane % 2 of the group's pulse lane / 2
                    const int pb = b0 + p32 + lane;
                    const double fv = pb < A.B ? field_at(A.field + (long long)pb * A.S, A.sps, A.k, A.h) : 0.0;
                    const int x0 = up && pb < A.B ? dig_pack(A.xmax + (long long)(l + 1) * ncol + 2 * pb) : 0;
                    const int x1 = dn && pb < A.B ? dig_pack(A.xmax + (long long)(l - 1) * ncol + 2 * pb) : 0;
                    int mine = 0;
                    const int pe = min(p32 + 32, np);
#pragma unroll 1
                    for (int p = p32 + grp; p < pe; p += DIG_UPD_GROUPS) {
                        DigOut o;
                        o.f = nx.f;
                        nx.f = scr[min(p + DIG_UPD_GROUPS, BN / 2 - 1) * DBM].f;
                        const int it = it0 + p, s = it % DIG_NSU;
                        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&st_full[s], (uint32_t)((it / DIG_NSU) & 1), abort, DIG_WAIT_NS)) != 0;
                        if (!ok) return;
                        const double2 *sl = reinterpret_cast<const double2 *>(slots + s * DIG_SLOT) + r0;
                        DigIn in;
                        in.c = sl[0];
                        in.x = first_stage ? in.c : sl[DBM];
                        in.acc = sl[2 * DBM];
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&st_empty[s]);
                        const int q = p & 31;
                        const double f = __shfl_sync(0xffffffffu, fv, q);
                        const int s0 = __shfl_sync(0xffffffffu, x0, q), s1 = __shfl_sync(0xffffffffu, x1, q);
                        const int bad = s0 | s1 | ubad;
                        double d[2];
#pragma unroll
                        for (int w = 0; w < 2; ++w) {
                            if constexpr (dig_int(S)) {
                                d[w] = w ? o.d.y : o.d.x;
                            } else {
                                const int e0 = eu0 + ((s0 >> (16 * w)) & 0x7fff), e1 = eu1 + ((s1 >> (16 * w)) & 0x7fff);
                                int ee = e0;
                                if (dn) ee = up ? e1 + max(e0 - e1 - 100, 0) : e1;
                                const float4 v = o.f;
                                d[w] = dig_join(w ? v.z : v.x, w ? v.w : v.y, ee - (2048 + 14));
                                if (dn && A.gauge) d[w] = -d[w];
                            }
                            if (bad & (0x8000 << (16 * w))) d[w] = __longlong_as_double(0x7ff8000000000000LL);
                        }
                        const DigNext nw = dig_update<KIND>(A, e, f, d[0], d[1], in);
                        if (valid) {
                            const long long at = a + (long long)p * A.N;
                            if (last_stage) {
                                A.c[at] = nw.out;
                            } else {
                                A.x[at] = nw.out;
                                A.acc[at] = nw.acc;
                            }
                        }
                        const int mr = (int)__reduce_max_sync(0xffffffffu, valid ? (unsigned)__double2hiint(nw.out.x) & 0x7fffffffu : 0u);
                        const int mi = (int)__reduce_max_sync(0xffffffffu, valid ? (unsigned)__double2hiint(nw.out.y) & 0x7fffffffu : 0u);
                        if ((lane >> 1) == (q >> 1)) mine = lane & 1 ? mi : mr;
                    }
                    const int pl = p32 + 2 * (lane >> 1) + grp;
                    if (pl < pe && mine > 0) atomicMax(A.xmax_next + (long long)l * ncol + 2 * (b0 + pl) + (lane & 1), mine);
                }
            };
            switch (A.mode != EPI_RK4 ? DIG_TAYLOR : A.stage == 0 ? DIG_RK4_FIRST : A.stage < 3 ? DIG_RK4_MID : DIG_RK4_LAST) {
            case DIG_RK4_FIRST: pulses(std::integral_constant<int, DIG_RK4_FIRST>{}); break;
            case DIG_RK4_MID: pulses(std::integral_constant<int, DIG_RK4_MID>{}); break;
            case DIG_RK4_LAST: pulses(std::integral_constant<int, DIG_RK4_LAST>{}); break;
            default: pulses(std::integral_constant<int, DIG_TAYLOR>{});
            }
            if (!ok) break;
            it0 += np;
            __syncwarp();
            if (lane == 0) mbar_arrive(&d_empty);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) {
        // Let copies still in flight land before the CTA's shared memory goes
        // away (a pair's copies complete on the even CTA's barriers).
        volatile int never = 0;
        for (int q = consumed; rank == 0 && q < max(issued[0], issued[1]); ++q)
            mbar_wait_bounded(&full[q % NST], (uint32_t)((q / NST) & 1), &never, DIG_WAIT_NS);
        // (a slot's earlier copies had landed when it was filled again, and a wait by parity would not see them)
        for (int q = max(st_issued - DIG_NSU, 0); q < st_issued; ++q)
            mbar_wait_bounded(&st_full[q % DIG_NSU], (uint32_t)((q / DIG_NSU) & 1), &never, DIG_WAIT_NS);
        atomicOr(A.err, kErrTimeout);
    }
    if (warp == 1 && rank == 0 && *abort) {
        // Products already issued may still write tensor memory: free it
        // only after a commit of all of them has arrived.
        if (lane == 0) {
            if constexpr (CG == 2) mma_commit_pair(&mma_drain);
            else mma_commit(&mma_drain);
            volatile int never = 0;
            mbar_wait_bounded(&mma_drain, 0u, &never, DIG_WAIT_NS);
        }
        __syncwarp();
    }
    if constexpr (CG == 2) {
        __syncthreads();
        cluster_sync_all();                              // nothing of the pair is in flight any more
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_free<CG>(tmem, 4 * BN);
    }
}

}  // namespace tdse
