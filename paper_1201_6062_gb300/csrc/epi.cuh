// Update of one stage (paper Sec. 4: H x = E x + f D x with D x assembled from
// the row sums R and the column-partial slots P; App. B: the RK4 stage and
// Taylor term combinations), all in FP64.  Used by the update kernel that
// follows each block product and by the persistent stepping kernel.
#pragma once
#include "kernels.h"

namespace tdse {

// Inputs of one amplitude that no kernel of a call writes (its energy and
// the slot range of its column partials): the epilogue kernel reads them
// before it waits for the block product.
struct EpiPre {
    double e;
    int m, i, b0, b1;
};

__device__ __forceinline__ EpiPre epi_pre(const SysDesc &S, long long a)
{
    EpiPre p;
    p.m = (int)((unsigned)a / (unsigned)S.n);                // (a < 2^31)
    p.i = (int)a - p.m * S.n;
    p.e = S.E[a];
    p.b0 = p.m >= 1 ? S.sb[p.m - 1] : 0;
    p.b1 = p.m >= 1 ? S.sb[p.m] : 0;
    return p;
}

// The update in halves: a thread assembles one component (own) of D x, and
// with it h = E x + f D x, whose k = -i h is the other component's derivative,
// so it updates that one (tgt) and no values are exchanged.  Twice the threads,
// half the dependent FP64 instructions of each; KIND is a template parameter
// because the compiler evaluates short alternatives of a uniform branch side by
// side and every FP64 instruction takes 64 cycles of its scheduler.  Bound by the
// latency of those instructions and of the loads: a stage of the persistent
// kernel 21.0 -> 18.7 us float-float and 47.6 -> 44.7 us FP64 at lmax=15, n=500,
// 27.2 -> 23.9 us FP64 at lmax=7, n=301 (from one thread an amplitude).
enum EpiKind { EK_RK4_FIRST, EK_RK4_MID, EK_RK4_LAST, EK_TAYLOR, EK_HX, EK_MIHX };

struct EpiHalf {
    double f, s;           // field value; RK4: a_{s+1} dt (last stage dt/6), Taylor: dt/m
    bool first, last;      // Taylor: first and last term
    double2 *st_x, *st_c;  // as EpiArgs
};

// One component of D x at (m, i): row sum plus column partials in slot order,
// read eight at a time (velocity gauge D x = i (R - sum P)).  kCG: through L2
// only (in a persistent launch other CTAs wrote R and P moments ago).
template <bool kCG>
__device__ __forceinline__ double dx_comp(const SysDesc &S, long long a, const EpiPre &pre, int own)
{
    const int src = S.gauge ? own ^ 1 : own;
    const double *R = reinterpret_cast<const double *>(S.R) + 2 * a + src;
    const double *Pp = reinterpret_cast<const double *>(S.P) + 2 * ((long long)pre.b0 * S.n + pre.i) + src;
    const long long step = 2LL * S.n;
    auto ld = [](const double *p) { return kCG ? __ldcg(p) : *p; };
    const double r = pre.m < S.lmax ? ld(R) : 0.0;
    double p = 0.0;
    for (int s = pre.b0; s < pre.b1; s += 8, Pp += 8 * step) {
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = s + j < pre.b1 ? ld(Pp + j * step) : 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (s + j < pre.b1) p += v[j];
    }
    if (S.gauge == 0) return r + p;
    return own == 0 ? -(r - p) : r - p;
}

// What an update reads besides D x (nothing that other threads' updates of
// the same stage write, but for the other component's lane).
struct EpiIn {
    EpiPre pre;
    double xo, ct, at;     // own component of the stage input; the other one's state and accumulator
};

template <int KIND>
__device__ __forceinline__ EpiIn epi_load(const SysDesc &S, long long a, int own, bool live, const EpiHalf &A)
{
    const int tgt = own ^ 1;
    const double *c = reinterpret_cast<const double *>(S.c) + 2 * a, *x = reinterpret_cast<const double *>(S.x) + 2 * a;
    constexpr bool kRk = KIND == EK_RK4_FIRST || KIND == EK_RK4_MID || KIND == EK_RK4_LAST;
    const bool from_c = KIND == EK_RK4_FIRST || (KIND == EK_TAYLOR && A.first);
    EpiIn in{};
    if (live) {
        in.pre = epi_pre(S, a);
        in.xo = from_c ? c[own] : x[own];
        if (kRk || from_c) in.ct = c[tgt];
        if (KIND == EK_RK4_MID || KIND == EK_RK4_LAST || (KIND == EK_TAYLOR && !A.first))
            in.at = reinterpret_cast<const double *>(S.acc)[2 * a + tgt];
    }
    return in;
}

// Called by whole warps, the two components of an amplitude on adjacent lanes;
// live: whether this lane has one.
template <class P, int KIND, bool kCG>
__device__ __forceinline__ void epi_half(const SysDesc &S, long long a, int own, bool live, const EpiIn &in, const EpiHalf &A)
{
    const int tgt = own ^ 1;
    double *c = reinterpret_cast<double *>(S.c) + 2 * a, *x = reinterpret_cast<double *>(S.x) + 2 * a;
    double *acc = reinterpret_cast<double *>(S.acc) + 2 * a;
    const double h = live ? in.pre.e * in.xo + A.f * dx_comp<kCG>(S, a, in.pre, own) : 0.0;
    __syncwarp();                          // both components are read before either is written
    if (!live) return;
    if constexpr (KIND == EK_HX) {
        acc[own] = h;
        return;
    }
    const double k = own ? h : -h;         // (k_re, k_im) = (h_im, -h_re)
    if constexpr (KIND == EK_MIHX) {
        acc[tgt] = k;
    } else if constexpr (KIND == EK_RK4_FIRST || KIND == EK_RK4_MID) {
        acc[tgt] = KIND == EK_RK4_FIRST ? k : in.at + 2.0 * k;
        const double xn = in.ct + A.s * k;
        x[tgt] = xn;
        P::store_xq1(S.xq, a, tgt, xn);
        if (A.st_x) reinterpret_cast<double *>(A.st_x)[2 * a + tgt] = xn;
    } else if constexpr (KIND == EK_RK4_LAST) {
        const double cn = in.ct + A.s * (in.at + k);
        c[tgt] = cn;
        P::store_xq1(S.xq, a, tgt, cn);
        if (A.st_c) reinterpret_cast<double *>(A.st_c)[2 * a + tgt] = cn;
    } else {
        const double T = A.s * k;
        const double sum = (A.first ? in.ct : in.at) + T;
        const double xn = A.last ? sum : T;
        if (A.last) {
            c[tgt] = sum;
        } else {
            acc[tgt] = sum;
            x[tgt] = T;
        }
        P::store_xq1(S.xq, a, tgt, xn);
        double2 *st = A.last ? A.st_c : A.st_x;
        if (st) reinterpret_cast<double *>(st)[2 * a + tgt] = xn;
    }
}

// The amplitudes [a0, a1) of S by the nthr threads of whole warps (tid: this
// thread's number), two threads each.  ready() is called once the first
// amplitudes' own data are requested, before any of D x is read (false: give
// up); later ones' are requested an iteration ahead.
template <class P, int KIND, bool kCG, class Ready>
__device__ __forceinline__ bool epi_span_kind(const SysDesc &S, long long a0, long long a1, int tid, int nthr, const EpiHalf &A, Ready ready)
{
    const int own = tid & 1;
    long long a = a0 + tid / 2;
    EpiIn in = epi_load<KIND>(S, a, own, a < a1, A);
    if (!ready()) return false;
#pragma unroll 1
    for (long long b = a0; b < a1; b += nthr / 2, a += nthr / 2) {
        const long long an = a + nthr / 2;
        const EpiIn nx = epi_load<KIND>(S, an, own, an < a1, A);
        epi_half<P, KIND, kCG>(S, a, own, a < a1, in, A);
        in = nx;
    }
    return true;
}

template <class P, bool kCG, class Ready>
__device__ __forceinline__ bool epi_span(const SysDesc &S, long long a0, long long a1, int tid, int nthr, int kind, const EpiHalf &A, Ready ready)
{
    switch (kind) {
    case EK_RK4_FIRST: return epi_span_kind<P, EK_RK4_FIRST, kCG>(S, a0, a1, tid, nthr, A, ready);
    case EK_RK4_MID: return epi_span_kind<P, EK_RK4_MID, kCG>(S, a0, a1, tid, nthr, A, ready);
    case EK_RK4_LAST: return epi_span_kind<P, EK_RK4_LAST, kCG>(S, a0, a1, tid, nthr, A, ready);
    }
    return epi_span_kind<P, EK_TAYLOR, kCG>(S, a0, a1, tid, nthr, A, ready);
}

}  // namespace tdse
