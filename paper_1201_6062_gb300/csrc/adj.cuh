// Per-amplitude update of one reverse stage of the discrete adjoint (used by
// the reverse-stage kernel in adj.cu and by the persistent stepping kernel).
//
// For a step c' = Phi(c; f) built from products k = M(f) x with
// M(f) = -i (diag(E) + f D) and D Hermitian, the cotangents run backwards
// through the same products with M^dagger = +i H:
//   g_x = i (E g_k + f D g_k),   dL/df += Re<g_k, -i D x> = Im<D g_k, x>.
// D g_k is in R/P (the block product of the cotangent input, sys.x).  Writes
// the next product input to sys.x/xq, the running cotangents to sys.acc and
// A.G, and returns this amplitude's Im(conj(D g_k) x).  All FP64.
#pragma once
#include "epi.cuh"
#include "kernels.h"

namespace tdse {

// kCG: read R and P through L2 only (in a persistent launch).
template <class P, bool kCG = false>
__device__ __forceinline__ double adj_amp(const SysDesc &S, long long a, const AdjArgs &A)
{
    // u = D g (D Hermitian in either gauge, so the same products serve the adjoint)
    const double2 u = dx_at<kCG>(S, a);
    const double ur = u.x, ui = u.y;
    const double2 g = S.x[a];
    const double e = S.E[a];
    double f;
    if (A.scheme == 0) {
        const int h = (A.stage == 0) ? 0 : (A.stage == 3 ? 2 : 1);
        f = field_at(S.field, A.sps, A.k, h);
    } else {
        f = field_at(S.field, A.sps, A.k, A.hold ? 1 : 0);
    }
    // g_x = i (E g + f u) = i (p + i q) = (-q, p)
    const double p = e * g.x + f * ur;
    const double q = e * g.y + f * ui;
    const double gxr = -q, gxi = p;
    const double2 xs = A.fwd[a];
    const double dot = ur * xs.y - ui * xs.x;     // Im(conj(u) x)
    const double2 G = A.G[a];
    const double dt = A.dt;
    double2 next;
    if (A.scheme == 0) {
        if (A.stage == 3) {
            S.acc[a] = make_double2(G.x + gxr, G.y + gxi);
            next = make_double2(dt / 3.0 * G.x + dt * gxr, dt / 3.0 * G.y + dt * gxi);
        } else if (A.stage == 2) {
            const double2 gc = S.acc[a];
            S.acc[a] = make_double2(gc.x + gxr, gc.y + gxi);
            next = make_double2(dt / 3.0 * G.x + 0.5 * dt * gxr, dt / 3.0 * G.y + 0.5 * dt * gxi);
        } else if (A.stage == 1) {
            const double2 gc = S.acc[a];
            S.acc[a] = make_double2(gc.x + gxr, gc.y + gxi);
            next = make_double2(dt / 6.0 * G.x + 0.5 * dt * gxr, dt / 6.0 * G.y + 0.5 * dt * gxi);
        } else {
            const double2 gc = S.acc[a];
            const double2 Gn = make_double2(gc.x + gxr, gc.y + gxi);   // dL/dc_k
            A.G[a] = Gn;
            next = make_double2(dt / 6.0 * Gn.x, dt / 6.0 * Gn.y);     // input of step k-1, stage 3
        }
    } else {
        // term m: Gamma_{m-1} = G + g_x; next input (dt/(m-1)) Gamma_{m-1},
        // or at m = 1 the new G and the previous step's (dt/K) G.
        const double2 Gm = make_double2(G.x + gxr, G.y + gxi);
        if (A.stage > 1) {
            const double s = dt / (double)(A.stage - 1);
            next = make_double2(s * Gm.x, s * Gm.y);
        } else {
            A.G[a] = Gm;
            const double s = dt / (double)A.order;
            next = make_double2(s * Gm.x, s * Gm.y);
        }
    }
    S.x[a] = next;
    P::store_xq(S.xq, a, next);
    return dot;
}

// The same in halves (epi.cuh, per component): a thread assembles one
// component of u = D g and updates the other one's cotangents; returns its
// part of Im(conj(u) x).  lmax=15, n=500, FP64, 64 RK4 steps and gradient:
// 36.6 -> 34.6 ms.
enum AdjKind { AK_RK4_LAST, AK_RK4_MID, AK_RK4_FIRST, AK_TAYLOR };      // RK4 stage 3; 2, 1; 0

struct AdjHalf {
    double f, cG, cg;      // field value; the next input's weights of G and g_x (RK4 stage 0: of the new G; Taylor: cg)
    bool to_G;             // Taylor: last reverse term of a step
    const double2 *fwd;
    double2 *G;
};

struct AdjIn {
    EpiPre pre;
    double g, xs, Gt, gt;
};

template <int KIND>
__device__ __forceinline__ AdjIn adj_load(const SysDesc &S, long long a, int own, bool live, const AdjHalf &A)
{
    const int tgt = own ^ 1;
    AdjIn in{};
    if (live) {
        in.pre = epi_pre(S, a);
        in.g = reinterpret_cast<const double *>(S.x)[2 * a + own];
        in.xs = reinterpret_cast<const double *>(A.fwd)[2 * a + tgt];
        if (KIND != AK_RK4_FIRST) in.Gt = reinterpret_cast<const double *>(A.G)[2 * a + tgt];
        if (KIND == AK_RK4_MID || KIND == AK_RK4_FIRST) in.gt = reinterpret_cast<const double *>(S.acc)[2 * a + tgt];
    }
    return in;
}

template <class P, int KIND, bool kCG>
__device__ __forceinline__ double adj_half(const SysDesc &S, long long a, int own, bool live, const AdjIn &in, const AdjHalf &A)
{
    const int tgt = own ^ 1;
    double *x = reinterpret_cast<double *>(S.x) + 2 * a, *acc = reinterpret_cast<double *>(S.acc) + 2 * a;
    double *G = reinterpret_cast<double *>(A.G) + 2 * a;
    double h = 0.0, dot = 0.0;
    if (live) {
        const double u = dx_comp<kCG>(S, a, in.pre, own);
        h = in.pre.e * in.g + A.f * u;
        dot = own ? -u * in.xs : u * in.xs;
    }
    __syncwarp();                          // both components are read before either is written
    if (!live) return 0.0;
    const double gx = own ? -h : h;        // g_x = i h
    double next;
    if constexpr (KIND == AK_RK4_LAST) {
        acc[tgt] = in.Gt + gx;
        next = A.cG * in.Gt + A.cg * gx;
    } else if constexpr (KIND == AK_RK4_MID) {
        acc[tgt] = in.gt + gx;
        next = A.cG * in.Gt + A.cg * gx;
    } else if constexpr (KIND == AK_RK4_FIRST) {
        const double Gn = in.gt + gx;      // dL/dc_k
        G[tgt] = Gn;
        next = A.cG * Gn;                  // input of step k-1, stage 3
    } else {
        const double Gm = in.Gt + gx;
        if (A.to_G) G[tgt] = Gm;
        next = A.cg * Gm;
    }
    x[tgt] = next;
    P::store_xq1(S.xq, a, tgt, next);
    return dot;
}

// As epi_span_kind; the sum of the returned parts goes to *dot.
template <class P, int KIND, bool kCG, class Ready>
__device__ __forceinline__ bool adj_span(const SysDesc &S, long long a0, long long a1, int tid, int nthr, const AdjHalf &A, double *dot, Ready ready)
{
    const int own = tid & 1;
    long long a = a0 + tid / 2;
    AdjIn in = adj_load<KIND>(S, a, own, a < a1, A);
    if (!ready()) return false;
    double t = 0.0;
#pragma unroll 1
    for (long long b = a0; b < a1; b += nthr / 2, a += nthr / 2) {
        const long long an = a + nthr / 2;
        const AdjIn nx = adj_load<KIND>(S, an, own, an < a1, A);
        t += adj_half<P, KIND, kCG>(S, a, own, a < a1, in, A);
        in = nx;
    }
    *dot = t;
    return true;
}

}  // namespace tdse
