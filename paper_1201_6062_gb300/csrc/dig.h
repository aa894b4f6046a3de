// Batched propagation with digit-sliced products on the tensor cores:
// arguments and launchers (dig.cuh, dig.cu).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include "common.cuh"

namespace tdse {

// Digits per operand (8 bits each): 7 for FP32 and float-float, 11 for FP64
// contexts.  The error bounds are in dig.cuh.
constexpr int dig_slices(int prec) { return prec == 0 ? 11 : 7; }

// TMA descriptors: dipole digits [2 (U, U^T)][S][lmax][n][ldb] as (K, row,
// plane) and state digits [S][2B][plane] as (column, pulse plane, digit).
struct DigMaps {
    CUtensorMap U, X;
};

struct DigArgs {
    int n, lmax, B, nb;
    long long N;            // amplitudes per pulse
    const double *E;        // [N]
    const int *eu;          // [2][lmax][n]: exponents of the rows of U_l and U_l^T
    const double *field;    // samples [B][S]; this stage's value is field_at(.., sps, k, h)
    int S, sps, h;
    long long k;
    double2 *c, *x, *acc;   // FP64 states [B][N]
    const int *xmax;        // [lmax+1][2B]: high word of max |x| per (block, plane), this stage's input
    int *xmax_next;         // the same of the next stage's input (atomicMax; cleared before the launch)
    int mode, stage, order; // EPI_RK4 stage 0..3 / EPI_TAYLOR term 1..order
    int gauge;              // 1: D x = i (U x_{l+1} - U^T x_{l-1})
    double step;            // RK4: a_{s+1} dt, last stage dt/6; Taylor: dt/m
    void *scratch;          // dig_scratch_bytes: D x of the tile each CTA has just finished
    int *err;
};

// Tile of the batched product: cg CTAs share 128 cg rows, bn pulse planes.
struct DigTile { int cg, bn; };
DigTile dig_tile(int slices, int n, int lmax, int B);
size_t dig_scratch_bytes(DigTile t);
cudaError_t launch_dig(int slices, DigTile t, const DigMaps &m, const DigArgs &A, cudaStream_t stream);
const void *dig_fn7(int cg, int bn);
const void *dig_fn11(int cg, int bn);

// Dipole blocks in the storage format of `prec` -> digits and row exponents
// (eu must hold 2*lmax*n ints; digits 2*S*lmax*n*ldb bf16, padding zeroed here).
cudaError_t launch_dig_u(int prec, const void *U, long long bstride, int ld, int n, int lmax, int ldb, int *eu,
                         __nv_bfloat16 *digits, cudaStream_t stream);
// High word of max |x| per (block, plane) of the states src [B][N] (xmax cleared by the caller).
cudaError_t launch_dig_max(const double2 *src, int n, int lmax, int B, int *xmax, cudaStream_t stream);
// States src [B][N] -> digits [S][2B][plane], scaled by xmax; clears xmax_next.
cudaError_t launch_dig_x(int slices, const double2 *src, int n, int nb, int lmax, int B, const int *xmax,
                         int *xmax_next, __nv_bfloat16 *digits, cudaStream_t stream);

}  // namespace tdse
