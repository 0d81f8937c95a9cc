// chol32.cuh -- Cholesky factor and inverse of one 32 x 32 block in shared
// memory, the serial part of every Cholesky-QR panel.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "internal.h"

namespace sldqmc {

// 1/sqrt(d) of a pivot: the FP32 value y (relative error 2^-22) and one step of
// third order, y + y e (1/2 + 3/8 e) with e = 1 - d y^2, whose remainder is below
// 2^-66: five FP64 operations, four of them in sequence.  Conversions and
// comparisons would take the FP64 pipe as well, so they are made on the bits:
// one integer comparison tells a positive d of binary exponent -100 .. 99, and
// for those d truncated to FP32 and y as a double are shifts.  Otherwise the
// library's function; a pivot that is not positive and finite raises the
// flag and counts as 1 (d is set to it).
__device__ __forceinline__ double chol_rsqrt(double &d, bool real, int *flag)
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    if (hi - (923u << 20) >= (200u << 20)) {
        if (!(d > 0.0) || !isfinite(d)) {
            if (real) atomicOr(flag, FLAG_NUMERICAL);
            d = 1.0;
        }
        return rsqrt(d);
    }
    const float f = rsqrtf(__uint_as_float(((hi << 3) | (lo >> 29)) - (896u << 23)));
    const double y = __longlong_as_double(((long long)__float_as_uint(f) << 29) + (896ll << 52));
    const double e = fma(-(d * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// The row X[j][lane] = v with its pivot in lane j is final once scaled by y =
// 1/sqrt(pivot); lane j then holds y, the diagonal of the inverse.
__device__ __forceinline__ void chol32_finalise(double (*X)[33], double *root, int j, int lane, double v, int kb, int *flag)
{
    double d = __shfl_sync(0xffffffffu, v, j);
    const double y = chol_rsqrt(d, lane == 0 && j < kb, flag);
    X[j][lane] = lane == j ? y : v * y;
    if (lane == 0) root[j] = d;
}

// W = R^T R of the block W (X[r][c], c >= r; X[r][c] = 0 below the diagonal;
// rows and columns kb..31 the identity, which stay as they are), by all warps
// of the CTA.  On return X holds R above the diagonal and T = R^-T on and below
// it, root[j] = R_jj (j < kb).
// Right-looking, with R's and T's rows (T by forward substitution of R^T T =
// 1) in one array: at step j row r > j loses X[j][r] times row j in the lanes
// c >= r (R) and c <= j (T), one FMA per row.  Warp 0 updates row j + 1 and
// finalises it while the others update the rows below, so a step costs one
// barrier, and the chain of pivots is what bounds the kernel: a warp's FP64
// instruction holds its sub-partition's pipe for 64 cycles however few lanes
// work, and a step has seven in sequence or nearly.
// All threads of the CTA call it between barriers; blockDim.x a multiple of 32.
__device__ __forceinline__ void chol32(double (*X)[33], double *root, int kb, int *flag)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (wid == 0) chol32_finalise(X, root, 0, lane, X[0][lane], kb, flag);
    __syncthreads();
    for (int j = 0; j < kb - 1; ++j) {
        if (wid == 0) {
            const int r = j + 1;
            double v = X[r][lane];
            const double xj = X[j][lane], xr = X[j][r];
            if (lane >= r || lane <= j) v -= xr * xj;
            chol32_finalise(X, root, r, lane, v, kb, flag);
        } else {
            const double xj = X[j][lane];
            for (int r = j + 1 + wid; r < kb; r += nw - 1)
                if (lane >= r || lane <= j) X[r][lane] -= X[j][r] * xj;
        }
        __syncthreads();
    }
    // R_jj = d y
    if (threadIdx.x < kb) root[threadIdx.x] *= X[threadIdx.x][threadIdx.x];
    __syncthreads();
}

}  // namespace sldqmc
