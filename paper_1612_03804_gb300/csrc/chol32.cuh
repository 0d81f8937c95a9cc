// chol32.cuh -- Cholesky factor and inverse of one 32 x 32 block in shared
// memory, the serial part of every Cholesky-QR panel.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "internal.h"

namespace sldqmc {

// Scratch of chol32.
struct CholScratch {
    double mult[2][32];  // row j over its pivot, for the step j's updates; at the end 1 / sqrt of the pivots
    double pivot[32];
};

// 1/d of a pivot by integers (an FP64 operation of a warp takes some 100 cycles
// of the chain of pivots, an integer one 5).  With d = M 2^k, M of 53 bits, and
// the FP32 reciprocal R0 2^-24 of M 2^-52 rounded to FP32, the remainder e = 1 - M
// R0 2^-76 is below 3 2^-24, so its integer is the low 64 bits of -M R0, and 1/d =
// R0 (1 + e + e^2) 2^.. (e^3 is below 2^-67), within 1.3 quarters of a unit in the last
// place.  So the nearest double is those quarters rounded down, q, or the next, and the
// remainder 2^105 - q M (its integer again the low 64 bits) says which: 1/d correctly
// rounded, as the division gives it (no reciprocal lies half way).
// u: the bits of d (positive, biased exponent 523 .. 1522); rb: those of the FP32
// reciprocal, which may be off by one unit in the last place, also to just below
// 1/2 or above 1, where it counts as 1/2 or 1.
// EXACT = false: the quarters rounded to the nearest unit, within 0.9 units.
template <bool EXACT = true>
__host__ __device__ __forceinline__ long long chol_reciprocal_bits(long long u, uint32_t rb)
{
    const unsigned long long M = ((unsigned long long)u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const uint32_t R0 = rb >= 0x3F800000u ? 1u << 24 : rb <= 0x3F000000u ? 1u << 23 : (rb & 0x7FFFFFu) | 0x800000u;
    const long long e = -(long long)(M * (unsigned long long)R0);  // units of 2^-76
    const long long s = e >> 40;
    const long long R = ((long long)R0 << 31) + (((e >> 15) * (long long)R0 + (1ll << 29)) >> 30) +
                        ((s * s * (long long)R0 + (1ll << 40)) >> 41);  // units of 2^-55
    if (!EXACT) return ((2044 - (u >> 52)) << 52) + ((R + 2) >> 2);
    const long long q = R >> 2;
    const long long rem = -(long long)(M * (unsigned long long)q);  // |rem| < 1.4 M
    return ((2044 - (u >> 52)) << 52) + q + (2 * rem > (long long)M);
}

// The bits of M 2^-52 rounded to FP32, in [1, 2].
__host__ __device__ __forceinline__ uint32_t chol_seed_bits(long long u)
{
    return 0x3F800000u + (uint32_t)((((unsigned long long)u & 0xFFFFFFFFFFFFFull) + (1ull << 28)) >> 29);
}

// A pivot that is not positive and finite raises the flag and counts as 1 (d is
// set to it); binary exponents beyond -500 .. 499 take the division.
template <bool EXACT = true>
__device__ __forceinline__ double chol_reciprocal(double &d, bool real, int *flag)
{
    const long long u = __double_as_longlong(d);
    const int ef = (int)(u >> 52);  // negative for negative d
    if ((unsigned)(ef - 523) >= 1000u) {
        if (!(d > 0.0) || !isfinite(d)) {
            if (real) atomicOr(flag, FLAG_NUMERICAL);
            d = 1.0;
        }
        return 1.0 / d;
    }
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(chol_seed_bits(u))));
    return __longlong_as_double(chol_reciprocal_bits<EXACT>(u, __float_as_uint(r)));
}

// W = R^T R of the block W (X[r][c], c >= r; X[r][c] = 0 below the diagonal;
// rows and columns kb..31 the identity, which stay as they are), by all warps
// of the CTA.  On return X holds R above the diagonal and T = R^-T on and below
// it, root[j] = R_jj (j < kb).
// Right-looking without square roots (W = L D L^T), L^-1 formed with it (by
// forward substitution) in the same array: at step j row r > j loses
// X[j][r] / d_j times row j in the lanes c >= r (D L^T) and c <= j (L^-1, whose
// diagonal is 1), one FMA per row; the rows are scaled by 1 / sqrt(d_j) at the
// end, all pivots at once (R_jj is sqrt(d_j), not d_j / sqrt(d_j), which rounds twice;
// warp 0 has the roots, warp 1 their reciprocals, each on a pipe of its own).
// Warp 0 updates row j + 1, divides it by its pivot and leaves it to the next
// step while the others update the rows below, so a step costs one barrier and
// two FP64 operations in sequence (seven when the rows were scaled by 1 / sqrt as
// they went; a panel's preparation 20.4 -> 18.7 us by events, 32 x 32, 4 items).
// EXACT: reciprocals and roots correctly rounded, as the FP64 mode has them.  The
// mixed modes' factors never were (their panels took the library's rsqrt, now
// reciprocals within 0.9 units and R_jj = d_j / sqrt(d_j)), and a bit changed there
// moves a BF16 log|det| by 2e-8 through the products that follow (50 x 48, M = 181),
// so they keep that form (18.7 us a panel's preparation, 19.0 with EXACT).
// All threads of the CTA call it between barriers; blockDim.x a multiple of 32
// (at least 64).
template <bool EXACT = true>
__device__ __forceinline__ void chol32(double (*X)[33], double *root, CholScratch &sc, int kb, int *flag)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double m = 0.0;  // warp 0: the current row over its pivot
    for (int j = -1; j < kb - 1; ++j) {
        if (wid == 0) {
            const int r = j + 1;
            double v = X[r][lane];
            if (j >= 0) {
                const double mr = __shfl_sync(0xffffffffu, m, r), xj = X[j][lane];
                if (lane >= r || lane <= j) v -= mr * xj;
            }
            double d = __shfl_sync(0xffffffffu, v, r);
            const double inv = chol_reciprocal<EXACT>(d, lane == 0, flag);
            m = v * inv;
            X[r][lane] = lane == r ? 1.0 : v;
            sc.mult[r & 1][lane] = m;
            if (lane == 0) sc.pivot[r] = d;
        } else if (j >= 0) {
            const double xj = X[j][lane];
            for (int r = j + 1 + wid; r < kb; r += nw - 1)
                if (lane >= r || lane <= j) X[r][lane] -= sc.mult[j & 1][r] * xj;
        }
        __syncthreads();
    }
    if (EXACT && wid == 0 && lane < kb) root[lane] = sqrt(sc.pivot[lane]);
    if (wid == 1 && lane < kb) {
        const double d = sc.pivot[lane], y = rsqrt(d);
        sc.mult[0][lane] = y;
        if (!EXACT) root[lane] = d * y;
    }
    __syncthreads();
    for (int r = wid; r < kb; r += nw) X[r][lane] *= sc.mult[0][r];
    __syncthreads();
}

}  // namespace sldqmc
