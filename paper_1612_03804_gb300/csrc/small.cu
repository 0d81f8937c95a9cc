// small.cu -- the whole stabilised weight of a configuration in one CTA, for
// lattices of up to 32 sites.
//
// A weight of such a lattice is a chain of some forty dependent steps (slice
// products, Gram matrix, pivot sort, Cholesky, V update per block, then the LU),
// each of a few microseconds of launch latency and almost no work: 4 x 4, 20
// slices 675 us as 42 launches, 104 us here.  All matrices live in shared memory (five
// of 32 x 33 doubles), a step costs a barrier instead of a launch, and the FP64
// pipe is the bound: a warp's instruction holds it for 64 cycles, so elements
// are dealt to threads without gaps (thread e, e + 256, ... of the N x N).
// The method and its error flags are those of stab.cu: X^T <- X^T D E per
// slice; per block pre-pivoted Cholesky-QR (twice in the last block), D, V;
// then M_mid = D_b^-1 U^T + D_s V, LU with partial pivoting, G by substitution.
#include <cuda_runtime.h>
#include <math.h>

#include "chol32.cuh"
#include "internal.h"

namespace sldqmc {

namespace {

constexpr int SM_N = 32, SM_LD = 33, SM_THREADS = 256;
typedef double (*Mat)[SM_LD];

struct SmallArgs {
    const double *E;
    const int8_t *s;
    int N, M, n_wrap, tau0;
    double cu, cd;
    double *ld;
    int *sign;
    double *G;
    double scale;
    int accumulate;
    int *flag;
};

// C = A B (sum over k0(r) <= k < k1(c)) for N x N matrices, C distinct from both;
// with a field slice sl, column c times cu where sl[c] > 0 and cd otherwise.
template <class K0, class K1, class Load>
__device__ __forceinline__ void sm_product(Mat C, int N, K0 k0, K1 k1, Load ab, const int8_t *sl = nullptr, double cu = 1.0,
                                           double cd = 1.0)
{
    for (int e = threadIdx.x; e < N * N; e += SM_THREADS) {
        const int r = e / N, c = e - r * N;
        double a0 = 0.0, a1 = 0.0;  // two chains
        int k = k0(r);
        const int kend = k1(c);
        const double d = sl ? (sl[c] > 0 ? cu : cd) : 1.0;
        for (; k + 1 < kend; k += 2) {
            a0 = ab(a0, r, k, c);
            a1 = ab(a1, r, k + 1, c);
        }
        if (k < kend) a0 = ab(a0, r, k, c);
        C[r][c] = sl ? (a0 + a1) * d : a0 + a1;
    }
    __syncthreads();
}

// W <- R^-T W for the N rows of W, R above the diagonal of F, 1 / R_jj on it.
__device__ __forceinline__ void sm_solve(Mat W, Mat F, int N)
{
    for (int l = 0; l < N; ++l) {
        for (int c = threadIdx.x; c < N; c += SM_THREADS) W[l][c] *= F[l][l];
        __syncthreads();
        for (int e = threadIdx.x; e < (N - 1 - l) * N; e += SM_THREADS) {
            const int q = e / N, r = l + 1 + q, c = e - q * N;
            W[r][c] -= F[l][r] * W[l][c];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(SM_THREADS) k_small_weight(SmallArgs a)
{
    __shared__ double buf[5][SM_N][SM_LD];
    __shared__ double D[SM_N], Dp[SM_N], root[SM_N], piv[SM_N], part[SM_N];
    __shared__ unsigned long long key[SM_N];
    __shared__ int perm[SM_N], s_p;
    __shared__ CholScratch sc;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = a.N;
    const int8_t *s = a.s + (long long)b * a.M * N;
    Mat E = buf[0], U = buf[1], F = buf[2], V = buf[3], W = buf[4];
    for (int e = tid; e < N * N; e += SM_THREADS) {
        const int r = e / N, c = e - r * N;
        E[r][c] = a.E[e];
        U[r][c] = V[r][c] = r == c ? 1.0 : 0.0;
    }
    if (tid < N) D[tid] = 1.0;
    int sgn = 1;  // warp 0
    __syncthreads();
    const auto from0 = [](int) { return 0; };
    const auto toN = [N](int) { return N; };
    int slice = a.tau0;
    for (int m = 0; m < a.M; m += a.n_wrap) {
        const int nb = a.n_wrap < a.M - m ? a.n_wrap : a.M - m;
        const int passes = m + nb >= a.M ? 2 : 1;
        {
            const int8_t *sl = s + (long long)slice * N;
            for (int e = tid; e < N * N; e += SM_THREADS) {
                const int r = e / N, c = e - r * N;
                U[r][c] *= sl[c] > 0 ? a.cu : a.cd;
            }
            __syncthreads();
        }
        for (int j = 0; j < nb; ++j) {
            if (++slice == a.M) slice = 0;
            // the next slice's D with the result, while there is one in the block
            sm_product(F, N, from0, toN, [=](double x, int r, int k, int c) { return fma(U[r][k], E[k][c], x); },
                       j + 1 < nb ? s + (long long)slice * N : nullptr, a.cu, a.cd);
            Mat t = U;
            U = F;
            F = t;
        }
        // Gram matrix of the rows of U = X^T
        sm_product(W, N, from0, toN, [=](double x, int r, int k, int c) { return fma(U[r][k], U[c][k], x); });
        // sort by sqrt(W_jj) D_j, largest first (non-negative doubles order like
        // their bit patterns); the parity of the permutation by its inversions
        if (wid == 0) {
            if (lane < N) key[lane] = (unsigned long long)__double_as_longlong(sqrt(W[lane][lane]) * D[lane]);
            __syncwarp();
            int rank = 0;
            if (lane < N) {
                for (int i = 0; i < N; ++i) rank += key[i] > key[lane] || (key[i] == key[lane] && i < lane);
                perm[rank] = lane;
            }
            int inv = 0;
            for (int i = 0; i < N; ++i) {
                const int ri = __shfl_sync(0xffffffffu, rank, i);
                inv += lane < N && i < lane && ri > rank;
            }
            if (__popc(__ballot_sync(0xffffffffu, inv & 1)) & 1) sgn = -sgn;
            __syncwarp();
            if (lane < N) Dp[lane] = D[perm[lane]];
        }
        __syncthreads();
        // the permuted Gram matrix for the factor, then the permuted rows in its place
        for (int e = tid; e < SM_N * SM_N; e += SM_THREADS) {
            const int r = e >> 5, c = e & 31;
            F[r][c] = r < N && c < N ? (c >= r ? W[perm[r]][perm[c]] : 0.0) : (r == c ? 1.0 : 0.0);
        }
        __syncthreads();
        for (int e = tid; e < N * N; e += SM_THREADS) {
            const int r = e / N, c = e - r * N;
            W[r][c] = U[perm[r]][c];
        }
        chol32(F, root, sc, N, a.flag);
        sm_solve(W, F, N);
        if (tid < N) F[tid][tid] = root[tid];
        __syncthreads();
        if (passes == 2) {
            // W = Q1^T: its Gram matrix into U, factor R2, solve, R = R2 R1
            for (int e = tid; e < SM_N * SM_N; e += SM_THREADS) {
                const int r = e >> 5, c = e & 31;
                double x = r == c ? 1.0 : 0.0;
                if (r < N && c < N) {
                    x = 0.0;
                    if (c >= r)
                        for (int k = 0; k < N; ++k) x = fma(W[r][k], W[c][k], x);
                }
                U[r][c] = x;
            }
            __syncthreads();
            chol32(U, root, sc, N, a.flag);
            sm_solve(W, U, N);
            if (tid < N) U[tid][tid] = root[tid];
            __syncthreads();
            double x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = tid + q * SM_THREADS, r = e / N, c = e - r * N;
                x[q] = 0.0;
                if (e < N * N)
                    for (int k = r; k <= c; ++k) x[q] = fma(U[r][k], F[k][c], x[q]);
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = tid + q * SM_THREADS, r = e / N, c = e - r * N;
                if (e < N * N && c >= r) F[r][c] = x[q];
            }
            __syncthreads();
        }
        if (tid < N) {
            double d = F[tid][tid] * Dp[tid];
            if (!(d > 0.0) || !isfinite(d)) {
                atomicOr(a.flag, FLAG_NUMERICAL);
                d = 1.0;
            }
            D[tid] = d;
            part[tid] = 1.0 / d;
        }
        __syncthreads();
        // V <- (D^-1 R D_p) P^T V: the factor's upper triangle in place, V into U
        for (int e = tid; e < N * N; e += SM_THREADS) {
            const int r = e / N, c = e - r * N;
            if (c >= r) F[r][c] = F[r][c] * Dp[c] * part[r];
        }
        __syncthreads();
        sm_product(U, N, [](int r) { return r; }, toN,
                   [=](double x, int r, int k, int c) { return fma(F[r][k], V[perm[k]][c], x); });
        Mat t = V;  // V <- U, U <- W (= Q^T)
        V = U;
        U = W;
        W = t;
    }
    // M_mid = D_b^-1 U^T + D_s V in W, its right-hand side D_b^-1 U^T in U
    if (tid < N) {
        const double d = D[tid];
        part[tid] = d > 1.0 ? log(d) : 0.0;
        Dp[tid] = d > 1.0 ? 1.0 / d : 1.0;
    }
    __syncthreads();
    for (int e = tid; e < N * N; e += SM_THREADS) {
        const int r = e / N, c = e - r * N;
        const double u = U[r][c] * Dp[r], d = D[r];
        U[r][c] = u;
        W[r][c] = u + (d > 1.0 ? 1.0 : d) * V[r][c];
    }
    __syncthreads();
    const int cols = a.G ? 2 * N : N;
    for (int j = 0; j < N; ++j) {
        if (wid == 0) {
            // the largest |entry| of the column, the lowest row on ties
            unsigned long long bk = lane >= j && lane < N ? (unsigned long long)__double_as_longlong(fabs(W[lane][j])) : 0ull;
            int bi = lane >= j && lane < N ? lane : N;
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (oi < N && (bi >= N || ok > bk || (ok == bk && oi < bi))) {
                    bk = ok;
                    bi = oi;
                }
            }
            if (bi != j) sgn = -sgn;
            double v = W[bi][j];
            if (v == 0.0 || !isfinite(v)) {
                if (lane == 0) atomicOr(a.flag, FLAG_NUMERICAL);
                v = 1.0;
            }
            if (v < 0.0) sgn = -sgn;
            if (lane == 0) {
                s_p = bi;
                piv[j] = v;
                root[j] = 1.0 / v;
            }
        }
        __syncthreads();
        const int p = s_p;
        // rows j and p change places (row j holds U12 from now on)
        for (int c = tid; c < cols; c += SM_THREADS) {
            double *x = c < N ? &W[j][c] : &U[j][c - N], *y = c < N ? &W[p][c] : &U[p][c - N];
            if (p != j) {
                const double t = *x;
                *x = *y;
                *y = t;
            }
            if (c == j) *x = piv[j];
        }
        __syncthreads();
        const double rv = root[j];
        const int nc = cols - 1 - j;
        for (int e = tid; e < (N - 1 - j) * nc; e += SM_THREADS) {
            const int q = e / nc, r = j + 1 + q, c = j + 1 + (e - q * nc);
            const double f = W[r][j] * rv;
            if (c < N) W[r][c] -= f * W[j][c];
            else U[r][c - N] -= f * U[j][c - N];
        }
        __syncthreads();
    }
    if (a.G) {
        // back substitution: X_r = (Y_r - sum_{l > r} U_rl X_l) / U_rr
        for (int r = N - 1; r >= 0; --r) {
            for (int c = tid; c < N; c += SM_THREADS) U[r][c] *= root[r];
            __syncthreads();
            for (int e = tid; e < r * N; e += SM_THREADS) {
                const int q = e / N, c = e - q * N;
                U[q][c] -= W[q][r] * U[r][c];
            }
            __syncthreads();
        }
        for (int e = tid; e < N * N; e += SM_THREADS) {
            const int r = e / N, c = e - r * N;
            a.G[(long long)b * N * N + e] = U[r][c];
        }
    }
    if (wid == 0) {
        double x = lane < N ? part[lane] + log(fabs(piv[lane])) : 0.0;
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) {
            if (a.accumulate) {
                a.ld[b] += a.scale * x;
            } else {
                a.ld[b] = a.scale * x;
                if (a.sign) a.sign[b] = sgn;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// One stabilisation of an item of at most 64 sites in one CTA (FP64 mode): the
// steps of stabilize() in stab.cu with X^T and V in shared memory.  Sorted by
// the rows' norms alone, X^T is permuted in place, its Gram matrix formed in
// that order and factored in two panels of 32 (chol32, substitution, one
// update between them), and V multiplied by D^-1 R D_p.  Nine launches (thirteen
// with the second pass) of the FP64 pipe become one; the pipe stays the bound
// (0.44 M FMAs of one SM for 64 sites, 115 us of each SM whatever the number of
// items up to one per SM), so a step's elements are dealt to threads densely.
// Measured at 8 x 8, 64 items: 192 us; an 8 x 8 sweep of 64 chains (256
// stabilisations of 128 items) 141.6 -> 106.2 ms.
constexpr int ST_N = 64, ST_LD = 65, ST_THREADS = 512;
typedef double (*Mat64)[ST_LD];

struct StabArgs {
    const double *Xt;
    double *Y, *V, *D;
    int *sgn;
    int N, passes;
    int *flag;
};

// Element e of the upper triangle of an N x N matrix, row by row.
__device__ __forceinline__ void st_upper(int e, int N, int &r, int &c)
{
    const float t = (float)(2 * N + 1);
    r = (int)((t - sqrtf(t * t - 8.0f * (float)e)) * 0.5f);
    r = r < 0 ? 0 : r > N - 1 ? N - 1 : r;
    while (r > 0 && r * N - r * (r - 1) / 2 > e) --r;
    while ((r + 1) * N - (r + 1) * r / 2 <= e) ++r;
    c = r + e - (r * N - r * (r - 1) / 2);
}

// F (upper) <- the factor R of Y Y^T, Y <- R^-T Y (rows of Y: N).
__device__ void st_chol(Mat64 Y, Mat64 F, double (*Bk)[33], double *root, CholScratch &sc, int N, int *flag)
{
    const int tid = threadIdx.x;
    for (int e = tid; e < N * (N + 1) / 2; e += ST_THREADS) {
        int r, c;
        st_upper(e, N, r, c);
        double x = 0.0;
        for (int k = 0; k < N; ++k) x = fma(Y[r][k], Y[c][k], x);
        F[r][c] = x;
    }
    __syncthreads();
    for (int k0 = 0; k0 < N; k0 += 32) {
        const int kb = N - k0 < 32 ? N - k0 : 32, j0 = k0 + kb, nW = N - j0, cols = nW + N;
        for (int e = tid; e < 32 * 32; e += ST_THREADS) {
            const int r = e >> 5, c = e & 31;
            Bk[r][c] = r < kb && c < kb ? (c >= r ? F[k0 + r][k0 + c] : 0.0) : (r == c ? 1.0 : 0.0);
        }
        __syncthreads();
        chol32(Bk, root, sc, kb, flag);
        for (int e = tid; e < kb * kb; e += ST_THREADS) {
            const int r = e / kb, c = e - r * kb;
            if (c >= r) F[k0 + r][k0 + c] = c > r ? Bk[r][c] : root[r];
        }
        // rows k0.. of F right of the block and of Y, by substitution (1 / R_ll on Bk's diagonal)
        for (int l = 0; l < kb; ++l) {
            for (int c = tid; c < cols; c += ST_THREADS) {
                double *x = c < nW ? &F[k0 + l][j0 + c] : &Y[k0 + l][c - nW];
                *x *= Bk[l][l];
            }
            __syncthreads();
            for (int e = tid; e < (kb - 1 - l) * cols; e += ST_THREADS) {
                const int q = e / cols, r = l + 1 + q, c = e - q * cols;
                if (c < nW) F[k0 + r][j0 + c] -= Bk[l][r] * F[k0 + l][j0 + c];
                else Y[k0 + r][c - nW] -= Bk[l][r] * Y[k0 + l][c - nW];
            }
            __syncthreads();
        }
        // the rows below lose the panel's share
        for (int e = tid; e < nW * cols; e += ST_THREADS) {
            const int r = e / cols, c = e - r * cols;
            if (c < r) continue;  // below the diagonal of F
            double x = c < nW ? F[j0 + r][j0 + c] : Y[j0 + r][c - nW];
            for (int l = 0; l < kb; ++l) x -= F[k0 + l][j0 + r] * (c < nW ? F[k0 + l][j0 + c] : Y[k0 + l][c - nW]);
            if (c < nW) F[j0 + r][j0 + c] = x;
            else Y[j0 + r][c - nW] = x;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(ST_THREADS) k_stab_block(StabArgs a)
{
    extern __shared__ double st_sh[];
    Mat64 Y = (Mat64)st_sh, F = Y + ST_N, G = F + ST_N;  // G: V, or the second pass's factor
    __shared__ double Bk[32][33];
    __shared__ double D[ST_N], Dp[ST_N], root[32];
    __shared__ unsigned long long key[ST_N];
    __shared__ int perm[ST_N], s_odd;
    __shared__ CholScratch sc;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = a.N, nn = N * N;
    const double *Xt = a.Xt + (long long)b * nn;
    double *V = a.V + (long long)b * nn;
    // the rows of X^T and their norms times D (one warp per row)
    if (tid == 0) s_odd = 0;
    for (int r = wid; r < N; r += ST_THREADS / 32) {
        double x = 0.0;
        for (int c = lane; c < N; c += 32) {
            const double v = Xt[r * N + c];
            x = fma(v, v, x);
        }
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) {
            D[r] = a.D[(long long)b * N + r];
            key[r] = (unsigned long long)__double_as_longlong(sqrt(x) * D[r]);
        }
    }
    __syncthreads();
    // rank of each row, largest first; the parity of the permutation by its inversions
    if (tid < N) {
        int rank = 0;
        for (int i = 0; i < N; ++i) rank += key[i] > key[tid] || (key[i] == key[tid] && i < tid);
        perm[rank] = tid;
    }
    __syncthreads();
    if (tid < N) {
        int inv = 0;
        for (int i = 0; i < tid; ++i) inv += perm[i] > perm[tid];
        if (inv & 1) atomicXor(&s_odd, 1);
        Dp[tid] = D[perm[tid]];
    }
    for (int e = tid; e < nn; e += ST_THREADS) {
        const int r = e / N, c = e - r * N;
        Y[r][c] = Xt[perm[r] * N + c];
    }
    __syncthreads();
    st_chol(Y, F, Bk, root, sc, N, a.flag);
    if (a.passes == 2) {
        st_chol(Y, G, Bk, root, sc, N, a.flag);
        // R = R2 R1 in place of R1
        double x[(ST_N * (ST_N + 1) / 2 + ST_THREADS - 1) / ST_THREADS];
        int q = 0;
        for (int e = tid; e < N * (N + 1) / 2; e += ST_THREADS, ++q) {
            int r, c;
            st_upper(e, N, r, c);
            double s = 0.0;
            for (int k = r; k <= c; ++k) s = fma(G[r][k], F[k][c], s);
            x[q] = s;
        }
        __syncthreads();
        q = 0;
        for (int e = tid; e < N * (N + 1) / 2; e += ST_THREADS, ++q) {
            int r, c;
            st_upper(e, N, r, c);
            F[r][c] = x[q];
        }
        __syncthreads();
    }
    if (tid < N) {
        double d = F[tid][tid] * Dp[tid];
        if (!(d > 0.0) || !isfinite(d)) {
            atomicOr(a.flag, FLAG_NUMERICAL);
            d = 1.0;
        }
        a.D[(long long)b * N + tid] = d;
        D[tid] = 1.0 / d;
    }
    for (int e = tid; e < nn; e += ST_THREADS) {
        const int r = e / N, c = e - r * N;
        a.Y[(long long)b * nn + e] = Y[r][c];
        G[r][c] = V[perm[r] * N + c];
    }
    if (tid == 0 && s_odd) a.sgn[b] = -a.sgn[b];
    __syncthreads();
    // V <- (D^-1 R D_p) P^T V, every entry of V read by now
    for (int e = tid; e < nn; e += ST_THREADS) {
        const int r = e / N, c = e - r * N;
        if (c >= r) F[r][c] = F[r][c] * Dp[c] * D[r];
    }
    __syncthreads();
    for (int e = tid; e < nn; e += ST_THREADS) {
        const int r = e / N, c = e - r * N;
        double x = 0.0;
        for (int k = r; k < N; ++k) x = fma(F[r][k], G[k][c], x);
        V[e] = x;
    }
}

}  // namespace

// A CTA per item does N^3 FMAs per slice on one SM's FP64 pipe, so with several
// items per SM the launches over all items win from 26 sites on.  Measured, 40
// slices, one CTA per item against launches: 4 x 4, 1 / 1024 items 179 / 623 us
// against 635 / 1348; 5 x 5, 1024 items 1813 against 2093; 4 x 7, 128 / 512 items
// 585 / 1576 against 897 / 1247; 8 x 4, 128 / 512 items 670 / 2079 against 916 / 1277.
bool small_fits(const sldqmc_ctx *c)
{
    const double n3 = (double)c->N * c->N * c->N;
    return c->N <= SM_N && c->p.prec == SLDQMC_FP64 && c->kinetic != SLDQMC_KINETIC_SEPARABLE &&
           (c->N <= 25 || n3 * c->plan_cap <= 7.5e6);
}

void small_weight(sldqmc_ctx *c, const int8_t *d_s, int B, double cu, double cd, int tau0, double *d_ld, int *d_sign,
                  double *d_G, double scale, int accumulate)
{
    const SmallArgs a{c->d_E, d_s, c->N, c->M, c->p.n_wrap, tau0, cu, cd, d_ld, d_sign, d_G, scale, accumulate, c->d_flag};
    prof_begin(c, SLDQMC_KC_PANEL_F64, 2.0 * c->N * c->N * c->N * c->M * B, "small_weight");
    k_small_weight<<<B, SM_THREADS, 0, c->st>>>(a);
    prof_end(c);
    c->launches++;
}

// FP64 mode, at most 64 sites.
bool stab_block_fits(const sldqmc_ctx *c) { return c->N <= ST_N && c->p.prec == SLDQMC_FP64; }

constexpr size_t ST_SMEM = sizeof(double) * 3 * ST_N * ST_LD;

void stab_block(sldqmc_ctx *c, const double *Xt, double *Y, int B, int passes)
{
    const StabArgs a{Xt, Y, c->buf[1], c->d_D, c->d_sgn, c->N, passes, c->d_flag};
    const double n3 = (double)c->N * c->N * c->N;
    prof_begin(c, SLDQMC_KC_PANEL_F64, (passes * (1.0 + 4.0 / 3.0) + 1.0) * n3 * B, "stab_block");
    k_stab_block<<<B, ST_THREADS, ST_SMEM, c->st>>>(a);
    prof_end(c);
    c->launches++;
}

void stab_block_set_limits() { cudaFuncSetAttribute(k_stab_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST_SMEM); }

}  // namespace sldqmc
