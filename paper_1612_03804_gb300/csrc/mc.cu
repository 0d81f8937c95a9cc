// mc.cu -- Monte Carlo kernels: the DQMC local update ("Basics of DQMC"),
// the effective-model sweeps and features of the self-learned action
// (Eq. 2, step iii), the bare Ising weight and the cumulative-update
// acceptance (Eq. 4).  Every decision is that of FP64 with explicitly rounded
// operations, so that it matches a plain IEEE evaluation: flips are decided in
// FP32 only where they are clear by more than FP32's error bound.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "internal.h"

namespace sldqmc {

// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32 -> 64-bit products with the Weyl key schedule between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
        const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
        const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    }
}

// Uniform in [0,1) from the top 53 bits of (x1:x0); key = 64-bit seed.
__device__ __forceinline__ double philox_uniform(uint64_t seed, uint32_t a, uint32_t b, uint32_t c,
                                                 uint32_t purpose)
{
    uint32_t x[4] = {a, b, c, purpose};
    philox4x32_10(x, (uint32_t)seed, (uint32_t)(seed >> 32));
    const uint64_t w = ((uint64_t)x[1] << 32) | (uint64_t)x[0];
    return (double)(w >> 11) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ uint32_t philox_word(uint64_t seed, uint32_t a, uint32_t b, uint32_t c,
                                                uint32_t purpose)
{
    uint32_t x[4] = {a, b, c, purpose};
    philox4x32_10(x, (uint32_t)seed, (uint32_t)(seed >> 32));
    return x[0];
}

enum : uint32_t { PURPOSE_LOCAL = 1, PURPOSE_EFF = 2, PURPOSE_DIR = 3, PURPOSE_ACCEPT = 4 };
constexpr double MARGIN = 1e-8;

__device__ __forceinline__ int wrapi(int a, int L)
{
    a %= L;
    return a < 0 ? a + L : a;
}

// Flags any field value outside {-1, +1}.
__global__ void k_check_field(const int8_t *s, long long n, int *flag)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        int v = s[e];
        if (v != 1 && v != -1) atomicOr(flag, FLAG_ARG);
    }
}

// ------------------------------------------------------- bare weight phi
// log phi = dtau J sum_tau sum_<ij> s s + Kt sum_i sum_tau s_{i,tau} s_{i,tau+1}.
// Integer sums per configuration, then one FP64 combination.
__global__ void k_log_bare(const int8_t *s, int Lx, int Ly, int M, double dtauJ, double Kt, double *out,
                           int accumulate)
{
    const int b = blockIdx.x;
    const int N = Lx * Ly;
    const int8_t *sb = s + (long long)b * M * N;
    long long sp = 0, tm = 0;
    for (int v = threadIdx.x; v < M * N; v += blockDim.x) {
        int tau = v / N, i = v % N, x = i % Lx, y = i / Lx;
        int si = sb[v];
        if (Lx > 1) sp += si * sb[tau * N + wrapi(x + 1, Lx) + Lx * y];
        if (Ly > 1) sp += si * sb[tau * N + x + Lx * wrapi(y + 1, Ly)];
        tm += si * sb[((tau + 1) % M) * N + i];
    }
    __shared__ long long a1[32], a2[32];
    for (int o = 16; o > 0; o >>= 1) {
        sp += __shfl_down_sync(0xffffffffu, sp, o);
        tm += __shfl_down_sync(0xffffffffu, tm, o);
    }
    if ((threadIdx.x & 31) == 0) { a1[threadIdx.x >> 5] = sp; a2[threadIdx.x >> 5] = tm; }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t1 = 0, t2 = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { t1 += a1[w]; t2 += a2[w]; }
        double v = dtauJ * (double)t1 + Kt * (double)t2;
        if (accumulate) out[b] += v; else out[b] = v;
    }
}

// --------------------------------------------------------- local update
// Flips every site of slice tau in order i = 0..N-1 for one chain per CTA.
// Gt_f = E^{-1} G(tau) E for flavour f (eta = +1, -1): flipping s_{tau,i}
// gives R_f = 1 + Delta_f (1 - Gt_f[i][i]), Delta_f = exp(-2 eta dtau xi s) - 1;
// the Metropolis ratio is R_+^2 R_-^2 phi'/phi; on acceptance
// Gt_f <- Gt_f - (Delta_f / R_f) Gt_f[:,i] (e_i^T - Gt_f[i,:]).
struct LocalArgs {
    double *Gp, *Gm;   // per chain N x N (stride nn)
    long long nn;
    int8_t *s;         // per chain M x N
    int Lx, Ly, M, tau;
    uint32_t sweep;
    uint64_t seed;
    double dtxi;       // dtau * xi
    double dtauJ, Kt;
    long long *stats;  // per chain: accepted, proposed, margin
};

// The decision of one site: logr = -2 s (dtau J nsp + Kt ntm) + 2 log|R_+| +
// 2 log|R_-|, accepted iff log u < logr, R_f = 1 + Delta_f (1 - G_f[i][i]).  Taken
// in FP32 where it is clear by 1e-5 and by 1e-6 of the terms' magnitudes, those of
// the two bare parts before they cancel; otherwise by the FP64 expression, whose two
// logarithms are some eighty instructions of the FP64 pipe at 64 cycles a warp each.
// FP32 is off by less: 3 2^-24 of each bare part (constant, product, sum), 2^-23 of each
// logarithm and 4 2^-24 for its argument, 3 2^-24 of all terms for their sum.
struct FlipDecision {
    bool acc, margin;
    double R[2];
};

__device__ __forceinline__ FlipDecision flip_decide(const LocalArgs &a, double gp, double gm, const double (*dls)[2], int sold,
                                                    int nsp, int ntm, double lu)
{
    FlipDecision o;
    o.R[0] = __dadd_rn(1.0, __dmul_rn(dls[0][sold > 0], __dadd_rn(1.0, -gp)));
    o.R[1] = __dadd_rn(1.0, __dmul_rn(dls[1][sold > 0], __dadd_rn(1.0, -gm)));
    const float r0 = fabsf((float)o.R[0]), r1 = fabsf((float)o.R[1]), luf = (float)lu;
    const float l0 = 2.0f * logf(r0), l1 = 2.0f * logf(r1);
    const float sj = (float)a.dtauJ * (float)nsp, sk = (float)a.Kt * (float)ntm;
    const float d = -2.0f * (float)sold * (sj + sk) + l0 + l1 - luf;
    o.acc = d > 0.0f;
    o.margin = false;
    if (!(fabsf(d) > 1e-5f + 1e-6f * (2.0f * (fabsf(sj) + fabsf(sk)) + fabsf(l0) + fabsf(l1) + fabsf(luf))) ||
        !(r0 > 1e-30f && r0 < 1e30f) || !(r1 > 1e-30f && r1 < 1e30f)) {
        double logr = __dmul_rn(-2.0 * (double)sold,
                                __dadd_rn(__dmul_rn(a.dtauJ, (double)nsp), __dmul_rn(a.Kt, (double)ntm)));
        logr = __dadd_rn(logr, __dmul_rn(2.0, log(fabs(o.R[0]))));
        logr = __dadd_rn(logr, __dmul_rn(2.0, log(fabs(o.R[1]))));
        o.margin = fabs(logr - lu) <= MARGIN;
        o.acc = lu < logr;
    }
    return o;
}

// Delta_f / R_f of the site decided by lane `hit`, one flavour per lane (warp-wide).
__device__ __forceinline__ void flip_coef(const FlipDecision &d, int sold, int hit, const double (*dls)[2], double *cp,
                                          double *cm)
{
    const int lane = threadIdx.x & 31;
    const double rp = __shfl_sync(0xffffffffu, d.R[0], hit), rm = __shfl_sync(0xffffffffu, d.R[1], hit);
    const int so = __shfl_sync(0xffffffffu, sold, hit);
    if (lane < 2) *(lane ? cm : cp) = dls[lane][so > 0] / (lane ? rm : rp);
}

// Between two accepted flips nothing a decision depends on changes, so warp 0
// decides up to 32 sites at once, one per lane: the lowest accepted one is the
// next flip, the sites before it are rejected, those after it are decided
// again.  SMEM: both Green's functions stay in shared memory (row stride N + 1)
// for the slice; otherwise they are updated in global memory.  An accepted flip
// is 2 N^2 FMAs of this SM's FP64 pipe (2.1 us at N = 64), spread over all
// threads element by element.
// Measured, 8 x 8, 64 chains, a fifth of the flips accepted: 322 us per slice
// when every site was decided in FP64 in turn, 94 now.
template <bool SMEM>
__global__ void __launch_bounds__(512) k_local_flips(LocalArgs a)
{
    const int b = blockIdx.x;
    const int N = a.Lx * a.Ly, tid = threadIdx.x, lane = tid & 31;
    const int ld = SMEM ? N + 1 : N;
    int8_t *s = a.s + (long long)b * a.M * N;
    extern __shared__ double sh[];
    double *col = sh;           // 2N: coef * G[:, i]
    double *row = sh + 2 * N;   // 2N: e_i - G[i, :]
    double *lus = sh + 4 * N;   // N: log u of every site of the slice
    double *gG[2] = {a.Gp + (long long)b * a.nn, a.Gm + (long long)b * a.nn};
    double *G[2] = {SMEM ? sh + 5 * N : gG[0], SMEM ? sh + 5 * N + (long long)N * ld : gG[1]};
    // the slice's spins, and the sums of their neighbours in time
    int8_t *sp = SMEM ? reinterpret_cast<int8_t *>(sh + 5 * N + 2LL * N * ld) : s + (long long)a.tau * N, *nt = sp + N;
    __shared__ double coef[2], dls[2][2];
    __shared__ int s_hit;
    const uint64_t seed = a.seed + ((uint64_t)b << 32);
    const int tau = a.tau, nn = N * N;
    if (SMEM) {
        for (int e = tid; e < 2 * nn; e += blockDim.x) {
            const int f = e >= nn, q = e - f * nn, r = q / N;
            G[f][r * ld + (q - r * N)] = gG[f][q];
        }
        for (int i = tid; i < N; i += blockDim.x) {
            sp[i] = s[tau * N + i];
            nt[i] = (int8_t)(s[wrapi(tau + 1, a.M) * N + i] + s[wrapi(tau - 1, a.M) * N + i]);
        }
    }
    // off the serial chain: the uniforms of all sites, and Delta_f for both field values
    for (int i = tid; i < N; i += blockDim.x)
        lus[i] = log(philox_uniform(seed, (uint32_t)i, (uint32_t)tau, a.sweep, PURPOSE_LOCAL));
    if (tid < 4) {
        const int f = tid >> 1, sp = tid & 1;
        dls[f][sp] = exp(-2.0 * (f == 0 ? 1.0 : -1.0) * a.dtxi * (sp ? 1.0 : -1.0)) - 1.0;
    }
    __syncthreads();
    int q = 0, n_acc = 0, n_mg = 0;  // warp 0: the next site to decide
    for (;;) {
        if (tid < 32) {
            int hit = N;
            while (q < N && hit == N) {
                const int i = q + lane;
                FlipDecision d{false, false, {1.0, 1.0}};
                int sold = 1;
                if (i < N) {
                    sold = sp[i];
                    const int y = i / a.Lx, x = i - y * a.Lx;
                    int nsp = 0;
                    if (a.Lx > 1) nsp += sp[x + 1 < a.Lx ? i + 1 : i + 1 - a.Lx] + sp[x > 0 ? i - 1 : i - 1 + a.Lx];
                    if (a.Ly > 1) nsp += sp[y + 1 < a.Ly ? i + a.Lx : x] + sp[y > 0 ? i - a.Lx : i - a.Lx + N];
                    const int ntm = SMEM ? nt[i] : s[wrapi(tau + 1, a.M) * N + i] + s[wrapi(tau - 1, a.M) * N + i];
                    d = flip_decide(a, G[0][(long long)i * ld + i], G[1][(long long)i * ld + i], dls, sold, nsp, ntm, lus[i]);
                }
                const unsigned m = __ballot_sync(0xffffffffu, d.acc);
                const int first = m ? __ffs(m) - 1 : 32;  // lanes up to it are decided
                n_mg += __popc(__ballot_sync(0xffffffffu, d.margin && lane <= first));
                if (m) {
                    hit = q + first;
                    flip_coef(d, sold, first, dls, coef, coef + 1);
                    if (lane == first) sp[i] = (int8_t)(-sold);
                    __syncwarp();
                    n_acc++;
                }
                q += first + 1 < 32 ? first + 1 : 32;
            }
            if (lane == 0) s_hit = hit;
        }
        __syncthreads();
        const int i = s_hit;
        if (i >= N) break;
        for (int e = tid; e < 2 * N; e += blockDim.x) {
            const int f = e >= N, k = e - f * N;
            col[e] = coef[f] * G[f][(long long)k * ld + i];
            row[e] = (k == i ? 1.0 : 0.0) - G[f][(long long)i * ld + k];
        }
        __syncthreads();
        for (int e = tid; e < 2 * nn; e += blockDim.x) {
            const int f = e >= nn, p = e - f * nn, r = p / N, k = p - r * N;
            G[f][(long long)r * ld + k] -= col[f * N + r] * row[f * N + k];
        }
        __syncthreads();
    }
    if (SMEM) {
        for (int e = tid; e < 2 * nn; e += blockDim.x) {
            const int f = e >= nn, p = e - f * nn, r = p / N;
            gG[f][p] = G[f][r * ld + (p - r * N)];
        }
        for (int i = tid; i < N; i += blockDim.x) s[tau * N + i] = sp[i];
    }
    if (tid == 0) {
        a.stats[b * 4 + 0] += n_acc;
        a.stats[b * 4 + 1] += N;
        a.stats[b * 4 + 2] += n_mg;
    }
}

// ------------------------------------------------- delayed (rank-k) update
// The same sequence of flips, decisions and Green's functions with the
// Sherman-Morrison updates delayed: within a block of k <= 32 sites of slice
// tau the current Green's function of flavour f is
//   Gt_f = G0_f - U_f V_f,   U_f = [u_0 .. u_{n-1}] (N x n),  V_f = [v_0; ..; v_{n-1}] (n x N),
// one column/row pair per accepted flip so far.  A site needs only
// Gt_f[i][i] = G0_f[i][i] - U_f[i,:] V_f[:,i] (n terms); an accepted flip
// at i appends u_n = (Delta_f / R_f) Gt_f[:, i] and v_n = e_i^T - Gt_f[i, :],
// each formed from G0 and the n earlier pairs (2 N n multiply-adds instead
// of the N^2 of an immediate update).  After the block the pending rank-k
// correction G0 -= U V is applied by one batched GEMM over every chain
// (unused pairs are zero), so the N^2 work per accepted flip runs as a GEMM
// on all SMs instead of as rank-1 passes on one SM per chain.
// U: per chain N x 32 (row stride 32), V: per chain 32 x N; flavour f of
// chain b at U + (f * cap + b) * 32 N.
struct DelayArgs {
    LocalArgs l;
    double *U, *V;
    int cap;
    int i0, ns;   // sites i0 .. i0 + ns - 1 of slice tau (ns <= 32)
};

__global__ void __launch_bounds__(512) k_local_flips_delayed(DelayArgs d)
{
    const LocalArgs &a = d.l;
    const int b = blockIdx.x;
    const int N = a.Lx * a.Ly;
    const double *G[2] = {a.Gp + (long long)b * a.nn, a.Gm + (long long)b * a.nn};
    double *U[2], *V[2];
    for (int f = 0; f < 2; ++f) {
        U[f] = d.U + ((long long)f * d.cap + b) * 32 * N;
        V[f] = d.V + ((long long)f * d.cap + b) * 32 * N;
    }
    int8_t *s = a.s + (long long)b * a.M * N;
    __shared__ double ui[2][32], vi[2][32];  // U[i, :n] and V[:n, i] of the current site
    __shared__ double coef[2], dls[2][2], lus[32];
    __shared__ int accept;
    const uint64_t seed = a.seed + ((uint64_t)b << 32);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    long long n_acc = 0, n_mg = 0;
    const int tau = a.tau;
    int n = 0;  // pending pairs
    // off the serial chain: the block's uniforms, and Delta_f for both field values
    if (tid < d.ns)
        lus[tid] = log(philox_uniform(seed, (uint32_t)(d.i0 + tid), (uint32_t)tau, a.sweep, PURPOSE_LOCAL));
    if (tid >= 32 && tid < 36) {
        const int f = (tid - 32) >> 1, sp = tid & 1;
        const double eta = f == 0 ? 1.0 : -1.0;
        dls[f][sp] = exp(-2.0 * eta * a.dtxi * (sp ? 1.0 : -1.0)) - 1.0;
    }
    __syncthreads();
    for (int q = 0; q < d.ns; ++q) {
        const int i = d.i0 + q;
        if (wid == 0) {
            // U[i, j] and V[j, i] for j < n, and the current diagonals
            double dg[2];
            for (int f = 0; f < 2; ++f) {
                const double uu = lane < n ? U[f][(long long)i * 32 + lane] : 0.0;
                const double vv = lane < n ? V[f][(long long)lane * N + i] : 0.0;
                ui[f][lane] = uu;
                vi[f][lane] = vv;
                double p = uu * vv;
                for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
                dg[f] = G[f][(long long)i * N + i] - p;
            }
            if (lane == 0) {
                const int sold = s[tau * N + i];
                const int x = i % a.Lx, y = i / a.Lx;
                int nsp = 0;
                if (a.Lx > 1) nsp += s[tau * N + wrapi(x + 1, a.Lx) + a.Lx * y] + s[tau * N + wrapi(x - 1, a.Lx) + a.Lx * y];
                if (a.Ly > 1) nsp += s[tau * N + x + a.Lx * wrapi(y + 1, a.Ly)] + s[tau * N + x + a.Lx * wrapi(y - 1, a.Ly)];
                const int ntm = s[wrapi(tau + 1, a.M) * N + i] + s[wrapi(tau - 1, a.M) * N + i];
                double logr = __dmul_rn(-2.0 * (double)sold,
                                        __dadd_rn(__dmul_rn(a.dtauJ, (double)nsp), __dmul_rn(a.Kt, (double)ntm)));
                double R[2], Dl[2];
                for (int f = 0; f < 2; ++f) {
                    Dl[f] = dls[f][sold > 0];
                    R[f] = __dadd_rn(1.0, __dmul_rn(Dl[f], __dadd_rn(1.0, -dg[f])));
                    logr = __dadd_rn(logr, __dmul_rn(2.0, log(fabs(R[f]))));
                }
                const double lu = lus[q];
                if (fabs(logr - lu) <= MARGIN) n_mg++;
                const int acc = lu < logr;
                accept = acc;
                if (acc) {
                    coef[0] = Dl[0] / R[0];
                    coef[1] = Dl[1] / R[1];
                    s[tau * N + i] = (int8_t)(-sold);
                    n_acc++;
                }
            }
        }
        __syncthreads();
        if (accept) {
            // u_n = coef (G0[:, i] - U[:, :n] V[:n, i]),  v_n = e_i - (G0[i, :] - U[i, :n] V[:n, :])
            for (int e = tid; e < 2 * N; e += blockDim.x) {
                const int f = e >= N, r = e - f * N;
                double c = G[f][(long long)r * N + i];
                const double *ur = U[f] + (long long)r * 32;
                double w = G[f][(long long)i * N + r];
                for (int j = 0; j < n; ++j) {
                    c -= ur[j] * vi[f][j];
                    w -= ui[f][j] * V[f][(long long)j * N + r];
                }
                U[f][(long long)r * 32 + n] = coef[f] * c;
                V[f][(long long)n * N + r] = (r == i ? 1.0 : 0.0) - w;
            }
            ++n;
        }
        __syncthreads();
    }
    // unused pairs are zero for the batched correction
    for (int f = 0; f < 2; ++f) {
        for (long long e = tid; e < (long long)N * (32 - n); e += blockDim.x) {
            const int r = (int)(e / (32 - n)), j = n + (int)(e % (32 - n));
            U[f][(long long)r * 32 + j] = 0.0;
        }
        for (long long e = tid; e < (long long)(32 - n) * N; e += blockDim.x) V[f][(long long)n * N + e] = 0.0;
    }
    if (tid == 0) {
        a.stats[b * 4 + 0] += n_acc;
        a.stats[b * 4 + 1] += d.ns;
        a.stats[b * 4 + 2] += n_mg;
    }
}

// The decisions of one block on lattices of 128 sites and more.  They depend
// on the Green's functions only through the 32 x 32 blocks of rows and columns
// i0..i0+ns-1, so the block's serial chain runs on those alone, in shared
// memory, and what the accepted flips do to the other rows and columns is
// formed afterwards on all SMs (k_flip_pairs and a rank-32 product,
// oz_gram.cu).  One CTA per chain.  Warp 0 decides all sites still to come at
// once (see k_local_flips); then all warps subtract the accepted one's pair from
// the rows below.  Bound by the latency of dependent FP64 operations per
// accepted flip.
// A block of 32 sites of 8 chains at N = 576: 25 us, and 23 us for the pairs;
// 247 us when every pair was formed for all rows and columns inside the chain,
// and 651 us per 32 sites of 16 chains at N = 256 with immediate updates on one
// SM per chain (2 N^2 FMAs of the FP64 pipe per accepted flip and flavour).
__global__ void __launch_bounds__(256) k_flip_block(LocalArgs a, FlipPairs *out, int i0, int ns)
{
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = a.Lx * a.Ly, tau = a.tau;
    __shared__ double g[2][32][33], us[2][32][33], vs[2][32][33];
    __shared__ double coef[2][32], dls[2][2], lus[32];
    __shared__ int s_q, sites[32];
    const uint64_t seed = a.seed + ((uint64_t)b << 32);
    int8_t *s = a.s + (long long)b * a.M * N;
    FlipPairs &o = out[b];
    for (int e = tid; e < 2 * 32 * 32; e += 256) {
        const int f = e >> 10, r = (e >> 5) & 31, c = e & 31;
        const double *G = (f ? a.Gm : a.Gp) + (long long)b * a.nn;
        g[f][r][c] = (r < ns && c < ns) ? G[(long long)(i0 + r) * N + i0 + c] : 0.0;
    }
    // warp 0, lane j: spin and neighbour sums of site i0 + j
    int sold = 1, nsp = 0, ntm = 0, x = 0, y = 0;
    if (wid == 0) {
        if (lane < ns) {
            const int i = i0 + lane;
            x = i % a.Lx;
            y = i / a.Lx;
            sold = s[tau * N + i];
            if (a.Lx > 1) nsp += s[tau * N + wrapi(x + 1, a.Lx) + a.Lx * y] + s[tau * N + wrapi(x - 1, a.Lx) + a.Lx * y];
            if (a.Ly > 1) nsp += s[tau * N + x + a.Lx * wrapi(y + 1, a.Ly)] + s[tau * N + x + a.Lx * wrapi(y - 1, a.Ly)];
            ntm = s[wrapi(tau + 1, a.M) * N + i] + s[wrapi(tau - 1, a.M) * N + i];
            lus[lane] = log(philox_uniform(seed, (uint32_t)i, (uint32_t)tau, a.sweep, PURPOSE_LOCAL));
        }
    } else if (wid == 1 && lane < 4) {
        const int f = lane >> 1, sp = lane & 1;
        dls[f][sp] = exp(-2.0 * (f == 0 ? 1.0 : -1.0) * a.dtxi * (sp ? 1.0 : -1.0)) - 1.0;
    }
    __syncthreads();
    int n_mg = 0, q = 0, n = 0;
    for (;;) {
        if (wid == 0) {
            // all sites from q on at once: the lowest accepted one is the next flip
            FlipDecision d{false, false, {1.0, 1.0}};
            if (lane >= q && lane < ns) d = flip_decide(a, g[0][lane][lane], g[1][lane][lane], dls, sold, nsp, ntm, lus[lane]);
            const unsigned m = __ballot_sync(0xffffffffu, d.acc);
            const int hit = m ? __ffs(m) - 1 : ns;
            n_mg += __popc(__ballot_sync(0xffffffffu, d.margin && lane <= hit));
            if (m) flip_coef(d, sold, hit, dls, &coef[0][n], &coef[1][n]);
            if (lane == 0) {
                s_q = hit;
                if (hit < ns) sites[n] = hit;
            }
            if (hit < ns) {
                // the flipped spin, and the sums of its neighbours in the block
                const int so = __shfl_sync(0xffffffffu, sold, hit);
                const int xq = __shfl_sync(0xffffffffu, x, hit), yq = __shfl_sync(0xffffffffu, y, hit);
                int mult = 0;
                if (a.Lx > 1 && y == yq) mult += (wrapi(x + 1, a.Lx) == xq) + (wrapi(x - 1, a.Lx) == xq);
                if (a.Ly > 1 && x == xq) mult += (wrapi(y + 1, a.Ly) == yq) + (wrapi(y - 1, a.Ly) == yq);
                nsp -= 2 * so * mult;
                if (lane == hit) sold = -so;
                q = hit + 1;
            }
        }
        __syncthreads();
        const int hit = s_q;
        if (hit >= ns) break;
        if (tid < 64) {
            const int f = wid;
            us[f][n][lane] = coef[f][n] * g[f][lane][hit];
            vs[f][n][lane] = (lane == hit ? 1.0 : 0.0) - g[f][hit][lane];
        }
        __syncthreads();
        {
            const int f = wid >> 2;
            const double v = vs[f][n][lane];
            for (int r = hit + 1 + (wid & 3); r < ns; r += 4) g[f][r][lane] -= us[f][n][r] * v;
        }
        ++n;
        __syncthreads();
    }
    for (int e = tid; e < 2 * 32 * 32; e += 256) {
        const int f = e >> 10, r = (e >> 5) & 31, c = e & 31;
        // L[r][c] = u_c at accepted site r, X[r][c] = v_r at accepted site c
        o.L[f][r][c] = c < r && r < n ? us[f][c][sites[r]] : 0.0;
        o.X[f][r][c] = r < c && c < n ? vs[f][r][sites[c]] : 0.0;
    }
    if (tid < 64) o.coef[wid][lane] = lane < n ? coef[wid][lane] : 0.0;
    if (tid < 32) o.site[tid] = tid < n ? i0 + sites[tid] : 0;
    if (wid == 0) {
        if (lane < ns) s[tau * N + i0 + lane] = (int8_t)sold;
        if (lane == 0) {
            o.n = n;
            a.stats[b * 4 + 0] += n;
            a.stats[b * 4 + 1] += ns;
            a.stats[b * 4 + 2] += n_mg;
        }
    }
}

void launch_flip_block(sldqmc_ctx *c, double *Gp, double *Gm, FlipPairs *out, int8_t *d_s, int B, int tau, int i0, int ns,
                       uint32_t sweep, uint64_t seed, long long *stats)
{
    LocalArgs a;
    a.Gp = Gp; a.Gm = Gm; a.nn = c->nn; a.s = d_s;
    a.Lx = c->p.Lx; a.Ly = c->p.Ly; a.M = c->M; a.tau = tau; a.sweep = sweep; a.seed = seed;
    a.dtxi = c->p.dtau * c->p.xi; a.dtauJ = c->dtauJ; a.Kt = c->Ktau; a.stats = stats;
    prof_begin(c, SLDQMC_KC_LOCAL, 0.0, "flip_block");
    k_flip_block<<<B, 256, 0, c->st>>>(a, out, i0, ns);
    prof_end(c);
    c->launches++;
}

void launch_local_flips_delayed(sldqmc_ctx *c, double *Gp, double *Gm, double *U, double *V, int8_t *d_s, int B,
                                int tau, int i0, int ns, uint32_t sweep, uint64_t seed, long long *stats)
{
    DelayArgs d;
    LocalArgs &a = d.l;
    a.Gp = Gp; a.Gm = Gm; a.nn = c->nn; a.s = d_s;
    a.Lx = c->p.Lx; a.Ly = c->p.Ly; a.M = c->M; a.tau = tau; a.sweep = sweep; a.seed = seed;
    a.dtxi = c->p.dtau * c->p.xi; a.dtauJ = c->dtauJ; a.Kt = c->Ktau; a.stats = stats;
    d.U = U; d.V = V; d.cap = c->cap; d.i0 = i0; d.ns = ns;
    prof_begin(c, SLDQMC_KC_LOCAL, 0.0, "local_flips_delayed");
    k_local_flips_delayed<<<B, 512, 0, c->st>>>(d);
    prof_end(c);
    c->launches++;
}

// Gt <- D_tau Gt D_tau^{-1} applied after the two wrap GEMMs is fused into
// the GEMM epilogues; the drift check compares a wrapped Gt with a fresh one.
__global__ void k_drift(const double *Gw, const double *Gf, long long nn, long long *stats, int B2)
{
    const int b = blockIdx.y;
    double m = 0.0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn;
         e += (long long)gridDim.x * blockDim.x)
        m = fmax(m, fabs(Gw[(long long)b * nn + e] - Gf[(long long)b * nn + e]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0) {
        // non-negative doubles order like their bit patterns
        const int chain = b % B2;
        atomicMax(reinterpret_cast<unsigned long long *>(&stats[chain * 4 + 3]),
                  (unsigned long long)__double_as_longlong(m));
    }
}

// ------------------------------------------------------ effective model
// The model of one context travels with each launch as a kernel parameter
// (constant bank): class c has noff[c] offset triples (dx, dy, dtau), listed
// class after class in off, and coupling J[c].
// nb: the same offsets reduced to 0 <= dx < Lx, 0 <= dy < Ly, 0 <= dtau < M, each
// followed by its opposite, so that a neighbour is found by additions and one
// conditional subtraction per direction; Jn: the FP32 coupling of each of
// these neighbours (0 where the neighbour is the site itself).
struct EffNeighbour {
    short dx, dy;
    int dt;
};

struct EffModel {
    int n_class, n_nb;
    int noff[32];
    int off[64 * 3];
    double J[32];
    EffNeighbour nb[128];
    float Jn[128];
    float Jabs;  // sum of |Jn|
};

static EffModel eff_model_of(const sldqmc_ctx *c)
{
    EffModel m;
    memset(&m, 0, sizeof(m));
    m.n_class = c->n_class;
    memcpy(m.noff, c->h_n_off, sizeof(m.noff));
    memcpy(m.off, c->h_offsets, sizeof(m.off));
    memcpy(m.J, c->h_J, sizeof(m.J));
    auto wrap = [](int a, int L) { a %= L; return a < 0 ? a + L : a; };
    int q = 0;
    for (int k = 0; k < m.n_class; ++k)
        for (int t = 0; t < m.noff[k]; ++t, ++q)
            for (int sg = 1; sg >= -1; sg -= 2) {
                const int *o = m.off + 3 * q;
                EffNeighbour &n = m.nb[m.n_nb];
                n.dx = (short)wrap(sg * (o[0] % c->p.Lx), c->p.Lx);
                n.dy = (short)wrap(sg * (o[1] % c->p.Ly), c->p.Ly);
                n.dt = wrap(sg * (o[2] % c->M), c->M);
                const bool self = n.dx == 0 && n.dy == 0 && n.dt == 0;
                m.Jn[m.n_nb] = self ? 0.0f : (float)m.J[k];
                m.Jabs += fabsf(m.Jn[m.n_nb]);
                ++m.n_nb;
            }
    return m;
}

// Site (tau, y, x) moved by a reduced offset.
__device__ __forceinline__ int moved_site(int tau, int y, int x, int N, int Lx, int Ly, int M, int dt, int dy, int dx)
{
    x += dx;
    y += dy;
    tau += dt;
    x -= x >= Lx ? Lx : 0;
    y -= y >= Ly ? Ly : 0;
    tau -= tau >= M ? M : 0;
    return tau * N + y * Lx + x;
}

// The neighbours as the kernels read them.  A colour of a lattice in shared memory
// is bound by the integer work of its neighbour loop, not by its loads: with the
// offsets multiplied into units of sites beforehand (dx, dy Lx, dtau N), one 16-byte
// load an entry and the wrap an unsigned minimum, a sweep of 24 x 24 x 20 with 16
// classes takes 99 us instead of 143 (8-byte offsets, the coupling loaded apart,
// comparisons and two products an entry).  A table of 16-bit neighbour numbers, read
// from L2, took 187.
struct __align__(16) EffEntry {
    uint32_t dx, dy, dt;
    float J;
};

// One Metropolis decision of H_eff: log acceptance a = ((2 beta) * sum_c J_c
// n_c) * s with n_c the integer neighbour sums (self-pairs excluded),
// accumulated in class order, accepted iff log u < a.  The G lanes of a group
// (G a power of two, all lanes of the warp present) share the site's
// neighbours and take the decision in FP32 where it is clear: the sum of at most
// 128 couplings is off by less than 132 2^-24 of the sum of their magnitudes,
// the logarithm by less than 2^-23 of itself and 2^-23, and the margin is more
// than each of these.  Otherwise the group's first lane takes the FP64 decision,
// a hundred operations of the FP64 pipe at 64 cycles a warp: a margin ten times
// wider, met in every second colour, made a sweep of 24 x 24 x 20 with 16 classes
// 158 us instead of 143 (one CTA, the neighbours as 8-byte offsets).  Returns whether
// this lane flipped the site.
struct EffSite {
    const EffModel &em;
    int N, Lx, Ly, M;
    double twob;
    uint64_t key;
    uint32_t step;
};

// J times the spin s (+-1), by the sign bit.
__device__ __forceinline__ float eff_signed(float J, int8_t s)
{
    return __uint_as_float(__float_as_uint(J) ^ ((uint32_t)(int)s & 0x80000000u));
}

// a - L if that is not negative, a otherwise, given a < 2 L and a - L modulo 2^32.
__device__ __forceinline__ uint32_t eff_wrap(uint32_t a, uint32_t a_minus_L) { return min(a, a_minus_L); }

// What a decision needs that does not depend on the spins: the site's coordinates,
// its random word and the word's logarithm.
struct EffDraw {
    int v, tau, y, x;
    uint64_t w;
    float lf;
};

__device__ __forceinline__ EffDraw eff_draw(const EffSite &e, int v, int sw)
{
    EffDraw d;
    d.v = v;
    d.tau = v / e.N;
    const int i = v - d.tau * e.N;
    d.y = i / e.Lx;
    d.x = i - d.y * e.Lx;
    uint32_t r[4] = {(uint32_t)i, (uint32_t)d.tau, e.step, PURPOSE_EFF | ((uint32_t)sw << 8)};
    philox4x32_10(r, (uint32_t)e.key, (uint32_t)(e.key >> 32));
    d.w = (((uint64_t)r[1] << 32) | (uint64_t)r[0]) >> 11;
    d.lf = logf(__ull2float_rn(d.w) * (1.0f / 9007199254740992.0f));
    return d;
}

__device__ __forceinline__ bool eff_site(const EffSite &e, int8_t *s, const EffEntry *nb, const EffDraw &d, bool active, int G,
                                         long long &mg)
{
    const int sub = threadIdx.x & (G - 1);
    const int v = d.v, tau = d.tau, y = d.y, x = d.x;
    float sum = 0.0f;
    if (active) {
        const uint32_t x0 = x, yL = y * e.Lx, tN = (uint32_t)tau * e.N, xm = x0 - e.Lx, ym = yL - e.N,
                       tm = tN - (uint32_t)e.N * e.M;
#pragma unroll 5
        for (int k = sub; k < e.em.n_nb; k += G) {
            const EffEntry n = nb[k];
            sum += eff_signed(n.J, s[eff_wrap(tN + n.dt, tm + n.dt) + eff_wrap(yL + n.dy, ym + n.dy) + eff_wrap(x0 + n.dx, xm + n.dx)]);
        }
    }
    for (int o = G >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (!active || sub) return false;
    const int sv = s[v];
    const uint64_t w = d.w;
    const float af = (float)e.twob * sum * (float)sv, lf = d.lf;
    const float df = af - lf;
    bool acc = df > 0.0f;
    if (!(fabsf(df) > 1e-6f + 1e-5f * (fabsf((float)e.twob) * e.em.Jabs) + 1e-6f * fabsf(lf)) || w == 0) {
        double sm = 0.0;
        int k = 0;
        for (int c = 0; c < e.em.n_class; ++c) {
            int n = 0;
            for (int t = 0; t < 2 * e.em.noff[c]; ++t, ++k) {
                const EffNeighbour &o = e.em.nb[k];
                const int u = moved_site(tau, y, x, e.N, e.Lx, e.Ly, e.M, o.dt, o.dy, o.dx);
                if (u != v) n += s[u];
            }
            sm = __dadd_rn(sm, __dmul_rn(e.em.J[c], (double)n));
        }
        const double av = __dmul_rn(__dmul_rn(e.twob, sm), (double)sv);
        const double lu = log((double)w * (1.0 / 9007199254740992.0));
        if (fabs(av - lu) <= MARGIN) mg++;
        acc = lu < av;
    }
    if (acc) s[v] = (int8_t)(-sv);
    return acc;
}

__device__ __forceinline__ void eff_counts(long long acc, long long mg, int b, long long *n_accept, long long *n_margin)
{
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_down_sync(0xffffffffu, acc, o);
        mg += __shfl_down_sync(0xffffffffu, mg, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (n_accept && acc) atomicAdd((unsigned long long *)&n_accept[b], (unsigned long long)acc);
        if (n_margin && mg) atomicAdd((unsigned long long *)&n_margin[b], (unsigned long long)mg);
    }
}

__device__ __forceinline__ void eff_load_nb(const EffModel &em, EffEntry *nb, int Lx, int N)
{
    for (int k = threadIdx.x; k < em.n_nb; k += blockDim.x)
        nb[k] = EffEntry{(uint32_t)em.nb[k].dx, (uint32_t)em.nb[k].dy * Lx, (uint32_t)em.nb[k].dt * N, em.Jn[k]};
    __syncthreads();
}

// Copies n bytes, 16 at a time where both sides allow it.
__device__ __forceinline__ void eff_copy(int8_t *dst, const int8_t *src, int n)
{
    int v = threadIdx.x;
    if (!((((uintptr_t)dst) | (uintptr_t)src) & 15)) {
        for (int q = threadIdx.x; q < n / 16; q += blockDim.x) ((int4 *)dst)[q] = ((const int4 *)src)[q];
        v += n / 16 * 16;
    }
    for (; v < n; v += blockDim.x) dst[v] = src[v];
}

// n_sweeps colour-ordered sweeps of one chain per cluster of CTAs (or one CTA), its
// spins in each CTA's shared memory, G lanes per site.  A CTA takes its share of a
// colour's sites and writes a flipped spin into every CTA's copy; one cluster
// barrier per colour, and the next sites are drawn before the wait for it.  A colour's
// time in one CTA is its neighbour loop and its decisions, on one SM of 152: dividing
// them took 24 x 24 x 20 with 16 classes and 16 chains from 4.1 to 2.1 us a colour.
template <bool CLUSTER>
__global__ void __launch_bounds__(1024) k_eff_sweeps(int8_t *s_all, int Lx, int Ly, int M, double beta,
                                                     const __grid_constant__ EffModel em, const int *col_start,
                                                     const int *col_sites, int n_colors, int n_sweeps,
                                                     uint64_t seed, uint32_t step, int dir_fixed, int G,
                                                     long long *n_accept, long long *n_margin,
                                                     const uint32_t *d_step)
{
    if (d_step) step = *d_step;  // graph replays read the step from device memory
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = CLUSTER ? cl.num_blocks() : 1, rank = CLUSTER ? cl.block_rank() : 0;
    const int b = blockIdx.x / C;
    const int N = Lx * Ly;
    const int V = N * M;
    extern __shared__ __align__(16) int8_t s[];
    __shared__ EffEntry nb[128];
    int8_t *gs = s_all + (long long)b * V;
    const uint64_t key = seed + ((uint64_t)b << 32);
    eff_copy(s, gs, V);
    eff_load_nb(em, nb, Lx, N);
    if (CLUSTER) cl.sync();  // every copy is loaded: spins may be written into it
    int dir = dir_fixed;
    if (dir < 0) dir = (int)(philox_word(key, 0, 0, step, PURPOSE_DIR) & 1u);
    long long acc = 0, mg = 0;
    const EffSite e{em, N, Lx, Ly, M, 2.0 * beta, key, step};
    const int per = blockDim.x / G;
    int sw = 0, cc = 0, q = 0, q1 = 0;
    auto colour = [&] {  // this CTA's share of the cc-th colour
        const int col = dir ? (n_colors - 1 - cc) : cc;
        const int c0 = col_start[col], c1 = col_start[col + 1], share = (c1 - c0 + C - 1) / C;
        q = c0 + rank * share;
        q1 = min(q + share, c1);
    };
    EffDraw d{};
    auto draw = [&] {
        const int k = q + threadIdx.x / G;
        if (k < q1) d = eff_draw(e, col_sites[k], sw);
    };
    if (n_sweeps > 0) {
        colour();
        if (CLUSTER) draw();
        for (;;) {
            if (!CLUSTER) draw();
            const bool flip = eff_site(e, s, nb, d, q + (int)threadIdx.x / G < q1, G, mg);
            acc += flip;
            if (CLUSTER && flip) {
                const int8_t sv = s[d.v];
                for (int r = 0; r < C; ++r)
                    if (r != rank) *cl.map_shared_rank(s + d.v, r) = sv;
            }
            q += per;
            const bool last = q >= q1;
            if (last) {
                if (CLUSTER) cl.barrier_arrive();
                if (++cc == n_colors) {
                    cc = 0;
                    ++sw;
                }
                if (sw < n_sweeps) colour();
            }
            if (CLUSTER && sw < n_sweeps) draw();
            if (last) {
                if (CLUSTER)
                    cl.barrier_wait();
                else
                    __syncthreads();
            }
            if (sw == n_sweeps) break;
        }
    }
    if (!CLUSTER) {
        eff_copy(gs, s, V);
    } else {
        const int part = (V / C + 15) / 16 * 16, v0 = min(rank * part, V), v1 = rank == C - 1 ? V : min(v0 + part, V);
        eff_copy(gs + v0, s + v0, v1 - v0);
    }
    eff_counts(acc, mg, b, n_accept, n_margin);
}

// The cc-th colour of sweep sw (in each chain's own direction) of every chain
// on all SMs, the spins in global memory (sites of one colour do not interact).
__global__ void __launch_bounds__(256) k_eff_colour(int8_t *s_all, int Lx, int Ly, int M, double beta,
                                                    const __grid_constant__ EffModel em, const int *col_start,
                                                    const int *col_sites, int n_colors, int sw, int cc, uint64_t seed,
                                                    uint32_t step, int dir_fixed, long long *n_accept,
                                                    long long *n_margin, const uint32_t *d_step)
{
    if (d_step) step = *d_step;
    const int b = blockIdx.y;
    const int N = Lx * Ly;
    __shared__ EffEntry nb[128];
    eff_load_nb(em, nb, Lx, N);
    const uint64_t key = seed + ((uint64_t)b << 32);
    int dir = dir_fixed;
    if (dir < 0) dir = (int)(philox_word(key, 0, 0, step, PURPOSE_DIR) & 1u);
    const int col = dir ? (n_colors - 1 - cc) : cc;
    long long acc = 0, mg = 0;
    const EffSite e{em, N, Lx, Ly, M, 2.0 * beta, key, step};
    const int q0 = col_start[col], n = col_start[col + 1] - q0;
    for (int k0 = blockIdx.x * blockDim.x; k0 < n; k0 += gridDim.x * blockDim.x) {
        const int k = k0 + threadIdx.x;
        acc += eff_site(e, s_all + (long long)b * N * M, nb, eff_draw(e, k < n ? col_sites[q0 + k] : 0, sw), k < n, 1, mg);
    }
    eff_counts(acc, mg, b, n_accept, n_margin);
}

// f_c(C) = sum_x sum_{o in c} s_x s_{x+o} (self-pairs give 1), one CTA per
// configuration and class; out[b*n_class + c].
__global__ void __launch_bounds__(512) k_features(const int8_t *s_all, int Lx, int Ly, int M,
                                                  const __grid_constant__ EffModel em, long long *out)
{
    const int b = blockIdx.x, c = blockIdx.y;
    const int N = Lx * Ly, V = N * M;
    const int8_t *s = s_all + (long long)b * V;
    __shared__ long long red[16];
    int k0 = 0;
    for (int k = 0; k < c; ++k) k0 += 2 * em.noff[k];
    long long acc = 0;
    for (int v = threadIdx.x; v < V; v += blockDim.x) {
        const int tau = v / N, i = v - tau * N, y = i / Lx, x = i - y * Lx;
        int n = 0;
        for (int k = k0; k < k0 + 2 * em.noff[c]; k += 2)
            n += s[moved_site(tau, y, x, N, Lx, Ly, M, em.nb[k].dt, em.nb[k].dy, em.nb[k].dx)];
        acc += s[v] * n;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        out[(long long)b * em.n_class + c] = t;
    }
}

// Eq. 4 in log form, per chain:
//   log r = [lw1 - lw0] - [-beta sum_c J_c (f1_c - f0_c)],  accept iff log u < log r.
__global__ void k_cumulative_accept(const double *lw1, double *lw0, const long long *f0, const long long *f1,
                                    const __grid_constant__ EffModel em, double beta, uint64_t seed, uint32_t step, int B,
                                    int *accepted, int *accept_count, double *log_r, long long *margin,
                                    const uint32_t *d_step)
{
    if (d_step) step = *d_step;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int n_class = em.n_class;
    double acc = 0.0;
    for (int c = 0; c < n_class; ++c)
        acc = __dadd_rn(acc, __dmul_rn(em.J[c], (double)(f1[(long long)b * n_class + c] - f0[(long long)b * n_class + c])));
    const double dlweff = __dmul_rn(-beta, acc);
    const double lr = __dadd_rn(__dadd_rn(lw1[b], -lw0[b]), -dlweff);
    const uint64_t key = seed + ((uint64_t)b << 32);
    const double u = philox_uniform(key, 0, 0, step, PURPOSE_ACCEPT);
    const double lu = log(u);
    if (margin && fabs(lr - lu) <= MARGIN) margin[b]++;
    const int a = lu < lr;
    accepted[b] = a;
    if (a) lw0[b] = lw1[b];
    if (accept_count) accept_count[b] += a;
    if (log_r) log_r[b] = lr;
}

// s[b] <- s'[b] where accepted[b]
__global__ void k_commit(int8_t *s, const int8_t *sp, const int *accepted, long long V)
{
    const int b = blockIdx.y;
    if (!accepted[b]) return;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < V;
         e += (long long)gridDim.x * blockDim.x)
        s[(long long)b * V + e] = sp[(long long)b * V + e];
}

// ------------------------------------------------------------ launchers
static inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

void launch_check_field(sldqmc_ctx *c, const int8_t *d_s, long long n)
{
    int g = cdiv(n, 256);
    if (g > 1024) g = 1024;
    if (g < 1) g = 1;
    k_check_field<<<g, 256, 0, c->st>>>(d_s, n, c->d_flag);
    c->launches++;
}

void launch_log_bare(sldqmc_ctx *c, const int8_t *d_s, int B, double *out, int accumulate)
{
    k_log_bare<<<B, 256, 0, c->st>>>(d_s, c->p.Lx, c->p.Ly, c->M, c->dtauJ, c->Ktau, out, accumulate);
    c->launches++;
}

// Both Green's functions and the vectors of a slice within 200 KB (N <= 111).
static size_t resident_bytes(int N) { return sizeof(double) * ((size_t)5 * N + (size_t)2 * N * (N + 1)) + 2 * (size_t)N; }
bool local_flips_resident(int N) { return resident_bytes(N) <= 200 * 1024; }

void launch_local_flips(sldqmc_ctx *c, double *Gp, double *Gm, int8_t *d_s, int B, int tau,
                        uint32_t sweep, uint64_t seed, long long *stats)
{
    LocalArgs a;
    a.Gp = Gp; a.Gm = Gm; a.nn = c->nn; a.s = d_s;
    a.Lx = c->p.Lx; a.Ly = c->p.Ly; a.M = c->M; a.tau = tau; a.sweep = sweep; a.seed = seed;
    a.dtxi = c->p.dtau * c->p.xi; a.dtauJ = c->dtauJ; a.Kt = c->Ktau; a.stats = stats;
    size_t sh = sizeof(double) * 5 * (size_t)c->N;
    int nt = c->N * c->N >= 512 ? 512 : 256;
    prof_begin(c, SLDQMC_KC_LOCAL, 0.0, "local_flips");
    if (local_flips_resident(c->N)) k_local_flips<true><<<B, nt, resident_bytes(c->N), c->st>>>(a);
    else k_local_flips<false><<<B, nt, sh, c->st>>>(a);
    prof_end(c);
    c->launches++;
}

void launch_drift(sldqmc_ctx *c, const double *Gw, const double *Gf, int B2x, int B, long long *stats)
{
    dim3 g(cdiv(c->nn, 256) < 32 ? cdiv(c->nn, 256) : 32, B2x);
    k_drift<<<g, 256, 0, c->st>>>(Gw, Gf, c->nn, stats, B);
    c->launches++;
}

static const int EFF_SMEM = 200 * 1024;  // the largest chain held in shared memory

static cudaLaunchConfig_t eff_config(const sldqmc_ctx *c, int B, int C, int threads, long long V)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(B * C);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = (size_t)V;
    cfg.stream = c->st;
    return cfg;
}

static cudaLaunchAttribute eff_attribute(int C)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    return at;
}

// CTAs per chain: as many (up to the portable 8) as leave each EFF_READS neighbour
// reads of a colour, while all chains run at once.  A colour ends with a cluster
// barrier and with flips on their way to the other copies, which costs about as much
// as that: 12 x 12 x 20 with 4 classes (4000 reads a colour) takes 14.8 us a sweep in
// one CTA and 19.5 in two; with 16 classes (7200) 62 in one, 47 in two.
static const int EFF_READS = 3072;
static int eff_cluster(const sldqmc_ctx *c, int B, long long cs, int n_nb, long long V)
{
    if (V > EFF_SMEM) return 1;
    for (int C = 8; C > 1; --C) {
        if ((long long)B * C > c->num_sms || cs * n_nb < EFF_READS * C) continue;
        cudaLaunchConfig_t cfg = eff_config(c, B, C, 1024, V);
        cudaLaunchAttribute at = eff_attribute(C);
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_eff_sweeps<true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (n >= B) return C;
    }
    return 1;
}

// A chain's spins stay in the shared memory of one CTA or of a cluster's CTAs while
// its colours are small or the chains fill the GPU; otherwise each colour is one
// launch over all SMs.  In units of the time of one pass of 1024 sites (about 1.5
// us, a launch three of them): passes per colour in the chain's CTAs, times the waves
// of chains, against a launch and the passes spread over all SMs; a cluster's barrier
// counts as one more (48 x 48 x 80, 4 chains: 71 us a sweep spread, 79 in clusters).
// Measured per sweep: 100 x 100 x 100, one chain, 4 classes 15.2 ms (one CTA, spins in
// global memory) -> 89 us (spread); 64 x 64 x 100, 16 classes 12.2 ms -> 218 us (spread);
// 32 x 32 x 160, 16 classes, 4 chains 5.0 ms -> 283 us (spread) -> 182 (clusters of 8);
// 16 x 16 x 160, 4 classes, 16 chains 648 -> 99 us (one CTA) -> 36 (clusters); 24 x 24 x
// 20, 16 classes, 16 chains 490 -> 99 us (one CTA) -> 50 (clusters).
void launch_eff_sweeps(sldqmc_ctx *c, int8_t *d_s, int B, int n_sweeps, uint64_t seed, uint32_t step,
                       int dir, long long *n_accept, long long *n_margin)
{
    const long long V = (long long)c->N * c->M;
    const EffModel em = eff_model_of(c);
    const long long cs = (V + c->n_colors - 1) / c->n_colors;  // sites per colour
    const int C = eff_cluster(c, B, cs, em.n_nb, V);  // CTAs per chain
    const long long share = (cs + C - 1) / C;
    const long long in_cta = ((share + 1023) / 1024) * (((long long)B * C + c->num_sms - 1) / c->num_sms);
    const long long spread = 3 + (cs * B + 1024LL * c->num_sms - 1) / (1024LL * c->num_sms);
    prof_begin(c, SLDQMC_KC_EFF, 0.0, "eff_sweeps");
    if (V <= EFF_SMEM && (C == 1 ? in_cta <= spread : in_cta + 1 < spread)) {
        // Lanes per site, while a colour leaves them idle; at most four in a cluster,
        // where more would only add warps (24 x 24 x 20, 16 classes: 54, 50 and 58 us a
        // sweep with up to 2, 4 and 8).
        int G = 1;
        const long long most = C > 1 ? (c->max_color + C - 1) / C : cs;  // a CTA's sites
        while (G < (C > 1 ? 4 : 8) && 2 * G * most <= 1024) G *= 2;
        const int threads = C > 1 && most * G < 1024 ? (int)((most * G + 31) / 32 * 32) : 1024;
        cudaLaunchConfig_t cfg = eff_config(c, B, C, threads, V);
        cudaLaunchAttribute at = eff_attribute(C);
        cfg.attrs = &at;
        cfg.numAttrs = C > 1;
        cudaLaunchKernelEx(&cfg, C > 1 ? k_eff_sweeps<true> : k_eff_sweeps<false>, d_s, c->p.Lx, c->p.Ly, c->M, c->p.beta, em,
                           (const int *)c->d_col_start, (const int *)c->d_col_sites, c->n_colors, n_sweeps, seed, step, dir,
                           G, n_accept, n_margin, (const uint32_t *)c->step_dev);
        c->launches++;
    } else {
        const int bx = cdiv(cs, 256) < 1024 ? cdiv(cs, 256) : 1024;
        for (int b0 = 0; b0 < B; b0 += 32768) {  // grid y limit
            const int nb = B - b0 < 32768 ? B - b0 : 32768;
            for (int sw = 0; sw < n_sweeps; ++sw)
                for (int cc = 0; cc < c->n_colors; ++cc) {
                    k_eff_colour<<<dim3(bx, nb), 256, 0, c->st>>>(
                        d_s + V * b0, c->p.Lx, c->p.Ly, c->M, c->p.beta, em, c->d_col_start, c->d_col_sites, c->n_colors,
                        sw, cc, seed + ((uint64_t)b0 << 32), step, dir, n_accept ? n_accept + b0 : nullptr,
                        n_margin ? n_margin + b0 : nullptr, c->step_dev);
                    c->launches++;
                }
        }
    }
    prof_end(c);
}

void launch_features(sldqmc_ctx *c, const int8_t *d_s, int B, long long *out)
{
    k_features<<<dim3(B, c->n_class), 512, 0, c->st>>>(d_s, c->p.Lx, c->p.Ly, c->M, eff_model_of(c), out);
    c->launches++;
}

void launch_cumulative_accept(sldqmc_ctx *c, const double *lw1, double *lw0, const long long *f0,
                              const long long *f1, uint64_t seed, uint32_t step, int B, int *accepted,
                              int *accept_count, double *log_r, long long *margin)
{
    k_cumulative_accept<<<cdiv(B, 128), 128, 0, c->st>>>(lw1, lw0, f0, f1, eff_model_of(c), c->p.beta, seed,
                                                        step, B, accepted, accept_count, log_r, margin,
                                                        c->step_dev);
    c->launches++;
}

void launch_commit(sldqmc_ctx *c, int8_t *d_s, const int8_t *d_sp, const int *accepted, int B)
{
    const long long V = (long long)c->N * c->M;
    dim3 g(cdiv(V, 256) < 64 ? cdiv(V, 256) : 64, B);
    k_commit<<<g, 256, 0, c->st>>>(d_s, d_sp, accepted, V);
    c->launches++;
}

__global__ void k_step_advance(uint32_t *d_step) { *d_step += 1u; }

void launch_step_advance(sldqmc_ctx *c, uint32_t *d_step)
{
    k_step_advance<<<1, 1, 0, c->st>>>(d_step);
    c->launches++;
}

void set_eff_smem_limits()
{
    cudaFuncSetAttribute(k_eff_sweeps<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, EFF_SMEM);
    cudaFuncSetAttribute(k_eff_sweeps<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, EFF_SMEM);
    cudaFuncSetAttribute(k_local_flips<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_local_flips<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

}  // namespace sldqmc
