// internal.h -- shared declarations of the sldqmc CUDA library (not part of
// the public C ABI).  All kernels are written for sm_103a (GB300).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

struct sldqmc_ctx;

#include "sldqmc.h"

namespace sldqmc {

struct FlipPairs;

// Error bits raised by kernels into the context's device flag word.
enum : int {
    FLAG_NUMERICAL = 1,  // non-positive Cholesky pivot, zero LU pivot or non-finite value
    FLAG_ARG = 2,        // field value outside {-1, +1}
    FLAG_TIMEOUT = 4,    // a bounded device wait ran out
};

// Batched FP64 GEMM description: for each batch item b,
//   C = alpha * op(A) * diag(kscale) * op(B) * diag(nscale) * diag(mscale) + beta * C
// op(A) is M x K: A[m*lda + k] (TA = false) or A[k*lda + m] (TA = true).
// op(B) is K x N: B[k*ldb + n] (TB = false) or B[n*ldb + k] (TB = true).
// kscale/nscale/(s_m row scale) come from a field slice: value cu where s > 0, cd otherwise.
// mscale is a double vector (or its reciprocal when ms_recip).
// a_upper: A is upper triangular (op(A)[m][k] = 0 for k < m): skip those k.
// c_upper: only tiles touching the upper triangle of C (n >= m) are written.
struct GemmF64 {
    int M, N, K;
    const double *A;
    long long lda, sA;
    const double *B;
    long long ldb, sB;
    double *C;
    long long ldc, sC;
    double alpha, beta;
    const int8_t *s_k;
    long long sSk;
    const int8_t *s_n;
    long long sSn;
    const int8_t *s_m;  // row scale of C from a field slice
    long long sSm;
    double cu, cd;
    const double *ms;
    long long sMs;
    int ms_recip;
    int a_upper;
    int b_upper;  // op(B) upper triangular (op(B)[k][n] = 0 for k > n): skip those k
    int c_upper;
    int batch;
};

void gemm_f64(const GemmF64 &g, bool TA, bool TB, cudaStream_t st);
// Algorithmic flops of a GEMM description (triangles counted once).
double gemm_flops(const GemmF64 &g);
GemmF64 gemm_desc(int M, int N, int K, const double *A, long long lda, long long sA,
                  const double *B, long long ldb, long long sB, double *C, long long ldc,
                  long long sC, int batch);

// N >= 128: W = X X^T to FP64 accuracy on the
// BF16 tensor cores (Ozaki splitting; X row stride N, batch stride sX; W row
// stride ldw, batch stride sW; tiles on or above the diagonal written).
// oz_prepare leaves c->oz_ws null when the planes of the FP64 mode (made at any
// N) would take more than a third of the free memory; the FP64 pipe then does
// these products.  Defined in oz_gram.cu.
int oz_prepare(sldqmc_ctx *c);
void oz_release(sldqmc_ctx *c);
// Gives the twin t the context's ways of the FP64 mode's products: what c lacks t
// gives back; false if t has no room for what c has.
bool oz_match(const sldqmc_ctx *c, sldqmc_ctx *t);
void oz_gram(sldqmc_ctx *c, const double *X, long long sX, double *W, long long sW, int ldw, int B);
// Left-looking Cholesky-QR on the tensor cores (same N range):
// oz_chol_begin fixes the digit exponents of R's columns from diag(W);
// oz_chol_update subtracts the contributions of the finished rows
// kstart..k0-1 from rows k0..k0+kb of W and of Y = Q^T (k0 - kstart a
// multiple of 32 and > 0); oz_chol_panel factors the
// panel's diagonal block, forms its rows of R and Q^T as products with the
// block's inverse and splits them for the later panels.  W row stride N,
// item stride sW; R, Y row stride N, item stride N*N.
void oz_chol_begin(sldqmc_ctx *c, const double *W, long long sW, int B);
void oz_chol_update(sldqmc_ctx *c, int k0, int kb, int kstart, double *W, long long sW, double *Y, int B);
void oz_chol_panel(sldqmc_ctx *c, int k0, int kb, const double *W, long long sW, double *Y, double *R, int B);
// Rank-32 updates (row stride lda, item stride sA; panel k0..k0+kb), FP64-
// accurate on the tensor cores: the finalisation's LU (rhs: also the
// right-hand side in columns N..2N-1), its back substitution, and the pending
// pairs G_f -= U_f V_f of the delayed local update (U: N x 32, V: 32 x N).
void oz_lu_update(sldqmc_ctx *c, double *A, long long sA, int lda, int k0, int kb, int B, int rhs);
void oz_back_update(sldqmc_ctx *c, double *A, long long sA, int lda, int k0, int kb, int B);
void oz_delayed_update(sldqmc_ctx *c, double *const *G, const FlipPairs *pairs, int B);
// Products with exp(-+dtau K) on the tensor cores, FP64-accurate.  oz_have_e
// builds the digit planes of both propagators on first use and says whether
// they are there; oz_slice_product: Xt = X diag(d) E (d from the field slice
// sk); oz_similarity: dst_f = P src_f P^-1 of both flavours, P = E or, with
// inv, E^-1, rows and columns then scaled by d_i / d_j of the field slice s
// (null: no scaling), T_f an N x N scratch per item.
// oz_worth: whether they are the faster way for `times` plan_cap items; oz_full: every
// product of the context runs there (N >= 128).  oz_chain_block: the slice
// products of a whole block in one launch (oz_chain_fits: N <= 64).
bool oz_have_e(sldqmc_ctx *c);
bool oz_worth(const sldqmc_ctx *c, int times);
bool oz_full(const sldqmc_ctx *c);
bool oz_chain_fits(const sldqmc_ctx *c);
void oz_chain_block(sldqmc_ctx *c, const double *Ut, const int8_t *d_s, int B, double cu, double cd, int t0, int nb,
                    double *Xt_out);
void oz_slice_product(sldqmc_ctx *c, const double *X, const int8_t *sk, double cu, double cd, double *Xt, int B);
void oz_similarity(sldqmc_ctx *c, const double *const *src, double *const *T, double *const *dst, int inv,
                   const int8_t *s, const double (*ex)[2], int B);
// R = R2 R1 of the two passes on the tensor cores (tiles on or above the
// diagonal written); oz_keep_bounds saves the first pass's column bounds of R
// before the second pass replaces them.
void oz_keep_bounds(sldqmc_ctx *c, int B);
// V <- (D^-1 R D_p) P^T V, FP64-accurate on the tensor cores (R upper
// triangular; D, D_p, P from the context; Ts an N x N FP64 scratch per item).
void oz_update_V(sldqmc_ctx *c, const double *R, double *V, double *Ts, int B);
void oz_r2r1(sldqmc_ctx *c, const double *R2, const double *R1, double *R, int B);

// The whole weight of a configuration in one CTA (small.cu: FP64 mode, dense
// propagator, N <= 32).
bool small_fits(const sldqmc_ctx *c);
void small_weight(sldqmc_ctx *c, const int8_t *d_s, int B, double cu, double cd, int tau0, double *d_ld, int *d_sign,
                  double *d_G, double scale, int accumulate);

// One stabilisation of every item in one launch (small.cu: FP64 mode, N <= 64):
// Xt -> Y = Q^T, D, V and the sign of the context updated.
bool stab_block_fits(const sldqmc_ctx *c);
void stab_block(sldqmc_ctx *c, const double *Xt, double *Y, int B, int passes);
void stab_block_set_limits();

// Slice products with the separable exp(-dtau K) (sep.cu): X^T_out =
// U^T D_t0 E D_t0+1 E ... for nb slices, one row per CTA in shared memory.
bool sep_supported(int Lx, int Ly);
void sep_set_limits();
void sep_chain_block(sldqmc_ctx *c, const double *Ut, const int8_t *d_s, int B, double cu, double cd, int t0,
                     int nb, const double *ring, double *Xt_out);

// The accepted flips of one block of up to 32 sites of a slice, one record
// per chain: the sites in order, and per flavour what is needed to form the
// pairs u_n, v_n (G <- G - sum_n u_n v_n) at every row and column:
//   L[n][m] = u_m at site n,  X[m][n] = v_m at site n  (m < n),  coef[n] = Delta_n / R_n.
struct FlipPairs {
    double L[2][32][32], X[2][32][32], coef[2][32];
    int site[32], n;
};

// Event-bracketed timing of launches (sldqmc_profile_*).
struct ProfRec {
    cudaEvent_t a, b;
    int cls;
    double flops;
    const char *site;  // the launch site (a static string)
};
struct Prof {
    bool on = false;
    std::vector<ProfRec> recs;
    std::vector<cudaEvent_t> pool;
    size_t used = 0;
    int open_cls = -1;
    double open_flops = 0.0;
};
void prof_begin(sldqmc_ctx *c, int cls, double flops, const char *site = nullptr);
void prof_end(sldqmc_ctx *c);
// Launch an FP64 GEMM on the context's stream (counted and, when on, timed).
void gemm_ctx(sldqmc_ctx *c, const GemmF64 &g, bool TA, bool TB);

}  // namespace sldqmc

// The context (opaque in the public header).
struct sldqmc_ctx {
    sldqmc_params p;
    int N, M;
    cudaStream_t st;
    long long launches;
    int *d_flag;  // device error bits
    // constants
    double *d_K, *d_E, *d_Einv;  // N x N
    float *d_Ehi, *d_Elo;        // split-TF32 copies of E (3xTF32 mode)
    void *d_Ebf;                 // BF16 copy of E (BF16 mode)
    double ex_scale[2][2];       // [eta==-1][s<0]: exp(eta*dtau*xi*s)
    double dtauJ, Ktau;          // bare-weight constants
    // stabilisation workspace, cap items each
    int cap;
    int plan_cap;      // items per call that a choice between two ways of a product goes by: the caller's
                       // max_batch also on the twin, so that both give the same bits
    long long nn;      // N*N
    double *buf[9];    // Ut, V, X1, X2, W(2*nn), Y, R1, R2, Vg
    double *d_D, *d_Dp, *d_logacc;
    int *d_perm, *d_sgn, *d_piv;
    int *d_tslu;       // row nominations of the tournament-pivoting LU panels (24 * 32 per item)
    void *tc_ws;       // tensor-core operand workspace (split copies)
    void *oz_ws;       // digit planes of the tensor-core Gram and Cholesky-QR (mixed modes, N >= 128)
    // Monte Carlo state
    int8_t *d_s_tmp;   // cap * M * N proposal buffer
    int8_t *d_s_one;   // staging for host calls
    double *d_G[2];    // Gt for the local sweep: cap items per flavour
    double *d_U, *d_V; // pending pairs of the delayed local update: 2 flavours x cap x 32 N each
    int local_rank;    // sites per delayed-update block (1: immediate rank-1 updates)
    int tile_n;        // output tile width of the tensor-core slice products (64 or 128)
    double *d_ld_tmp, *d_ld_tmp2;
    int *d_sg_tmp;
    long long *d_stats; // cap * 4 (accepted, proposed, margin, drift bits)
    // effective model
    int n_class, n_off_total;
    int h_n_off[32];
    int h_offsets[64 * 3];
    double h_J[32];
    double E0;
    int have_model;
    int n_colors, max_color;  // colours and the sites of the largest
    int *d_col_start, *d_col_sites;
    long long *d_feat0, *d_feat1;
    double *d_Jdev;
    int *d_offdev, *d_noffdev;
    sldqmc::Prof *prof;
    const uint32_t *step_dev;  // when set (graph capture), kernels read the MC step from here
    uint32_t *d_step;          // this context's device step counter
    sldqmc_ctx *twin;          // second workspace (twice the capacity) + stream for the exact log weight
    cudaEvent_t ev_fork, ev_join;
    int no_twin;               // set on a twin itself, or when the twin could not be created
    int num_sms;               // streaming multiprocessors of the context's device
    int kinetic;               // SLDQMC_KINETIC_*: form in which exp(-dtau K) enters the slice products
};
