// oz_gram.cu -- FP64-accurate products on the BF16 tensor cores (Ozaki's
// error-free splitting).  For N >= 128: the stabilisation and the determinant in
// every mode (Gram matrices, the left-looking Cholesky-QR updates and panel
// products with the inverse of each 32 x 32 diagonal factor, formed here in
// FP64, R = R2 R1, the V update, the trailing updates of the LU and the back
// substitution of G), the slice products of the FP64 mode, and the wraps and
// delayed corrections of the local sweep's Green's functions.  Below: the FP64
// mode's slice products up to 64 sites (k_oz_chain), and those and the wraps to 127
// sites where there is enough work (oz_worth); the FP64 pipe keeps the rest.
//
// Why not the FP64 pipe in the FP64 mode: it runs at 1.05-1.10 TFLOP/s however
// a product is tiled (64 lanes-clocks per warp instruction), these products
// at 11-33 TFLOP/s (N = 400, 4 items: 47 us against 560; N = 576, 8 items and
// two flavours: 185 us against 5600).  The largest error of a product against
// extended precision is about a tenth of the FP64 GEMM's (Q D E, G E^-1,
// E G E^-1 at N = 144 .. 576: 0.7e-16 .. 1.2e-16 against 1.0e-15 .. 1.7e-15 of the
// largest element).
//
// The Gram matrix shows the scheme:
//
// W = X X^T for the rows x_i of X (N x N per batch item).  Each row is
// scaled by a power of two, 2^-E_i with |x_ik| < 2^E_i, and written as eight
// balanced base-2^7 digits,
//   x_ik 2^-E_i = sum_{p=1..8} a_p,ik 2^-(7p+1)   (|a_1| <= 256, |a_p| <= 64, p > 1),
// exact up to the rounding of x_ik 2^-E_i to a multiple of 2^-57.  Then
//   W_ij 2^-(E_i+E_j) = sum_{p,q} 2^-(7(p+q)+2) sum_k a_p,ik a_q,jk,
// of which the 36 products with p + q <= 9 are kept: each dropped term is
// below 2^-58 of the row maxima.  (The leading digit may use all of BF16's
// integers up to 256.  With |a_1| <= 128 the dropped terms are four times as
// large, 5e-17 rms of the row maxima's product at K = 256, which at the block
// condition limit, 16 x 16, n_wrap = 16, dtau = 0.1, left G off by 1.5e-13 where
// the FP64 pipe's is off by 4e-14.)  The digit planes are BF16 integers; the products of one group
// g = p + q share one FP32 tensor-memory accumulator, and every partial sum
// of a group is an integer of magnitude <= K 2^16 (the leading group; K (2^15 +
// 6 * 4096) the others) <= 2^24 for K <= 256, so the tensor-core accumulation
// is exact.  Longer contractions run in chunks of at most 256: the epilogue converts each chunk's eight
// group sums to integers and adds them, shifted, to two 64-bit integers, which
// hold the whole sum exactly (|h| <= K 2^37) and are rounded to FP64 once.
//
// One persistent CTA per SM walks the 128 x 32 output tiles of every item
// (for a Gram matrix only those on or above the diagonal; a launch may carry
// two parts with their own A rows and outputs): warp 0 streams the 8 + 8
// digit-plane tiles of a 32-wide K-block by TMA (64-byte swizzle), warp 1
// issues the 36 digit products per 16-wide K-step as eight MMAs (A's plane p
// against B's planes 0..7-p at once), and sixteen epilogue warps drain one
// of two tensor-memory buffers (8 groups x 32 columns each) while the next
// tile accumulates into the other.  Every mbarrier wait is bounded; a wait
// that runs out raises the context's timeout flag and the CTA frees its
// tensor memory and exits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "chol32.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace sldqmc {

namespace {

using namespace tcx;

constexpr int OZ_S = 8;           // digit planes
constexpr int OZ_BETA = 7;        // bits per digit
constexpr int OZ_G = 8;           // groups p + q = 2..9
constexpr int OZ_BITS = 57;       // bits of a scaled entry: x 2^-E = v 2^-57, seven digits below the leading one
constexpr int OZ_KCHUNK = 8;      // K-blocks (of 32) per exactly accumulated chunk: K <= 256
constexpr int OBM = 128, OBN = 32;
constexpr int OKE = 32;           // BF16 elements per K-block (64-byte rows)
constexpr int OSTAGES = 2;
constexpr int OTILE_A = OBM * 64;  // one digit plane of A per stage
constexpr int OTILE_B = OBN * 64;
constexpr int OSTAGE = OZ_S * (OTILE_A + OTILE_B);
constexpr int OEPI = 16;           // epilogue warps, four per TMEM lane quarter
constexpr int OCOL = OBN * 4 / OEPI;  // accumulator columns drained by one of them
constexpr int OTHREADS = 64 + 32 * OEPI;
constexpr int OTMEM = 2 * OZ_G * OBN;  // two buffers of eight 32-column accumulators

constexpr int OZ_NONFINITE = 1 << 20;  // exponent of a row with an infinity or a NaN

// Exponent of a row whose largest |entry| has the biased exponent ef_max.
__device__ __forceinline__ int oz_exponent(int ef_max)
{
    return ef_max == 0x7FF ? OZ_NONFINITE : (ef_max > 0 ? ef_max - 1022 : 0);
}

constexpr size_t oz_smem_bytes() { return (size_t)OSTAGES * OSTAGE + 1024 + 256; }

// Shared-memory descriptor of a K-major BF16 operand with 64-byte rows and the
// 64-byte swizzle (8-row atoms of 512 bytes).
__device__ __forceinline__ uint64_t smem_desc64(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;
    d |= (uint64_t)(512u >> 4) << 32;
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)4u << 61;
    return d;
}

// kind::f16 with BF16 operands, FP32 accumulator, K-major A and B, M = 128,
// N = n (a multiple of 32 up to 256).
__device__ __forceinline__ constexpr uint32_t oz_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OBM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// The balanced base-2^7 digits of x 2^-E = sum_p dg[p] 2^-(7p+8), p = 0..7, for
// |x| < 2^E (E the frexp exponent of its row's maximum, or a bound; subnormals
// count as zero): v = x 2^(57-E) rounded to an integer, plus the bias that makes
// each of the seven low 7-bit fields a digit + 64, so that the digits are
// fields, without carries.
__device__ __forceinline__ long long oz_fixed(double x, int E)
{
    const long long u = __double_as_longlong(x);
    const int ef = (int)((u >> 52) & 0x7FF);
    const unsigned long long m = ((unsigned long long)u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int r = E - ef + 1075 - OZ_BITS;  // x = m 2^(ef - 1075); r >= -4 since |x| < 2^E
    long long v = 0;
    if (ef > 0 && r < 60) v = r <= 0 ? (long long)(m << (r < -4 ? 4 : -r)) : (long long)((m + (1ull << (r - 1))) >> r);
    constexpr long long bias = 64ll * (1 + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35) + (1ll << 42));
    return (u < 0 ? -v : v) + bias;
}

// Digit p of two such values as a pair of BF16: an integer below 2^23 placed
// in the mantissa of 2^23 (1.5 2^23 for the signed leading digit) is converted
// by one FP32 subtraction, and BF16 is the upper half of its FP32.
__device__ __forceinline__ uint32_t oz_pair(long long a, long long b, int p)
{
    float fa, fb;
    if (p == 0) {
        fa = __uint_as_float(0x4B400000u + (uint32_t)(int)(a >> 49)) - 12582912.0f;
        fb = __uint_as_float(0x4B400000u + (uint32_t)(int)(b >> 49)) - 12582912.0f;
    } else {
        const int s = 7 * (7 - p);
        fa = __uint_as_float(0x4B000000u | ((uint32_t)(a >> s) & 127u)) - 8388672.0f;
        fb = __uint_as_float(0x4B000000u | ((uint32_t)(b >> s) & 127u)) - 8388672.0f;
    }
    return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// Plane p of eight values, 16 bytes.
__device__ __forceinline__ uint4 oz_pair8(const long long (&v)[8], int p)
{
    return make_uint4(oz_pair(v[0], v[1], p), oz_pair(v[2], v[3], p), oz_pair(v[4], v[5], p), oz_pair(v[6], v[7], p));
}

// Digits of the rows of one or two matrices (rows x cols, row stride ld, item
// stride sX; blockIdx.z selects the matrix): row i becomes plane row i (prow
// plane rows per item, leading dimension ldp) with K positions 0..cols-1 and
// exponent E[b * prow + i]; the planes' columns from cols to the next multiple
// of 32 are zero, those beyond are left as they are (zero pads of the buffer).
// With a field slice sk the entries of column k are first multiplied by cu
// where sk > 0 and by cd otherwise (the D of a slice product X D E).  One warp per row, eight rows per CTA: the row's
// maximum by warp shuffles, then each lane converts pairs of adjacent entries
// and stores each plane's pair as one BF16x2.
struct OzRows {
    const double *X[2];
    __nv_bfloat16 *planes[2];
    int *E[2];
    const int8_t *sk;
    long long sSk;
    double cu, cd;
};

template <bool SCALE>
__global__ void __launch_bounds__(256) k_oz_slice(OzRows a, long long sX, int rows, int cols, int ld, int prow,
                                                  int ldp, long long plane_stride)
{
    const int b = blockIdx.y, lane = threadIdx.x & 31;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= rows) return;  // whole warps
    const int N = cols;
    const double *x = (blockIdx.z ? a.X[1] : a.X[0]) + (long long)b * sX + (long long)i * ld;
    const int8_t *sk = SCALE ? a.sk + (long long)b * a.sSk : nullptr;
    auto at = [&](int k) {
        const double v = x[k];
        return SCALE ? v * (sk[k] > 0 ? a.cu : a.cd) : v;
    };
    // the largest |x_ik| (non-negative doubles order like their bit patterns)
    unsigned long long mx = 0;
    for (int k = lane; k < N; k += 32) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(at(k)) & 0x7FFFFFFFFFFFFFFFull;
        mx = u > mx ? u : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = v > mx ? v : mx;
    }
    const int ef_max = (int)(mx >> 52);
    const int Ei = oz_exponent(ef_max);
    if (lane == 0) (blockIdx.z ? a.E[1] : a.E[0])[(long long)b * prow + i] = Ei;
    __nv_bfloat16 *row = (blockIdx.z ? a.planes[1] : a.planes[0]) + ((long long)b * prow + i) * ldp;
    for (int k = 2 * lane; k < (N + 31) / 32 * 32; k += 64) {
        const long long v0 = oz_fixed(k < N ? at(k) : 0.0, Ei), v1 = oz_fixed(k + 1 < N ? at(k + 1) : 0.0, Ei);
#pragma unroll
        for (int p = 0; p < OZ_S; ++p)
            *reinterpret_cast<uint32_t *>(row + (long long)p * plane_stride + k) = oz_pair(v0, v1, p);
    }
}

// Digits of krows rows of a row-major matrix (row stride ld), in blocks of 32
// rows (blockIdx.z), stored from K-block koff/32 of the planes on: plane row
// j (j0 <= j < Nc) gets src[l * ld + j] at K position koff + l (0 beyond
// krows within the last block).
// The exponents are given (Ej[b * sE + j]; sE = 0 for one shared row of
// exponents), chosen by the caller as bounds known before the values exist;
// a value at or above its bound raises the numerical flag.  LOCAL: krows <=
// 32 (one block), and each plane row takes the exponent of its own largest
// entry, written to Ej.  One CTA converts 32 plane rows; eight threads share
// a row.
template <bool LOCAL>
__device__ __forceinline__ void oz_slice_block(int bx, const double *src, long long sS, long long ld, int j0, int Nc,
                                               int krows, int koff, long long plane_stride, int rows_cap, int ldk,
                                               __nv_bfloat16 *planes, int *Ej, long long sE, int *flag,
                                               const int *rowidx, long long sR, double (*tile)[33])
{
    const int b = blockIdx.y, c0 = j0 + bx * 32;
    // blockIdx.z: the 32-row block of the krows source rows (K positions koff + 32 z ..);
    // source row l is rowidx[b * sR + l] when a row index is given
    const int kz = 32 * blockIdx.z;
    const int kb = krows - kz < 32 ? krows - kz : 32;
    koff += kz;
    const double *s = src + (long long)b * sS;
    const int *ri = rowidx ? rowidx + (long long)b * sR + kz : nullptr;
    for (int idx = threadIdx.x; idx < 32 * 32; idx += blockDim.x) {
        const int l = idx >> 5, r = idx & 31;
        double v = 0.0;
        if (l < kb && c0 + r < Nc) v = s[(long long)(ri ? ri[l] : kz + l) * ld + c0 + r];
        tile[l][r] = v;
    }
    __syncthreads();
    const int r = threadIdx.x >> 3, q = threadIdx.x & 7;
    const int j = c0 + r;
    long long v4[4];
    if (LOCAL) {
        // the row's largest |entry| over its eight threads (lanes 8r'..8r'+7)
        unsigned long long mx = 0;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const unsigned long long u =
                (unsigned long long)__double_as_longlong(tile[4 * q + jj][r]) & 0x7FFFFFFFFFFFFFFFull;
            mx = u > mx ? u : mx;
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = v > mx ? v : mx;
        }
        if (j >= Nc) return;
        const int ef_max = (int)(mx >> 52);
        const int E = oz_exponent(ef_max);
        if (q == 0) Ej[(long long)b * sE + j] = E;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) v4[jj] = oz_fixed(tile[4 * q + jj][r], E);
    } else {
        if (j >= Nc) return;
        const int E = Ej[(long long)b * sE + j];
        const unsigned long long bound = (unsigned long long)(E + 1023) << 52;  // bit pattern of 2^E
        bool over = false;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const double x = tile[4 * q + jj][r];
            over |= ((unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull) >= bound;
            v4[jj] = oz_fixed(x, E);
        }
        if (over) atomicOr(flag, FLAG_NUMERICAL);
    }
    const long long row = ((long long)b * rows_cap + j) * ldk + koff + 4 * q;
#pragma unroll
    for (int p = 0; p < OZ_S; ++p)
        *reinterpret_cast<uint2 *>(planes + (long long)p * plane_stride + row) =
            make_uint2(oz_pair(v4[0], v4[1], p), oz_pair(v4[2], v4[3], p));
}

__global__ void __launch_bounds__(256) k_oz_slice_fixed(const double *src, long long sS, long long ld, int j0, int Nc,
                                                        int krows, int koff, long long plane_stride, int rows_cap,
                                                        int ldk, __nv_bfloat16 *planes, int *Ej, long long sE,
                                                        int *flag, const int *rowidx = nullptr, long long sR = 0)
{
    __shared__ double tile[32][33];
    oz_slice_block<false>(blockIdx.x, src, sS, ld, j0, Nc, krows, koff, plane_stride, rows_cap, ldk, planes, Ej, sE,
                          flag, rowidx, sR, tile);
}

// The unsolved rows k0..k0+kb of a Cholesky-QR panel in one launch, each
// plane row with its own maximum (LOCAL): blocks x < nb0 split Y's rows (all
// N columns, into the Q^T planes), the others W's (columns j0.., into the R
// planes).
struct OzPanelSlice {
    const double *src[2];
    long long sS[2];
    int j0[2], nb0;
    __nv_bfloat16 *planes[2];
    int *E[2];
};

__device__ __forceinline__ void oz_slice_panel(const OzPanelSlice &a, int x, int N, int ld, int kb, int koff,
                                               long long plane_stride, int ldk, int *flag, double (*tile)[33])
{
    const int part = x < a.nb0 ? 0 : 1;
    oz_slice_block<true>(part ? x - a.nb0 : x, part ? a.src[1] : a.src[0], part ? a.sS[1] : a.sS[0], ld,
                         part ? a.j0[1] : a.j0[0], N, kb, koff, plane_stride, N, ldk, part ? a.planes[1] : a.planes[0],
                         part ? a.E[1] : a.E[0], N, flag, nullptr, 0, tile);
}

__global__ void __launch_bounds__(256) k_oz_slice_panel(OzPanelSlice a, int N, int ld, int kb, int koff,
                                                        long long plane_stride, int ldk, int *flag)
{
    __shared__ double tile[32][33];
    oz_slice_panel(a, blockIdx.x, N, ld, kb, koff, plane_stride, ldk, flag, tile);
}

// Bounds for the entries of R's columns in a Cholesky factorisation of the
// Gram matrix W: sum_l R_lj^2 = W_jj, so |R_lj| <= sqrt(W_jj) < 2^E_j with
// E_j = ceil(e/2) + 1, W_jj < 2^e (one bit of margin for rounding).
__global__ void k_oz_col_exponents(const double *W, long long sW, int ldw, int N, int *E)
{
    const int b = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        const unsigned long long u =
            (unsigned long long)__double_as_longlong(W[(long long)b * sW + (long long)j * ldw + j]) & 0x7FFFFFFFFFFFFFFFull;
        const int ef = (int)(u >> 52);
        const int e = ef > 0 ? ef - 1022 : -1022;
        E[(long long)b * N + j] = ((e + 1) >> 1) + 1;
    }
}

// E[b][j] = frexp exponent of max_r |src[r][j]| (|src[r][j]| < 2^E; 0 for a
// zero column).  A CTA covers 32 columns with eight row groups (each warp
// reads one 256-byte row segment per row); the eight partial maxima meet in
// shared memory.
__global__ void __launch_bounds__(256) k_oz_col_max_exponents(const double *src, long long sS, int rows, int cols,
                                                              int *E)
{
    __shared__ unsigned long long part[8][32];
    const int b = blockIdx.y, lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + lane;
    const double *s = src + (long long)b * sS;
    unsigned long long mx = 0;
    if (j < cols) {
#pragma unroll 4
        for (int r = g; r < rows; r += 8) {
            const unsigned long long u = (unsigned long long)__double_as_longlong(s[(long long)r * cols + j]) & 0x7FFFFFFFFFFFFFFFull;
            mx = u > mx ? u : mx;
        }
    }
    part[g][lane] = mx;
    __syncthreads();
    if (g == 0 && j < cols) {
#pragma unroll
        for (int q = 1; q < 8; ++q) mx = part[q][lane] > mx ? part[q][lane] : mx;
        const int ef = (int)(mx >> 52);
        E[(long long)b * cols + j] = oz_exponent(ef);
    }
}

// T[m][k] = R[m][k] Dp[k] / D[m] for k >= m, 0 below (FP64), the triangular
// factor of the V update V <- T P^T V.
__global__ void k_oz_make_T(const double *R, long long nn, int N, const double *D, const double *Dp, double *T)
{
    const int b = blockIdx.z, m = blockIdx.y;
    __shared__ double s_rd;  // one division per row (FP64 division is a long chain on this pipe)
    if (threadIdx.x == 0) s_rd = 1.0 / D[(long long)b * N + m];
    __syncthreads();
    const double rd = s_rd;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x)
        T[(long long)b * nn + (long long)m * N + k] =
            k >= m ? R[(long long)b * nn + (long long)m * N + k] * Dp[(long long)b * N + k] * rd : 0.0;
}

// What a Cholesky-QR panel needs before its product [R_k,k+ | Q_k^T] = T
// [W_k,k+ | Y_k] on the tensor cores, in one launch.  Block x = 0 of an item: the
// factor of the diagonal block, W_kk = R_kk^T R_kk (written to R), and the digit
// planes of T = R_kk^-T (each row with its own maximum as exponent, ET); the
// other blocks: the digits of the unsolved rows of Y and W.  Both read only
// what the previous launch wrote, and the splitting hides behind the factor's
// chain of pivots.  By events around the launches (32 x 32, 4 items): 34 us for
// a factor with the library's rsqrt and separate arrays for R and T and 8 us
// for the splitting; 18.7 us together.
struct OzPanelPrep {
    const double *W;
    long long sW;
    double *R;
    long long sR;
    int N, k0, kb;
    __nv_bfloat16 *tplanes;
    long long tps;
    int *ET;
};

template <bool EXACT>
__global__ void __launch_bounds__(256) k_oz_panel_prep(OzPanelPrep f, OzPanelSlice a, long long plane_stride, int ldk,
                                                       int *flag)
{
    __shared__ double X[32][33];
    __shared__ double root[32];
    __shared__ CholScratch sc;
    if (blockIdx.x > 0) {
        oz_slice_panel(a, blockIdx.x - 1, f.N, f.N, f.kb, f.k0, plane_stride, ldk, flag, X);
        return;
    }
    const int b = blockIdx.y, tid = threadIdx.x, kb = f.kb;
    const double *Wb = f.W + (long long)b * f.sW + (long long)f.k0 * f.N + f.k0;
    for (int e = tid; e < 32 * 32; e += 256) {
        const int r = e >> 5, c = e & 31;
        X[r][c] = r < kb && c < kb ? (c >= r ? Wb[(long long)r * f.N + c] : 0.0) : (r == c ? 1.0 : 0.0);
    }
    __syncthreads();
    chol32<EXACT>(X, root, sc, kb, flag);
    double *Rb = f.R + (long long)b * f.sR + (long long)f.k0 * f.N + f.k0;
    for (int e = tid; e < 32 * 32; e += 256) {
        const int r = e >> 5, c = e & 31;
        if (r < kb && c < kb) Rb[(long long)r * f.N + c] = c > r ? X[r][c] : (c == r ? root[r] : 0.0);
    }
    // digits of T's rows: eight threads per row, four K positions each
    const int r = tid >> 3, q = tid & 7;
    double tv[4];
    unsigned long long mx = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        tv[i] = 4 * q + i <= r ? X[r][4 * q + i] : 0.0;
        const unsigned long long u = (unsigned long long)__double_as_longlong(tv[i]) & 0x7FFFFFFFFFFFFFFFull;
        mx = u > mx ? u : mx;
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = v > mx ? v : mx;
    }
    const int ef_max = (int)(mx >> 52);
    const int E = oz_exponent(ef_max);
    if (q == 0) f.ET[b * 32 + r] = E;
    long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = oz_fixed(tv[i], E);
    const long long row = ((long long)b * 32 + r) * 32 + 4 * q;
#pragma unroll
    for (int p = 0; p < OZ_S; ++p)
        *reinterpret_cast<uint2 *>(f.tplanes + (long long)p * f.tps + row) =
            make_uint2(oz_pair(v[0], v[1], p), oz_pair(v[2], v[3], p));
}

// One part of a product's rows: rows m of C (rows of A, starting at plane row
// arow0 of the part's A map), their exponents, and where C goes; with SLICE,
// where the digits of C's values go as well (plane rows srow0 + m, K
// positions skoff + n, exponents SE[b * sSE + srow0 + m]).
struct OzPart {
    int M, arow0;
    const int *EA;
    long long sEA;
    const int *EB;  // row exponents of the part's B
    long long sEB;
    double *C;
    long long sC;
    int ldc;
    __nv_bfloat16 *sp;
    const int *SE;
    long long sSE;
    int srow0;
};

// h 2^e + l 2^(e-28), rounded once to nearest even.  FP64: two conversions and
// an FMA (a warp's FP64 instruction holds its sub-partition's pipe for 64
// cycles), the scale through the exponent field while the result stays normal.
// NaN for the exponent of a row that holds an infinity or a NaN (its digits
// are zero).
__device__ __forceinline__ double oz_round_fp(long long h, long long l, int e)
{
    const double x = fma((double)l, 0x1p-28, (double)h);
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF);
    if (ex != 0 && ex + e > 0 && ex + e < 2047) return __longlong_as_double(bits + ((long long)e << 52));
    if (e > OZ_NONFINITE / 2) return __longlong_as_double(0x7FF8000000000000ll);
    return scalbn(x, e);
}

// The same by integer operations, for the updates: their subtraction takes the
// FP64 pipe as well, and with K = 32 there are few MMAs to hide either behind
// (rank-32 update at N = 576, 16 items: 78 -> 73 us; a Gram matrix at N = 256,
// 128 items, whose epilogue hides behind its MMAs: 125 -> 128 us, so products
// without a subtraction keep the form above).
__device__ __forceinline__ double oz_round(long long h, long long l, int e)
{
    // T = h 2^28 + l in three words, then |T|
    unsigned long long lo = ((unsigned long long)h << 28) + (unsigned long long)l;
    long long hi = (h >> 36) + (l >> 63) + (lo < (unsigned long long)l ? 1 : 0);
    const unsigned long long sign = (unsigned long long)hi & 0x8000000000000000ull;
    if (hi < 0) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0ull ? 1 : 0);
    }
    uint32_t t2 = (uint32_t)hi, t1 = (uint32_t)(lo >> 32), t0 = (uint32_t)lo;
    int ex = e + 95 - 28 + 1023;
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (t2 == 0u) {
            t2 = t1;
            t1 = t0;
            t0 = 0u;
            ex -= 32;
        }
    const int s = __clz((int)t2);
    ex -= s;
    if (t2 == 0u || (unsigned)(ex - 1) >= 2045u) {  // zero, subnormal, too large, NaN
        if ((t2 | t1 | t0) == 0u && e <= OZ_NONFINITE / 2) return 0.0;
        return oz_round_fp(h, l, e);
    }
    const uint32_t a = __funnelshift_l(t1, t2, s), b = __funnelshift_l(t0, t1, s);
    const uint32_t rem = (b << 21) | ((t0 << s) != 0u ? 1u : 0u);  // the bits below the 53rd
    unsigned long long m = ((unsigned long long)a << 21) | (b >> 11);
    m += (rem > 0x80000000u || (rem == 0x80000000u && (m & 1ull))) ? 1ull : 0ull;
    return __longlong_as_double((long long)(sign | (((unsigned long long)(ex - 1) << 52) + m)));
}

// acc + v 2^s in one multiply-add
__device__ __forceinline__ void oz_fold(long long &acc, int v, int s)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(v), "r"(1 << s));
}

struct OzArgs {
    OzPart pt[2];           // pt[1] only with nparts = 2 (its A rows and B through the second maps)
    int nparts;
    int Nn, brow0;          // rows of B (columns of C), first plane row of B
    int batch, nk;          // items, 32-wide K-blocks
    int kA0, kB0;           // first K positions (elements) of A and B in their planes
    int b_shared;           // one B for every item
    int stack;              // > 0: the items' rows lie one after another (batch = 1, M = items x stack), and
                            // row m of the product belongs to row m % stack of item m / stack of C
    const int8_t *sgn;      // TRANS without SUB, stacked: C[n][i] is scaled by d_n / d_i, d = cu where the item's
    long long sSgn;         // field slice is > 0 and cd otherwise (r_ud = cu / cd, r_du = cd / cu)
    double r_ud[2], r_du[2];  // per part
    long long splane_stride;  // SLICE: plane stride, leading dimension, plane rows per item,
    int sldp, srows, skoff;   // and the K position of n = 0
    int a_tri, b_tri;         // A upper triangular (A[m][k] = 0 for k < m) / B^T upper triangular
                              // (B[n][k] = 0 for k > n): a tile's K-blocks start at m0 / 32 / end
                              // after the one holding n0 + 31 (kA0 = kB0 = 0)
    int *flag;
};

// K-blocks [k_lo, k_hi) that can hold nonzero products for the tile at (m0, n0).
__device__ __forceinline__ void oz_krange(const OzArgs &a, int m0, int n0, int &k_lo, int &k_hi)
{
    k_lo = a.a_tri ? m0 / OKE : 0;
    k_hi = a.nk;
    if (a.b_tri) {
        const int e = (n0 + OBN + OKE - 1) / OKE;
        if (e < k_hi) k_hi = e;
    }
    if (k_hi < k_lo) k_hi = k_lo;
}

// Tile t of the persistent walk -> (item, first row, first column).
// Without UPPER every tile, row strip by row strip, columns fastest (a wave
// of CTAs shares one row strip of A; the tiles of a strip have the same K
// range, which keeps the triangular products balanced).  UPPER: the
// 128 x 32 tiles on or above the diagonal (tile (tm, tn) with tn >= 4 tm)
// of a Gram matrix, in groups of OZ_GROUP_M row strips, column-major inside
// a group, so that the CTAs of one wave share a few row strips of A and a
// few of B: walking columns first, every CTA of a wave read its own B strip,
// and at N = 10^4 the digit planes (16 bytes per element) far exceed L2 (at
// N = 4096 the grouped walk reads 2.7 instead of 5.3 GB from DRAM per Gram,
// in the same time).  In a group of gm strips starting at m_first, the walk
// first meets the ramp of columns 4 (m_first + j) .. + 3 with j + 1 rows
// (j < gm - 1), then columns with all gm rows.
constexpr int OZ_GROUP_M = 8;

// Upper tiles of the group of gm row strips starting at m_first.
__host__ __device__ inline int oz_group_tiles(int m_first, int gm, int tiles_n)
{
    const int T = tiles_n - 4 * m_first, F = T / 4, R = T % 4;
    const int S = F <= gm ? F * (F + 1) / 2 : gm * (gm + 1) / 2 + (F - gm) * gm;
    return 4 * S + R * (F + 1 < gm ? F + 1 : gm);
}

template <bool UPPER>
__device__ __forceinline__ void oz_tile(int t, int tiles_m, int tiles_n, int per_item, int &b, int &m0, int &n0)
{
    b = t / per_item;
    int r = t - b * per_item;
    if (!UPPER) {
        m0 = (r / tiles_n) * OBM;
        n0 = (r % tiles_n) * OBN;
        return;
    }
    int m_first = 0, gm = 0;
    for (; m_first < tiles_m; m_first += OZ_GROUP_M) {
        gm = tiles_m - m_first < OZ_GROUP_M ? tiles_m - m_first : OZ_GROUP_M;
        const int cnt = oz_group_tiles(m_first, gm, tiles_n);
        if (r < cnt) break;
        r -= cnt;
    }
    for (int j = 0; j < gm - 1; ++j) {
        const int cols = tiles_n - 4 * (m_first + j) < 4 ? tiles_n - 4 * (m_first + j) : 4;
        const int n_in = cols * (j + 1);
        if (r < n_in) {
            m0 = (m_first + r % (j + 1)) * OBM;
            n0 = (4 * (m_first + j) + r / (j + 1)) * OBN;
            return;
        }
        r -= n_in;
    }
    m0 = (m_first + r % gm) * OBM;
    n0 = (4 * (m_first + gm - 1) + r / gm) * OBN;
}

template <bool UPPER>
__host__ __device__ inline int oz_per_item(int tiles_m, int tiles_n)
{
    if (!UPPER) return tiles_m * tiles_n;
    int n = 0;
    for (int tm = 0; tm < tiles_m; ++tm) n += tiles_n - 4 * tm;
    return n;
}

// Tiles of the whole launch: part 0's for all items, then part 1's.
template <bool UPPER>
__host__ __device__ inline int oz_part_tiles(const OzArgs &a, int part)
{
    const int M = part ? a.pt[1].M : a.pt[0].M;
    return oz_per_item<UPPER>((M + OBM - 1) / OBM, (a.Nn + OBN - 1) / OBN) * a.batch;
}

template <bool UPPER>
__device__ __forceinline__ void oz_locate(const OzArgs &a, int t, int tiles0, int &part, int &b, int &m0, int &n0)
{
    part = t < tiles0 ? 0 : 1;
    if (part) t -= tiles0;
    const int M = part ? a.pt[1].M : a.pt[0].M;
    const int tiles_m = (M + OBM - 1) / OBM, tiles_n = (a.Nn + OBN - 1) / OBN;
    oz_tile<UPPER>(t, tiles_m, tiles_n, oz_per_item<UPPER>(tiles_m, tiles_n), b, m0, n0);
}

// UPPER: only the tiles on or above the diagonal (C square, A and B the same
// rows); SUB: C -= A B^T, otherwise C = A B^T; TRANS: element (m, n) of the
// product lives at C[n * ldc + m] (a warp's 32 rows m are then contiguous);
// SLICE (with TRANS, not SUB): the results are also split into digit planes
// with given exponents, the value (m, n) at K position skoff + n of plane row
// srow0 + m (zero digits for n >= Nn up to the tile's 32).
template <bool UPPER, bool SUB, bool TRANS = false, bool SLICE = false>
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tA1,
              const __grid_constant__ CUtensorMap tB0, const __grid_constant__ CUtensorMap tB1, OzArgs a)
{
    static_assert(!SLICE || (TRANS && !SUB), "SLICE needs TRANS and C = A B^T");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(base + OSTAGES * OSTAGE);
    uint64_t *empty = full + OSTAGES;
    uint64_t *tmem_full = empty + OSTAGES;  // [2]
    uint64_t *tmem_free = tmem_full + 2;    // [2]
    uint32_t *tmem_slot = (uint32_t *)(tmem_free + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles0 = oz_part_tiles<UPPER>(a, 0);
    const int tiles = tiles0 + (a.nparts > 1 ? oz_part_tiles<UPPER>(a, 1) : 0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < OSTAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int u = 0; u < 2; ++u) {
            mbar_init(&tmem_full[u], 1);
            mbar_init(&tmem_free[u], 32 * OEPI);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(OTMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                int part, b, m0, n0;
                oz_locate<UPPER>(a, t, tiles0, part, b, m0, n0);
                const CUtensorMap *mA = part ? &tA1 : &tA0;
                const CUtensorMap *mB = part ? &tB1 : &tB0;
                const int bB = a.b_shared ? 0 : b;
                const int arow0 = part ? a.pt[1].arow0 : a.pt[0].arow0;
                int k_lo, k_hi;
                oz_krange(a, m0, n0, k_lo, k_hi);
                for (int kb = k_lo; kb < k_hi; ++kb, ++it) {
                    const int s = it % OSTAGES;
                    if (it >= OSTAGES && !mbar_wait(&empty[s], ((it / OSTAGES) - 1) & 1, a.flag)) { ok = false; break; }
                    mbar_expect_tx(&full[s], OSTAGE);
                    uint8_t *st = base + s * OSTAGE;
                    const int k0 = kb * OKE;
#pragma unroll
                    for (int p = 0; p < OZ_S; ++p) {
                        tma_load_4d(st + p * OTILE_A, mA, a.kA0 + k0, arow0 + m0, b, p, &full[s]);
                        tma_load_4d(st + OZ_S * OTILE_A + p * OTILE_B, mB, a.kB0 + k0, a.brow0 + n0, bB, p, &full[s]);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0, cc = 0;  // K-block and chunk counters of this CTA
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                int part, b, m0, n0, k_lo, k_hi;
                oz_locate<UPPER>(a, t, tiles0, part, b, m0, n0);
                oz_krange(a, m0, n0, k_lo, k_hi);
                for (int kc0 = k_lo; kc0 < k_hi && ok; kc0 += OZ_KCHUNK, ++cc) {
                    const int u = cc & 1;
                    // the epilogue must have drained this buffer (used two chunks ago)
                    if (cc >= 2 && !mbar_wait(&tmem_free[u], ((cc >> 1) - 1) & 1, a.flag)) { ok = false; break; }
                    fence_after();
                    const uint32_t acc0 = tmem + (uint32_t)(u * OZ_G * OBN);
                    const int kc1 = kc0 + OZ_KCHUNK < k_hi ? kc0 + OZ_KCHUNK : k_hi;
                    for (int kb = kc0; kb < kc1; ++kb, ++it) {
                        const int s = it % OSTAGES;
                        if (!mbar_wait(&full[s], (it / OSTAGES) & 1, a.flag)) { ok = false; break; }
                        fence_after();
                        const uint32_t sa = smem_u32(base + s * OSTAGE);
                        const uint32_t sb = sa + OZ_S * OTILE_A;
                        // The B planes of a stage lie one after another (32 rows each), so
                        // planes 0..7-p form one K-major operand of 32 (8 - p) rows: a single
                        // MMA multiplies A's plane p with all of them, and with its output
                        // starting at column 32 p the product with plane q lands in group
                        // p + q's accumulator.  Eight MMAs per K-step instead of 36, each
                        // reading A's plane from shared memory once.  The first MMA of a
                        // chunk (p = 0) spans every group and initialises all eight.
#pragma unroll
                        for (int k = 0; k < OKE / 16; ++k) {
#pragma unroll
                            for (int p = 0; p < OZ_S; ++p) {
                                mma_bf16(acc0 + (uint32_t)(p * OBN), smem_desc64(sa + p * OTILE_A + k * 32),
                                         smem_desc64(sb + k * 32), oz_idesc(OBN * (OZ_S - p)),
                                         (kb != kc0 || k != 0 || p != 0) ? 1u : 0u);
                            }
                        }
                        mma_commit(&empty[s]);
                    }
                    if (ok) mma_commit(&tmem_full[u]);
                }
            }
        }
    } else {
        // epilogue: warp w drains lane quarter w % 4, columns [hc, hc + OCOL)
        const int q4 = warp & 3;
        const int hc = ((warp - 2) >> 2) * OCOL;
        int cc = 0;  // chunk counter, in step with the MMA thread's
        bool ok = true;
        for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
            int part, b, m0, n0;
            oz_locate<UPPER>(a, t, tiles0, part, b, m0, n0);
            const int M = part ? a.pt[1].M : a.pt[0].M;
            const int *EA = part ? a.pt[1].EA : a.pt[0].EA;
            const long long sEA = part ? a.pt[1].sEA : a.pt[0].sEA;
            double *C = part ? a.pt[1].C : a.pt[0].C;
            const long long sC = part ? a.pt[1].sC : a.pt[0].sC;
            const int ldc = part ? a.pt[1].ldc : a.pt[0].ldc;
            const int mm = m0 + q4 * 32 + lane;
            const int Ei = mm < M ? EA[(long long)b * sEA + mm] : 0;
            // element (mm, n) at o[n * cs]; for an update, the old values of this
            // thread's row segment, fetched while the MMAs run
            const int item = a.stack ? mm / a.stack : b, mi = a.stack ? mm - item * a.stack : mm;
            double *o = C + (long long)item * sC + (TRANS ? (long long)mi : (long long)mi * ldc);
            const long long cs = TRANS ? ldc : 1;
            const int nb = n0 + hc;
            const int *eb = (part ? a.pt[1].EB : a.pt[0].EB) + (a.b_shared ? 0 : (long long)b * (part ? a.pt[1].sEB : a.pt[0].sEB));
            double cold[OCOL];
#pragma unroll
            for (int j = 0; j < OCOL; ++j) cold[j] = (SUB && mm < M && nb + j < a.Nn) ? o[(nb + j) * cs] : 0.0;
            // the columns' exponents, also fetched while the MMAs run (not for an
            // update, whose old values already take those registers)
            int ebv[OCOL];
#pragma unroll
            for (int j = 0; j < OCOL; ++j) ebv[j] = (!SUB && nb + j < a.Nn) ? eb[nb + j] : 0;
            // The group sums as exact integers, folded as they arrive and added
            // over the K-chunks (|h| <= K 2^37): groups 0..3 (p + q = 2..5) into h,
            // 4..7 (6..9) into l, so that sum_g acc_g 2^-(7(g+2)+2) = h 2^-37 + l 2^-65
            long long h[OCOL], l[OCOL];
#pragma unroll
            for (int j = 0; j < OCOL; ++j) h[j] = l[j] = 0;
            int k_lo, k_hi;
            oz_krange(a, m0, n0, k_lo, k_hi);
            for (int kc0 = k_lo; kc0 < k_hi; kc0 += OZ_KCHUNK, ++cc) {
                const int u = cc & 1;
                ok = mbar_wait(&tmem_full[u], (cc >> 1) & 1, a.flag);
                fence_after();
                const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(u * OZ_G * OBN + hc);
#pragma unroll
                for (int gg = 0; gg < OZ_G; gg += 4) {
                    uint32_t r[4][OCOL];
#pragma unroll
                    for (int g = 0; g < 4; ++g) tmem_ld8_nowait(lane_base + (uint32_t)((gg + g) * OBN), r[g]);
                    tmem_wait_ld8x4(r[0], r[1], r[2], r[3]);
#pragma unroll
                    for (int j = 0; j < OCOL; ++j)
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            oz_fold(gg ? l[j] : h[j], __float2int_rn(__uint_as_float(r[g][j])), OZ_BETA * (3 - g));
                }
                fence_before();
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tmem_free[u])) : "memory");
                if (!ok) break;
            }
            if (!ok) break;
            if (mm >= M) continue;
            const int8_t *sg = (TRANS && !SUB && !SLICE && a.sgn) ? a.sgn + (long long)item * a.sSgn : nullptr;
            const bool up = sg && sg[mi] > 0;
#pragma unroll
            for (int j = 0; j < OCOL; ++j) {
                const int n = nb + j;
                double v = 0.0;
                if (n < a.Nn) {
                    v = SUB ? oz_round(h[j], l[j], Ei + eb[n] - 37) : oz_round_fp(h[j], l[j], Ei + ebv[j] - 37);
                    if (sg) {
                        const bool un = sg[n] > 0;
                        if (un != up) v *= un ? a.r_ud[part] : a.r_du[part];
                    }
                    o[n * cs] = SUB ? cold[j] - v : v;
                }
                if (SLICE) h[j] = __double_as_longlong(v);
            }
            if (SLICE) {
                const int srow = (part ? a.pt[1].srow0 : a.pt[0].srow0) + mm;
                const int *SE = part ? a.pt[1].SE : a.pt[0].SE;
                const long long sSE = part ? a.pt[1].sSE : a.pt[0].sSE;
                __nv_bfloat16 *sp = part ? a.pt[1].sp : a.pt[0].sp;
                const int E = SE[(long long)b * sSE + srow];
                const unsigned long long bound = (unsigned long long)(E + 1023) << 52;  // bit pattern of 2^E
                bool over = false;
                __nv_bfloat16 *dst = sp + ((long long)b * a.srows + srow) * a.sldp + a.skoff + nb;
                // eight K positions per 16-byte store: each lane writes its own plane row,
                // so the stores cannot coalesce across lanes; wider stores halve the
                // sector writes
                long long v8[OCOL];
#pragma unroll
                for (int jj = 0; jj < OCOL; ++jj) {
                    over |= ((unsigned long long)h[jj] & 0x7FFFFFFFFFFFFFFFull) >= bound;
                    v8[jj] = oz_fixed(__longlong_as_double(h[jj]), E);
                }
#pragma unroll
                for (int p = 0; p < OZ_S; ++p)
                    *reinterpret_cast<uint4 *>(dst + (long long)p * a.splane_stride) = oz_pair8(v8, p);
                if (over) atomicOr(a.flag, FLAG_NUMERICAL);
            }
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OTMEM) : "memory");
}

// ---------------------------------------------------------------------------
// The slice products of a whole stabilisation block for N <= 64: X^T <- X^T D E
// acts on every row of X^T alone, so a CTA keeps 128 rows (of one item or of
// several, the rows of all items lie one after another) for all slices, as
// digit planes in shared memory (8 x 16 KB) beside E's (8 x 8 KB).  Per slice:
// 48 MMAs into eight 64-column groups (all of tensor memory), then every
// thread combines the groups of a row's 16 columns exactly, rounds, scales by
// the next slice's D, and splits again.  No global memory and no launch
// between slices.  Bound by the integer work of combining and splitting (about
// 110 instructions per element, 16 warps) after 2.4 us of MMAs.
// Measured at 8 x 8, 64 items: 12 us per slice (15 with FP64 rounding and scaling
// in between); one FP64 GEMM launch per slice took 44 us.
constexpr int CH_N = 64, CH_THREADS = 512;
constexpr int CH_TILE_A = OBM * 128, CH_TILE_B = CH_N * 128;  // one plane: 64 BF16 (128 bytes) per row
constexpr size_t CH_SMEM = OZ_S * (CH_TILE_A + CH_TILE_B) + 1024 + 4 * OBM * 4 + CH_N * 4 + 64;

struct ChainArgs {
    const double *U;
    double *X;
    const int8_t *s;
    long long sS;
    int rows, N, M, t0, nb;
    double cu, cd;
    const __nv_bfloat16 *ep;  // E's planes
    long long eps;
    int ldp;
    const int *EE;
    int *flag;
};

// A value of the row between two products: (-1)^neg m 2^(ex - 63), 2^63 <= m <
// 2^64, or m = 0.  Scaling, the row's maximum and the splitting need no FP64
// (a warp's FP64 instruction holds the pipe for 64 cycles) and no rounding to
// 53 bits in between.
struct ChValue {
    unsigned long long m;
    int ex, neg;
};
constexpr int CH_ZERO = -(1 << 24);  // exponent of zero

__device__ __forceinline__ ChValue ch_from(double x, double d)
{
    const double y = x * d;
    const long long u = __double_as_longlong(y);
    const int ef = (int)((u >> 52) & 0x7FF);
    ChValue v;
    v.neg = u < 0;
    v.m = ef ? (((unsigned long long)u << 11) | (1ull << 63)) : 0ull;
    v.ex = ef == 0x7FF ? OZ_NONFINITE : ef ? ef - 1023 : CH_ZERO;
    return v;
}

// (h + l 2^-28) 2^e times d = dm 2^(dex - 63) (2^63 <= dm)
__device__ __forceinline__ ChValue ch_scaled(long long h, long long l, int e, unsigned long long dm, int dex)
{
    unsigned long long lo = ((unsigned long long)h << 28) + (unsigned long long)l;
    long long hi = (h >> 36) + (l >> 63) + (lo < (unsigned long long)l ? 1 : 0);
    ChValue v;
    v.neg = hi < 0;
    if (hi < 0) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0ull ? 1 : 0);
    }
    uint32_t t2 = (uint32_t)hi, t1 = (uint32_t)(lo >> 32), t0 = (uint32_t)lo;
    int ex = e + 95 - 28 + dex;
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (t2 == 0u) {
            t2 = t1;
            t1 = t0;
            t0 = 0u;
            ex -= 32;
        }
    const int s = __clz((int)t2);
    const unsigned long long top = ((unsigned long long)__funnelshift_l(t1, t2, s) << 32) | __funnelshift_l(t0, t1, s);
    // dm / 2^63 is in [1, 2): the product's high word is half of top dm / 2^63
    v.m = __umul64hi(top, dm);
    const int up = (int)(v.m >> 63);
    v.m <<= 1 - up;
    v.ex = t2 == 0u ? CH_ZERO : ex - s + up;
    if (e > OZ_NONFINITE / 2) v.ex = OZ_NONFINITE;
    return v;
}

// As oz_fixed; |v| < 2^E.
__device__ __forceinline__ long long ch_fixed(const ChValue &v, int E)
{
    const int r = E - v.ex + 63 - OZ_BITS;  // >= 7
    long long w = 0;
    if (r < 64) w = (long long)(((v.m >> (r - 1)) + 1ull) >> 1);
    constexpr long long bias = 64ll * (1 + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35) + (1ll << 42));
    return (v.neg ? -w : w) + bias;
}

// Shared-memory descriptor of a K-major operand of 128-byte rows with the
// 128-byte swizzle (8-row atoms of 1024 bytes).
__device__ __forceinline__ uint64_t ch_desc(uint32_t saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1u << 16) | ((uint64_t)(1024u >> 4) << 32) |
           ((uint64_t)1u << 46) | ((uint64_t)2u << 61);
}

__global__ void __launch_bounds__(CH_THREADS, 1) k_oz_chain(ChainArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sA = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sB = sA + OZ_S * CH_TILE_A;
    int *s_ef = (int *)(sB + OZ_S * CH_TILE_B);  // [4][128]
    int *s_ee = s_ef + 4 * OBM;                  // [64]
    uint64_t *done = (uint64_t *)(s_ee + CH_N);
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // E's planes, 16 bytes at a time, in the swizzled layout; rows beyond N zero
    for (int e = tid; e < OZ_S * CH_N * 8; e += CH_THREADS) {
        const int p = e >> 9, r = (e >> 3) & 63, ch = e & 7;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < a.N) v = *reinterpret_cast<const uint4 *>(a.ep + p * a.eps + (long long)r * a.ldp + 8 * ch);
        *reinterpret_cast<uint4 *>(sB + p * CH_TILE_B + r * 128 + ((ch ^ (r & 7)) << 4)) = v;
    }
    if (tid < CH_N) s_ee[tid] = tid < a.N ? a.EE[tid] : 0;
    // this thread's row (tensor-memory lane quarter warp % 4) and 16 columns
    const int row = (warp & 3) * 32 + lane, cg = warp >> 2, n0 = 16 * cg;
    const int g = blockIdx.x * OBM + row;
    const bool live = g < a.rows;
    const int8_t *s = a.s + (live ? (long long)(g / a.N) * a.sS : 0) + n0;
    auto signs = [&](int slice) {  // bit j: spin of column n0 + j is up
        uint32_t m = 0;
        const int8_t *sl = s + (long long)slice * a.N;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (live && n0 + j < a.N && sl[j] > 0) m |= 1u << j;
        return m;
    };
    ChValue x[16];
    int slice = a.t0;
    uint32_t up = signs(slice);
#pragma unroll
    for (int j = 0; j < 16; ++j)
        x[j] = ch_from(live && n0 + j < a.N ? a.U[(long long)g * a.N + n0 + j] : 0.0, (up >> j) & 1u ? a.cu : a.cd);
    const unsigned long long mu = ((unsigned long long)__double_as_longlong(a.cu) << 11) | (1ull << 63),
                             md = ((unsigned long long)__double_as_longlong(a.cd) << 11) | (1ull << 63);
    const int eu = ((__double2hiint(a.cu) >> 20) & 0x7FF) - 1023, ed = ((__double2hiint(a.cd) >> 20) & 0x7FF) - 1023;
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    for (int j = 0; j < a.nb; ++j) {
        // split the row: its exponent over the four column groups, then the digits
        int exm = CH_ZERO;
#pragma unroll
        for (int k = 0; k < 16; ++k) exm = max(exm, x[k].ex);
        s_ef[cg * OBM + row] = exm;
        if (!__syncthreads_and(ok)) break;  // also: every thread has read the previous slice's tensor memory
        exm = max(max(s_ef[row], s_ef[OBM + row]), max(s_ef[2 * OBM + row], s_ef[3 * OBM + row]));
        // the exponent of a row of zeros is of no account; of one with an
        // infinity or a NaN, OZ_NONFINITE (all of its other digits are then zero)
        const int Ei = exm >= OZ_NONFINITE ? OZ_NONFINITE : exm == CH_ZERO ? 0 : exm + 1;
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) {
            if (n0 >= a.N) break;  // no MMA reads these columns
            long long v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = ch_fixed(x[8 * c8 + k], Ei);
            uint8_t *dst = sA + row * 128 + (((2 * cg + c8) ^ (row & 7)) << 4);
#pragma unroll
            for (int p = 0; p < OZ_S; ++p)
                *reinterpret_cast<uint4 *>(dst + p * CH_TILE_A) = oz_pair8(v, p);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fence_before();
        __syncthreads();
        if (tid == 0) {
            fence_after();
            const uint32_t ua = smem_u32(sA), ub = smem_u32(sB);
            for (int k = 0; k < (a.N + 15) / 16; ++k)
#pragma unroll
                for (int p = 0; p < OZ_S; ++p)
#pragma unroll
                    for (int q = 0; q < OZ_S - p; q += 4) {
                        // A's plane p times up to four of B's planes q.., into groups p + q..
                        const int nq = OZ_S - p - q < 4 ? OZ_S - p - q : 4;
                        mma_bf16(tmem + (uint32_t)((p + q) * CH_N), ch_desc(ua + p * CH_TILE_A + k * 32),
                                 ch_desc(ub + q * CH_TILE_B + k * 32), oz_idesc(CH_N * nq), (k != 0 || p != 0) ? 1u : 0u);
                    }
            mma_commit(done);
        }
        if (++slice == a.M) slice = 0;
        const bool last = j == a.nb - 1;
        up = last ? 0u : signs(slice);
        ok = mbar_wait(done, j & 1, a.flag);
        fence_after();
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)n0;
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) {
            if (n0 + 8 * c8 >= a.N) break;  // x stays zero
            // Group sums below 2^22 (64 products of at most 2^16, all at that bound
            // only for a constant row of exp(-dtau K)): with 1.5 2^23 added, the bits
            // of the FP32 are the integer plus a constant.  Two neighbouring groups
            // fit 32 bits (2^29), so one wide multiply-add joins four.
            long long hl[2][8];
#pragma unroll
            for (int gg = 0; gg < OZ_G; gg += 4) {
                uint32_t r[4][8];
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld8_nowait(lane_base + (uint32_t)((gg + q) * CH_N + 8 * c8), r[q]);
                tmem_wait_ld8x4(r[0], r[1], r[2], r[3]);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    uint32_t b[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) b[q] = __float_as_uint(__uint_as_float(r[q][k]) + 12582912.0f);
                    const int w0 = (int)((b[0] << 7) + b[1] - 0x4B400000u * 129u), w1 = (int)((b[2] << 7) + b[3] - 0x4B400000u * 129u);
                    hl[gg >> 2][k] = (long long)w0 * (1 << 14) + w1;
                }
            }
            if (last) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int n = n0 + 8 * c8 + k;
                    if (ok && live && n < a.N) a.X[(long long)g * a.N + n] = oz_round(hl[0][k], hl[1][k], Ei + s_ee[n] - 37);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const bool u = (up >> (8 * c8 + k)) & 1u;
                    x[8 * c8 + k] = ch_scaled(hl[0][k], hl[1][k], Ei + s_ee[n0 + 8 * c8 + k] - 37, u ? mu : md, u ? eu : ed);
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

struct OzWs {
    int ldp;
    long long plane_stride;
    __nv_bfloat16 *planes;  // digit planes of the Gram operand; in the Cholesky-QR, of Q's finished rows
    int *E;
    CUtensorMap mapA, mapB;
    // Cholesky-QR: digit planes of R's finished rows, stored by column of R
    // (plane row j holds R[l][j] at K position l), with fixed exponents ER
    // (bounds from the Gram diagonal) and EQ = 1 for Q's rows (|Q_lj| < 2)
    __nv_bfloat16 *rplanes;
    int *ER, *EQ;
    int *ER1;  // column bounds of the first pass's R (kept for R = R2 R1)
    CUtensorMap mapRA, mapRB;  // 128-row and 32-row boxes
    // Cholesky-QR panels: digit planes of T = R_kk^-T (32 x 32 per item) and
    // their row exponents; column exponents of the unsolved panel rows of Y
    // (EPY) and of W (EPW)
    __nv_bfloat16 *tplanes;
    long long tplane_stride;
    int *ET, *EPY, *EPW;
    CUtensorMap mapT;
    CUtensorMap mapAS, mapRAS;  // planes and rplanes with the items' rows one after another (128-row boxes)
    // rank-32 updates: digit planes of the N x 32 left factors (two matrices
    // per item), their row exponents; in the context's R2 and Vg buffers, which only
    // a stabilisation uses (1032 N bytes per item of 16 N^2)
    __nv_bfloat16 *lplanes[2];
    long long lplane_stride;
    int *EL[2];
    CUtensorMap mapL[2];
    // digit planes of exp(-dtau K) and exp(+dtau K) (built on first use)
    void *emem;
    long long eplane_stride;
    __nv_bfloat16 *eplanes[2];
    int *EE[2];
    CUtensorMap mapE[2];
    int e_tried;
    int num_sms;
};

bool encode4(CUtensorMap *map, void *ptr, int ldp, int rows, int batch, int box_rows)
{
    auto fn = get_encode();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)ldp, (cuuint64_t)rows, (cuuint64_t)batch, (cuuint64_t)OZ_S};
    cuuint64_t strides[3] = {(cuuint64_t)ldp * 2, (cuuint64_t)ldp * rows * 2, (cuuint64_t)ldp * rows * batch * 2};
    cuuint32_t box[4] = {(cuuint32_t)OKE, (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace

int oz_prepare(sldqmc_ctx *c)
{
    c->oz_ws = nullptr;
    // Below one 128-row tile only the FP64 mode's products with a propagator
    // shared by all items (slice products, wraps), whose rows are stacked
    const bool small = c->N < OBM;
    if (small && c->p.prec != SLDQMC_FP64) return SLDQMC_OK;
    OzWs *w = new OzWs();
    const int N = c->N;
    const int rows = c->cap * N < OBM ? OBM : c->cap * N;  // no fewer than a tensor-map box
    w->ldp = (N + 63) / 64 * 64;
    w->plane_stride = (long long)rows * w->ldp;
    const size_t pbytes = (size_t)OZ_S * w->plane_stride * sizeof(__nv_bfloat16);
    const size_t ebytes = sizeof(int) * (size_t)c->cap * N;
    w->tplane_stride = (long long)c->cap * 32 * 32;
    const size_t tbytes = (size_t)OZ_S * w->tplane_stride * sizeof(__nv_bfloat16);
    const size_t tebytes = sizeof(int) * (size_t)c->cap * 32;
    w->lplane_stride = (long long)c->cap * N * 32;
    const size_t lbytes = (size_t)OZ_S * w->lplane_stride * sizeof(__nv_bfloat16);
    const size_t eoff = 2 * pbytes + tbytes;  // the int arrays follow the planes
    const size_t total = eoff + 5 * ebytes + tebytes + sizeof(int) * N;
    // The FP64 mode also runs without this workspace (on the FP64 pipe), so
    // there it is taken only when it leaves most of the free memory.
    const bool optional = c->p.prec == SLDQMC_FP64;
    if (optional) {
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || 3.0 * (double)total > (double)free_b) {
            cudaGetLastError();
            delete w;
            return SLDQMC_OK;
        }
    }
    void *mem = nullptr;
    if (cudaMalloc(&mem, total) != cudaSuccess) {
        cudaGetLastError();
        delete w;
        return optional ? SLDQMC_OK : SLDQMC_ERR_OOM;
    }
    w->planes = (__nv_bfloat16 *)mem;
    w->rplanes = (__nv_bfloat16 *)((uint8_t *)mem + pbytes);
    w->tplanes = (__nv_bfloat16 *)((uint8_t *)mem + 2 * pbytes);
    uint8_t *left = (uint8_t *)c->buf[7];  // 64 cap N^2 bytes into the workspace: aligned for TMA
    for (int f = 0; f < 2; ++f) {
        w->lplanes[f] = small ? nullptr : (__nv_bfloat16 *)(left + f * lbytes);
        w->EL[f] = small ? nullptr : (int *)(left + 2 * lbytes + f * ebytes);
    }
    w->E = (int *)((uint8_t *)mem + eoff);
    w->ER = w->E + (size_t)c->cap * N;
    w->ER1 = w->ER + (size_t)c->cap * N;
    w->EPY = w->ER1 + (size_t)c->cap * N;
    w->EPW = w->EPY + (size_t)c->cap * N;
    w->ET = w->EPW + (size_t)c->cap * N;
    w->EQ = w->ET + (size_t)c->cap * 32;
    w->emem = nullptr;
    w->e_tried = 0;
    cudaMemsetAsync(mem, 0, eoff + 5 * ebytes + tebytes, c->st);  // zero pads: never written
    {
        std::vector<int> ones((size_t)N, 1);
        if (cudaMemcpyAsync(w->EQ, ones.data(), sizeof(int) * N, cudaMemcpyHostToDevice, c->st) != cudaSuccess ||
            cudaStreamSynchronize(c->st) != cudaSuccess) {
            cudaFree(mem);
            delete w;
            return SLDQMC_ERR_CUDA;
        }
    }
    bool mapped = encode4(&w->mapAS, w->planes, w->ldp, rows, 1, OBM) && encode4(&w->mapRAS, w->rplanes, w->ldp, rows, 1, OBM);
    if (!small)
        mapped = mapped && encode4(&w->mapA, w->planes, w->ldp, N, c->cap, OBM) &&
                 encode4(&w->mapB, w->planes, w->ldp, N, c->cap, OBN) &&
                 encode4(&w->mapRA, w->rplanes, w->ldp, N, c->cap, OBM) &&
                 encode4(&w->mapRB, w->rplanes, w->ldp, N, c->cap, OBN) &&
                 encode4(&w->mapT, w->tplanes, 32, 32, c->cap, OBN) &&
                 encode4(&w->mapL[0], w->lplanes[0], 32, N, c->cap, OBN) &&
                 encode4(&w->mapL[1], w->lplanes[1], 32, N, c->cap, OBN);
    if (!mapped) {
        cudaFree(mem);
        delete w;
        return SLDQMC_ERR_CUDA;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&w->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || w->num_sms < 1)
        w->num_sms = 148;
    const int sh = (int)oz_smem_bytes();
    cudaFuncSetAttribute(k_oz_gemm<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh);
    cudaFuncSetAttribute(k_oz_gemm<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh);
    cudaFuncSetAttribute(k_oz_gemm<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh);
    cudaFuncSetAttribute(k_oz_gemm<false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh);
    cudaFuncSetAttribute(k_oz_gemm<false, false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sh);
    cudaFuncSetAttribute(k_oz_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CH_SMEM);
    c->oz_ws = w;
    return SLDQMC_OK;
}

void oz_release(sldqmc_ctx *c)
{
    OzWs *w = (OzWs *)c->oz_ws;
    if (!w) return;
    cudaFree(w->planes);
    cudaFree(w->emem);
    delete w;
    c->oz_ws = nullptr;
}

namespace {

OzPart oz_part(int M, int arow0, const int *EA, long long sEA, const int *EB, long long sEB, double *C, long long sC,
               int ldc)
{
    OzPart p{};
    p.M = M;
    p.arow0 = arow0;
    p.EA = EA;
    p.sEA = sEA;
    p.EB = EB;
    p.sEB = sEB;
    p.C = C;
    p.sC = sC;
    p.ldc = ldc;
    return p;
}

// Rows of one matrix (or of two, X2 into rplanes and E2) split with their own maxima.
void oz_slice_rows(sldqmc_ctx *c, const double *X, const double *X2, int *E2, long long sX, int rows, int cols, int ld, int B,
                   const int8_t *sk = nullptr, double cu = 1.0, double cd = 1.0)
{
    OzWs *w = (OzWs *)c->oz_ws;
    OzRows r{{X, X2}, {w->planes, w->rplanes}, {w->E, E2}, sk, (long long)c->M * c->N, cu, cd};
    const dim3 grid((rows + 7) / 8, B, X2 ? 2 : 1);
    prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_slice");
    if (sk) k_oz_slice<true><<<grid, 256, 0, c->st>>>(r, sX, rows, cols, ld, c->N, w->ldp, w->plane_stride);
    else k_oz_slice<false><<<grid, 256, 0, c->st>>>(r, sX, rows, cols, ld, c->N, w->ldp, w->plane_stride);
    prof_end(c);
    c->launches++;
}

template <bool UPPER>
int oz_grid(const OzWs *w, const OzArgs &a)
{
    const int tiles = oz_part_tiles<UPPER>(a, 0) + (a.nparts > 1 ? oz_part_tiles<UPPER>(a, 1) : 0);
    return tiles < w->num_sms ? tiles : w->num_sms;
}

}  // namespace

// W = X X^T (rows of X: row stride N, batch stride sX); W row stride ldw,
// batch stride sW.  Tiles on or above the diagonal are written in full.
void oz_gram(sldqmc_ctx *c, const double *X, long long sX, double *W, long long sW, int ldw, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    oz_slice_rows(c, X, nullptr, nullptr, sX, N, N, N, B);
    OzArgs a{};
    a.pt[0] = oz_part(N, 0, w->E, N, w->E, N, W, sW, ldw);
    a.nparts = 1;
    a.Nn = N;
    a.batch = B;
    a.nk = w->ldp / OKE;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, (double)N * N * (N + 1) * B, "oz_gram");
    k_oz_gemm<true, false>
        <<<oz_grid<true>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapA, w->mapA, w->mapB, w->mapB, a);
    prof_end(c);
    c->launches++;
}

// Left-looking Cholesky-QR of W = X X^T (row stride N, item stride sW) that
// forms Q^T = R^-T X^T in Y (row stride N, item stride N*N): before the rows
// k0..k0+kb the products of the finished rows kstart..k0-1 are subtracted
// from them (the caller runs it once per block of up to 128 rows with all
// earlier rows, then per 32-row panel with the block's own finished rows),
//   Y[k0+r][n]    -= sum_{l<k0} Q^T[l][n] R[l][k0+r],
//   W[k0+r][k0+n] -= sum_{l<k0} R[l][k0+n] R[l][k0+r],
// FP64-accurate on the tensor cores in one launch of two parts (the product
// computed with rows n and columns r, stored transposed so that a warp's
// stores are contiguous); the panel then splits its finished rows of R and
// Q^T into K-block k0/32 of the digit planes.  oz_chol_begin fixes the
// exponents of R's columns from W's diagonal.
void oz_chol_begin(sldqmc_ctx *c, const double *W, long long sW, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_col_exponents");
    k_oz_col_exponents<<<dim3((N + 255) / 256, B), 256, 0, c->st>>>(W, sW, N, N, w->ER);
    prof_end(c);
    c->launches++;
}

void oz_chol_update(sldqmc_ctx *c, int k0, int kb, int kstart, double *W, long long sW, double *Y, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    OzArgs a{};
    // rows n of the parts: columns of Q^T, columns k0.. of R
    a.pt[0] = oz_part(N, 0, w->EQ, 0, w->ER + k0, N, Y + (long long)k0 * N, c->nn, N);
    a.pt[1] = oz_part(N - k0, k0, w->ER + k0, N, w->ER + k0, N, W + (long long)k0 * N + k0, sW, N);
    a.nparts = 2;
    a.Nn = kb;
    a.brow0 = k0;
    a.batch = B;
    a.kA0 = kstart;
    a.kB0 = kstart;
    a.nk = (k0 - kstart) / OKE;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * (2 * N - k0) * kb * (k0 - kstart) * B,
               kstart ? "oz_chol_update_inner" : "oz_chol_update");
    k_oz_gemm<false, true, true>
        <<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapA, w->mapRA, w->mapRB, w->mapRB, a);
    prof_end(c);
    c->launches++;
}

// The panel of rows k0..k0+kb once its rows of W and Y are up to date: the
// unsolved rows are split with each column's own maximum, the diagonal block
// is factored and inverted (FP64, one CTA per item), and
//   Y[k0+n][j] = sum_l T[n][l] Y[k0+l][j]   (all j: the rows of Q^T),
//   R[k0+n][j] = sum_l T[n][l] W[k0+l][j]   (j >= k0 + kb),
// run FP64-accurate on the tensor cores (K = 32, one exactly accumulated
// chunk) in place of the triangular solves, in one launch of two parts whose
// epilogue also splits the finished rows into K-block k0/32 of the digit
// planes (fixed exponents: EQ for Q^T, ER for R) for the later panels.
void oz_chol_panel(sldqmc_ctx *c, int k0, int kb, const double *W, long long sW, double *Y, double *R, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    const int j0 = k0 + kb, nW = N - j0;
    OzPanelSlice sl{};
    sl.src[0] = Y + (long long)k0 * N;
    sl.sS[0] = c->nn;
    sl.j0[0] = 0;
    sl.planes[0] = w->planes;
    sl.E[0] = w->EPY;
    sl.nb0 = (N + 31) / 32;
    sl.src[1] = W + (long long)k0 * N;
    sl.sS[1] = sW;
    sl.j0[1] = j0;
    sl.planes[1] = w->rplanes;
    sl.E[1] = w->EPW;
    const OzPanelPrep f{W, sW, R, c->nn, N, k0, kb, w->tplanes, w->tplane_stride, w->ET};
    prof_begin(c, SLDQMC_KC_PANEL_F64, (double)B * 2.0 * kb * kb * kb / 3.0, "oz_panel_prep");
    const dim3 grid(1 + sl.nb0 + (nW + 31) / 32, B);
    if (c->p.prec == SLDQMC_FP64) k_oz_panel_prep<true><<<grid, 256, 0, c->st>>>(f, sl, w->plane_stride, w->ldp, c->d_flag);
    else k_oz_panel_prep<false><<<grid, 256, 0, c->st>>>(f, sl, w->plane_stride, w->ldp, c->d_flag);
    prof_end(c);
    OzArgs a{};
    a.pt[0] = oz_part(N, 0, w->EPY, N, w->ET, 32, Y + (long long)k0 * N, c->nn, N);
    a.pt[0].sp = w->planes;
    a.pt[0].SE = w->EQ;
    a.pt[0].sSE = 0;
    a.pt[0].srow0 = 0;
    a.pt[1] = oz_part(nW, j0, w->EPW + j0, N, w->ET, 32, R + (long long)k0 * N + j0, c->nn, N);
    a.pt[1].sp = w->rplanes;
    a.pt[1].SE = w->ER;
    a.pt[1].sSE = N;
    a.pt[1].srow0 = j0;
    a.nparts = nW > 0 ? 2 : 1;
    a.Nn = kb;
    a.brow0 = 0;
    a.batch = B;
    a.nk = 1;
    a.kA0 = k0;
    a.kB0 = 0;
    a.splane_stride = w->plane_stride;
    a.sldp = w->ldp;
    a.srows = N;
    a.skoff = k0;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * (N + nW) * kb * kb * B, "oz_chol_panel");
    k_oz_gemm<false, false, true, true>
        <<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapA, w->mapRA, w->mapT, w->mapT, a);
    prof_end(c);
    c->launches += 2;
}

namespace {

// Rank-32 updates C[i][j] -= sum_l L[i][l] R[l][j] of up to two column ranges
// (L, R and C in one matrix of row stride lda, item stride sA), FP64-accurate on the tensor cores: the rows of L (rows x
// kb, row stride ldl) and the columns of R each split with their own maximum
// (K = kb <= 32, one exactly accumulated chunk).  The product is computed
// with rows j and columns i and stored transposed, so that a warp's 32 reads
// and writes of C are contiguous.
struct RankPart {
    const double *R;  // kb x cols, columns j0 .. j0 + cols - 1 of a matrix whose row 0 starts at R
    int j0, cols;
    double *C;        // element (0, j0)
};

void oz_rank_update(sldqmc_ctx *c, const double *L, const RankPart *pt, int nparts, int rows, int kb, int lda, long long sA,
                    int B, const char *site)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    {
        OzRows r{{L, nullptr}, {w->lplanes[0], nullptr}, {w->EL[0], nullptr}, nullptr, 0, 1.0, 1.0};
        prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_slice");
        k_oz_slice<false><<<dim3((rows + 7) / 8, B), 256, 0, c->st>>>(r, sA, rows, kb, lda, N, 32, w->lplane_stride);
        prof_end(c);
    }
    OzPanelSlice sl{};
    OzArgs a{};
    double cols = 0.0;
    __nv_bfloat16 *pl[2] = {w->rplanes, w->planes};
    int *ep[2] = {w->EPW, w->EPY};
    for (int p = 0; p < nparts; ++p) {
        sl.src[p] = pt[p].R;
        sl.sS[p] = sA;
        sl.j0[p] = pt[p].j0;
        sl.planes[p] = pl[p];
        sl.E[p] = ep[p];
        a.pt[p] = oz_part(pt[p].cols, pt[p].j0, ep[p] + pt[p].j0, N, w->EL[0], N, pt[p].C, sA, lda);
        cols += pt[p].cols;
    }
    const int nb0 = (pt[0].cols + 31) / 32, nb1 = nparts > 1 ? (pt[1].cols + 31) / 32 : 0;
    sl.nb0 = nb0;
    prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_slice_panel");
    k_oz_slice_panel<<<dim3(nb0 + nb1, B), 256, 0, c->st>>>(sl, N, lda, kb, 0, w->plane_stride, w->ldp, c->d_flag);
    prof_end(c);
    a.nparts = nparts;
    a.Nn = rows;
    a.batch = B;
    a.nk = 1;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * rows * cols * kb * B, site);
    k_oz_gemm<false, true, true><<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(
        w->mapRA, w->mapA, w->mapL[0], w->mapL[0], a);
    prof_end(c);
    c->launches += 3;
}

// Digit planes of exp(-dtau K) and exp(+dtau K), on first use; false when
// there is no room for them, or while the stream is being captured and they are
// not there yet (the callers then stay on the FP64 pipe).
bool oz_e_planes(sldqmc_ctx *c)
{
    OzWs *w = (OzWs *)c->oz_ws;
    if (w->e_tried) return w->emem != nullptr;
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(c->st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    w->e_tried = 1;
    const int N = c->N;
    const int erows = N < OBN ? OBN : N;
    w->eplane_stride = (long long)erows * w->ldp;
    const size_t pb = (size_t)OZ_S * w->eplane_stride * sizeof(__nv_bfloat16);
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || 6.0 * (double)pb > (double)free_b ||
        cudaMalloc(&w->emem, 2 * pb + 2 * sizeof(int) * N) != cudaSuccess) {
        cudaGetLastError();
        w->emem = nullptr;
        return false;
    }
    cudaMemsetAsync(w->emem, 0, 2 * pb, c->st);
    for (int e = 0; e < 2; ++e) {
        w->eplanes[e] = (__nv_bfloat16 *)((uint8_t *)w->emem + e * pb);
        w->EE[e] = (int *)((uint8_t *)w->emem + 2 * pb) + e * N;
        if (!encode4(&w->mapE[e], w->eplanes[e], w->ldp, erows, 1, OBN)) {
            cudaFree(w->emem);  // waits for the memset
            w->emem = nullptr;
            return false;
        }
    }
    OzRows r{{c->d_E, c->d_Einv}, {w->eplanes[0], w->eplanes[1]}, {w->EE[0], w->EE[1]}, nullptr, 0, 1.0, 1.0};
    k_oz_slice<false><<<dim3((N + 7) / 8, 1, 2), 256, 0, c->st>>>(r, 0, N, N, N, N, w->ldp, w->eplane_stride);
    c->launches++;
    return true;
}

}  // namespace

// Trailing update of the finalisation's blocked LU, A[i][j] -= sum_l L[i][k0+l]
// U[k0+l][j] for i, j >= k0 + kb; with rhs also for the right-hand side's
// columns N..2N-1.
void oz_lu_update(sldqmc_ctx *c, double *A, long long sA, int lda, int k0, int kb, int B, int rhs)
{
    const int N = c->N, j0 = k0 + kb;
    double *low = A + (long long)j0 * lda;  // row k0 + kb
    const RankPart pt[2] = {{A + (long long)k0 * lda, j0, N - j0, low + j0},
                            {A + (long long)k0 * lda + N, 0, N, low + N}};
    oz_rank_update(c, low + k0, pt, rhs ? 2 : 1, N - j0, kb, lda, sA, B, "oz_lu_update");
}

// Back substitution: the rows above k0 of the right-hand side lose the share
// of its solved rows k0..k0+kb, Y[i][j] -= sum_l U[i][k0+l] X[k0+l][j].
void oz_back_update(sldqmc_ctx *c, double *A, long long sA, int lda, int k0, int kb, int B)
{
    const int N = c->N;
    const RankPart pt = {A + (long long)k0 * lda + N, 0, N, A + N};
    oz_rank_update(c, A + k0, &pt, 1, k0, kb, lda, sA, B, "oz_back_update");
}

namespace {

// Forms the pairs of a block of flips at every row and column and splits them
// for the rank-32 product: blocks of even x the left vectors u_n at 128 rows
// (thread = row, its 32 values one plane row of lplanes), blocks of odd x the
// right vectors v_n at 128 columns.  u_n = coef_n (G[:, i_n] - sum_m u_m
// v_m[i_n]), v_n = e - (G[i_n, :] - sum_m u_m[i_n] v_m): 496 dependent-by-row FMAs
// per thread on the FP64 pipe, which bound it (17 us per wave; one wave up to
// 76 x 128 rows of both flavours).
struct PairArgs {
    const double *G[2];
    const FlipPairs *pairs;
    __nv_bfloat16 *lp[2], *rp[2];
    int *EL[2], *ER[2];
    long long lps, rps;
    int N, ldp;
};

__global__ void __launch_bounds__(128) k_flip_pairs(PairArgs a)
{
    __shared__ double T[32][32], cf[32];
    __shared__ int site[32];
    const int b = blockIdx.y, f = blockIdx.z, right = blockIdx.x & 1, tid = threadIdx.x;
    const FlipPairs &p = a.pairs[b];
    const int n = p.n, N = a.N;
    for (int e = tid; e < 32 * 32; e += 128) (&T[0][0])[e] = right ? (&p.L[f][0][0])[e] : (&p.X[f][0][0])[e];
    if (tid < 32) {
        cf[tid] = p.coef[f][tid];
        site[tid] = p.site[tid];
    }
    __syncthreads();
    const int r = (blockIdx.x >> 1) * 128 + tid;
    if (r >= N) return;
    const double *G = (f ? a.G[1] : a.G[0]) + (long long)b * N * N;
    double x[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = k < n ? (right ? G[(long long)site[k] * N + r] : G[(long long)r * N + site[k]]) : 0.0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (k < n) {
            double c = x[k];
#pragma unroll
            for (int m = 0; m < k; ++m) c -= x[m] * (right ? T[k][m] : T[m][k]);
            x[k] = right ? (r == site[k] ? 1.0 : 0.0) - c : cf[k] * c;
        }
    }
    unsigned long long mx = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(x[k]) & 0x7FFFFFFFFFFFFFFFull;
        mx = u > mx ? u : mx;
    }
    const int ef_max = (int)(mx >> 52);
    const int E = oz_exponent(ef_max);
    const long long row = (long long)b * N + r;
    (right ? a.ER[f] : a.EL[f])[row] = E;
    __nv_bfloat16 *dst = right ? a.rp[f] + row * a.ldp : a.lp[f] + row * 32;
    const long long ps = right ? a.rps : a.lps;
#pragma unroll
    for (int k8 = 0; k8 < 32; k8 += 8) {
        long long v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = oz_fixed(x[k8 + k], E);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q) *reinterpret_cast<uint4 *>(dst + q * ps + k8) = oz_pair8(v, q);
    }
}

}  // namespace

// G_f -= sum_n u_n v_n of both flavours for one block of flips.
void oz_delayed_update(sldqmc_ctx *c, double *const *G, const FlipPairs *pairs, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    PairArgs p{{G[0], G[1]}, pairs, {w->lplanes[0], w->lplanes[1]}, {w->rplanes, w->planes}, {w->EL[0], w->EL[1]},
               {w->EPW, w->EPY}, w->lplane_stride, w->plane_stride, N, w->ldp};
    prof_begin(c, SLDQMC_KC_LOCAL, 0.0, "flip_pairs");
    k_flip_pairs<<<dim3(2 * ((N + 127) / 128), B, 2), 128, 0, c->st>>>(p);
    prof_end(c);
    OzArgs a{};
    a.pt[0] = oz_part(N, 0, w->EPW, N, w->EL[0], N, G[0], c->nn, N);
    a.pt[1] = oz_part(N, 0, w->EPY, N, w->EL[1], N, G[1], c->nn, N);
    a.nparts = 2;
    a.Nn = N;
    a.batch = B;
    a.nk = 1;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * 2.0 * N * N * 32 * B, "oz_delayed_update");
    k_oz_gemm<false, true, true><<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(
        w->mapRA, w->mapA, w->mapL[0], w->mapL[1], a);
    prof_end(c);
    c->launches += 2;
}

bool oz_have_e(sldqmc_ctx *c) { return c->oz_ws && oz_e_planes(c); }

// A product with a propagator on the tensor cores is two launches of about
// 5 us each at least, one of the FP64 pipe 2 N^3 B / 1.1e12 s but no less than
// 8 us: below 128 sites (where an item fills no tile of its own) the tensor
// cores take it from N^3 B = 8e6 (14 us of the FP64 pipe) on.  Measured at 8 x
// 8, 64 chains, both flavours: 2 x 44 us against 10 + 15 us.
bool oz_worth(const sldqmc_ctx *c, int times)
{
    return c->N >= OBM || (double)c->N * c->N * c->N * c->plan_cap * times >= 8e6;
}

bool oz_match(const sldqmc_ctx *c, sldqmc_ctx *t)
{
    const OzWs *w = (const OzWs *)c->oz_ws;
    OzWs *v = (OzWs *)t->oz_ws;
    if (!w) {
        oz_release(t);
        return true;
    }
    if (!v) return false;
    if (c->p.prec != SLDQMC_FP64) return true;  // propagator planes serve the wraps alone, on the context
    if (!w->emem && v->emem) {
        cudaFree(v->emem);
        v->emem = nullptr;
    }
    return !w->emem == !v->emem;
}

bool oz_full(const sldqmc_ctx *c) { return c->oz_ws && c->N >= OBM; }

bool oz_chain_fits(const sldqmc_ctx *c) { return c->N <= CH_N; }

// X^T_out = U^T D_t0 E D_t0+1 E ... for nb slices (N <= 64), one launch.
void oz_chain_block(sldqmc_ctx *c, const double *Ut, const int8_t *d_s, int B, double cu, double cd, int t0, int nb,
                    double *Xt_out)
{
    OzWs *w = (OzWs *)c->oz_ws;
    ChainArgs a{Ut, Xt_out, d_s, (long long)c->M * c->N, B * c->N, c->N, c->M, t0, nb, cu, cd, w->eplanes[0],
                w->eplane_stride, w->ldp, w->EE[0], c->d_flag};
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * c->N * c->N * c->N * nb * B, "oz_chain");
    k_oz_chain<<<(a.rows + OBM - 1) / OBM, CH_THREADS, CH_SMEM, c->st>>>(a);
    prof_end(c);
    c->launches++;
}

// FP64-accurate slice product X^T D E for B items into Xt (which may be X
// itself): the rows of X^T D split with their own maxima against E's planes.
// The rows of all items lie one after another, so a 128-row tile may span
// items and only the last tile is ragged.
void oz_slice_product(sldqmc_ctx *c, const double *X, const int8_t *sk, double cu, double cd, double *Xt, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    oz_slice_rows(c, X, nullptr, nullptr, c->nn, N, N, N, B, sk, cu, cd);
    OzArgs a{};
    a.pt[0] = oz_part(B * N, 0, w->E, 0, w->EE[0], 0, Xt, c->nn, N);
    a.nparts = 1;
    a.Nn = N;
    a.batch = 1;
    a.b_shared = 1;
    a.stack = N;
    a.nk = w->ldp / OKE;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, 2.0 * N * N * N * B, "oz_slice_product");
    k_oz_gemm<false, false>
        <<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapAS, w->mapAS, w->mapE[0], w->mapE[0], a);
    prof_end(c);
    c->launches++;
}

// dst_f = P src_f P^-1 for both flavours f (B items each), with P = E (inv =
// 0) or E^-1 (inv = 1); with a field slice s, row i and column j of dst_f are
// scaled by d_i / d_j (d_f = cu[f] where s > 0, cd[f] otherwise).  T = src P^-1
// is stored transposed, so that its columns are the rows of the second
// product dst^T = T^T P.
void oz_similarity(sldqmc_ctx *c, const double *const *src, double *const *T, double *const *dst, int inv,
                   const int8_t *s, const double (*ex)[2], int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    for (int k = 0; k < 2; ++k) {
        const int e = k == 0 ? !inv : inv;  // E^-1 first in the wrap
        const double *const *in = k == 0 ? src : T;
        double *const *out = k == 0 ? T : dst;
        oz_slice_rows(c, in[0], in[1], w->EPW, c->nn, N, N, N, B);
        OzArgs a{};
        a.pt[0] = oz_part(B * N, 0, w->E, 0, w->EE[e], 0, out[0], c->nn, N);
        a.pt[1] = oz_part(B * N, 0, w->EPW, 0, w->EE[e], 0, out[1], c->nn, N);
        a.nparts = 2;
        a.Nn = N;
        a.batch = 1;
        a.b_shared = 1;
        a.stack = N;
        a.nk = w->ldp / OKE;
        if (k == 1 && s) {
            a.sgn = s;
            a.sSgn = (long long)c->M * N;
            for (int f = 0; f < 2; ++f) {
                a.r_ud[f] = ex[f][0] / ex[f][1];
                a.r_du[f] = ex[f][1] / ex[f][0];
            }
        }
        a.flag = c->d_flag;
        prof_begin(c, SLDQMC_KC_GEMM_OZ, 4.0 * N * N * N * B, "oz_similarity");
        k_oz_gemm<false, false, true>
            <<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapAS, w->mapRAS, w->mapE[e], w->mapE[e], a);
        prof_end(c);
        c->launches++;
    }
}

// V <- T P^T V with T = D^-1 R D_p (upper triangular; R row stride N),
// FP64-accurate on the tensor cores: T's rows split with their own maxima,
// the gathered rows V[p_k] split column-wise with each column's maximum.
// Ts: an N x N FP64 scratch per item (item stride N*N).
void oz_update_V(sldqmc_ctx *c, const double *R, double *V, double *Ts, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_make_T");
    k_oz_make_T<<<dim3((N + 255) / 256, N, B), 256, 0, c->st>>>(R, c->nn, N, c->d_D, c->d_Dp, Ts);
    prof_end(c);
    oz_slice_rows(c, Ts, nullptr, nullptr, c->nn, N, N, N, B);
    prof_begin(c, SLDQMC_KC_OTHER, 0.0, "k_oz_col_max_exponents");
    k_oz_col_max_exponents<<<dim3((N + 31) / 32, B), 256, 0, c->st>>>(V, c->nn, N, N, w->ER1);
    prof_end(c);
    k_oz_slice_fixed<<<dim3((N + 31) / 32, B, (N + 31) / 32), 256, 0, c->st>>>(
        V, c->nn, N, 0, N, N, 0, w->plane_stride, N, w->ldp, w->rplanes, w->ER1, N, c->d_flag, c->d_perm, N);
    OzArgs a{};
    a.pt[0] = oz_part(N, 0, w->E, N, w->ER1, N, V, c->nn, N);
    a.nparts = 1;
    a.Nn = N;
    a.batch = B;
    a.nk = w->ldp / OKE;
    a.a_tri = 1;  // T is upper triangular: tile rows m0.. need K >= m0 only
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, (double)N * N * (N + 1) * B, "oz_update_V");
    k_oz_gemm<false, false>
        <<<oz_grid<false>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapA, w->mapA, w->mapRB, w->mapRB, a);
    prof_end(c);
    c->launches += 4;
}

// Keeps the current column bounds of R (a first Cholesky-QR pass) for the
// product R = R2 R1 after the second pass.
void oz_keep_bounds(sldqmc_ctx *c, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    cudaMemcpyAsync(w->ER1, w->ER, sizeof(int) * (size_t)B * c->N, cudaMemcpyDeviceToDevice, c->st);
}

// R = R2 R1 of the two Cholesky-QR passes (upper triangular, row stride N,
// item stride N*N; only the tiles on or above the diagonal of R are
// written), FP64-accurate on the tensor cores: R2's rows with their own
// maxima as exponents, R1's columns with the first pass's bounds.
void oz_r2r1(sldqmc_ctx *c, const double *R2, const double *R1, double *R, int B)
{
    OzWs *w = (OzWs *)c->oz_ws;
    const int N = c->N;
    oz_slice_rows(c, R2, nullptr, nullptr, c->nn, N, N, N, B);
    k_oz_slice_fixed<<<dim3((N + 31) / 32, B, (N + 31) / 32), 256, 0, c->st>>>(
        R1, c->nn, N, 0, N, N, 0, w->plane_stride, N, w->ldp, w->rplanes, w->ER1, N, c->d_flag);
    OzArgs a{};
    a.pt[0] = oz_part(N, 0, w->E, N, w->ER1, N, R, c->nn, N);
    a.nparts = 1;
    a.Nn = N;
    a.batch = B;
    a.nk = w->ldp / OKE;
    a.a_tri = 1;  // R2[m][l] = 0 for l < m and R1[l][n] = 0 for l > n
    a.b_tri = 1;
    a.flag = c->d_flag;
    prof_begin(c, SLDQMC_KC_GEMM_OZ, (double)N * N * N / 3.0 * B, "oz_r2r1");
    k_oz_gemm<true, false>
        <<<oz_grid<true>(w, a), OTHREADS, oz_smem_bytes(), c->st>>>(w->mapA, w->mapA, w->mapRB, w->mapRB, a);
    prof_end(c);
    c->launches += 2;
}

}  // namespace sldqmc
