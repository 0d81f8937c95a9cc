"""The serial part of every panel on its own: pivot reciprocals against IEEE
division, bit for bit, over random mantissas, the mantissas where the FP32 seed or
a rounding can go wrong (zeros, ones, within 2^30 of either end, the seed's
rounding boundaries) and binary exponents at both ends of the integer range and
beyond it; the Cholesky factor of 32 x 32 blocks against their exact roots
(diagonal blocks: R_jj is the correctly rounded square root, its inverse within
one unit in the last place) and against extended precision (dense blocks).  The
mixed modes' form of both, within one unit and two."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "chol32.cuh"
using namespace sldqmc;
template <bool EXACT>
__global__ void k_recip(const double *d, double *out, int n, int *flag)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double x = d[i];
    out[i] = chol_reciprocal<EXACT>(x, true, flag);
}
template <bool EXACT>
__global__ void k_chol(const double *W, double *R, double *root, int kb, int *flag)
{
    __shared__ double X[32][33], rt[32];
    __shared__ CholScratch sc;
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) X[e >> 5][e & 31] = W[blockIdx.x * 1024 + e];
    __syncthreads();
    chol32<EXACT>(X, rt, sc, kb, flag);
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) R[blockIdx.x * 1024 + e] = X[e >> 5][e & 31];
    if (threadIdx.x < kb) root[blockIdx.x * 32 + threadIdx.x] = rt[threadIdx.x];
}
extern "C" int run_recip(const double *d, double *out, int n, int *flag, int exact)
{
    if (exact) k_recip<true><<<(n + 255) / 256, 256>>>(d, out, n, flag);
    else k_recip<false><<<(n + 255) / 256, 256>>>(d, out, n, flag);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_chol(const double *W, double *R, double *root, int blocks, int threads, int kb, int *flag, int exact)
{
    if (exact) k_chol<true><<<blocks, threads>>>(W, R, root, kb, flag);
    else k_chol<false><<<blocks, threads>>>(W, R, root, kb, flag);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    from paper_1612_03804_gb300 import build
    torch.cuda.set_device(0)
    torch.zeros(1, device="cuda")
    d = tmp_path_factory.mktemp("pivots")
    (d / "probe.cu").write_text(PROBE)
    lib = str(d / "probe.so")
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", str(d / "probe.cu"), "-o", lib],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _pivots():
    rng = np.random.default_rng(5)
    m = [rng.integers(0, 2 ** 52, 1 << 20), np.arange(64), 2 ** 52 - 1 - np.arange(64),
         rng.integers(0, 2 ** 30, 1 << 14), 2 ** 52 - 1 - rng.integers(0, 2 ** 30, 1 << 14)]
    step = rng.integers(0, 2 ** 23, 1 << 14) << 29  # the seed is the mantissa rounded to 23 bits
    m += [step, step + 2 ** 28, step + 2 ** 28 - 1, step + 1]
    m = np.concatenate(m).astype(np.uint64)
    ef = rng.integers(523, 1523, m.size).astype(np.uint64)
    ends = np.array([1, 2, 521, 522, 523, 524, 1022, 1023, 1024, 1521, 1522, 1523, 1524, 2044, 2045, 2046], dtype=np.uint64)
    me = np.concatenate([m[:256], m[1 << 20:(1 << 20) + 128]])
    bits = np.concatenate([(ef << np.uint64(52)) | m, ((ends[:, None] << np.uint64(52)) | me[None, :]).ravel()])
    return bits.view(np.float64)


def test_pivot_reciprocals_are_ieee_divisions(probe):
    import torch
    d = _pivots()
    dd = torch.from_numpy(d).cuda()
    out = torch.zeros_like(dd)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert probe.run_recip(_p(dd), _p(out), ctypes.c_int(d.size), _p(flag), ctypes.c_int(1)) == 0
    got, ref = out.cpu().numpy(), 1.0 / d
    assert flag.item() == 0
    wrong = got.view(np.int64) != ref.view(np.int64)
    worst = np.abs(got.view(np.int64) - ref.view(np.int64)).max()
    assert not wrong.any(), (int(wrong.sum()), d.size, int(worst), d[wrong][:4])


def test_bad_pivots_count_as_one_and_raise_the_flag(probe):
    import torch
    for x in (0.0, -0.0, -1.5, np.inf, -np.inf, np.nan):
        dd = torch.tensor([x], dtype=torch.float64, device="cuda")
        out = torch.zeros_like(dd)
        flag = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert probe.run_recip(_p(dd), _p(out), ctypes.c_int(1), _p(flag), ctypes.c_int(1)) == 0
        assert flag.item() == 1 and out.item() == 1.0


def _chol(probe, W, threads, kb, exact=1):
    import torch
    n = W.shape[0]
    dW = torch.from_numpy(np.ascontiguousarray(W)).cuda()
    R = torch.zeros_like(dW)
    root = torch.zeros((n, 32), dtype=torch.float64, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert probe.run_chol(_p(dW), _p(R), _p(root), ctypes.c_int(n), ctypes.c_int(threads), ctypes.c_int(kb), _p(flag),
                          ctypes.c_int(exact)) == 0
    assert flag.item() == 0
    return R.cpu().numpy(), root.cpu().numpy()


@pytest.mark.parametrize("threads", [64, 128, 512])
def test_roots_of_diagonal_blocks(probe, threads):
    d = _pivots()
    d = d[(d > 1e-140) & (d < 1e140)][: 32 * 4096].reshape(-1, 32)
    W = np.zeros((d.shape[0], 32, 32))
    W[:, np.arange(32), np.arange(32)] = d
    X, root = _chol(probe, W, threads, 32)
    np.testing.assert_array_equal(root, np.sqrt(d))
    inv = X[:, np.arange(32), np.arange(32)]
    exact = 1.0 / np.sqrt(d.astype(np.longdouble))
    assert np.abs((inv - exact) / exact).max() <= 2.0 ** -52
    off = X.copy()
    off[:, np.arange(32), np.arange(32)] = 0.0
    assert np.all(off == 0.0)


@pytest.mark.parametrize("kb", [1, 7, 31, 32])
def test_factor_and_inverse_of_dense_blocks(probe, kb):
    rng = np.random.default_rng(kb)
    A = rng.standard_normal((64, kb, kb + 8)) * np.exp(rng.uniform(-3, 3, (64, kb, 1)))
    S = A @ A.transpose(0, 2, 1)
    W = np.tile(np.eye(32), (64, 1, 1))
    W[:, :kb, :kb] = np.triu(S)
    X, root = _chol(probe, W, 128, kb)
    eps = 2.0 ** -53
    for b in range(64):
        R = np.triu(X[b, :kb, :kb], 1) + np.diag(root[b, :kb])
        T = np.tril(X[b, :kb, :kb])
        den = np.sqrt(np.outer(np.diag(S[b]), np.diag(S[b])))
        assert (np.abs((R.T @ R - S[b])) / den).max() <= 4 * (kb + 4) * eps  # backward error of a Cholesky factorisation
        assert np.abs(T @ R.T - np.eye(kb)).max() <= 4 * (kb + 4) * eps * np.linalg.cond(R)


def test_mixed_mode_reciprocals_and_roots(probe):
    import torch
    d = _pivots()
    dd = torch.from_numpy(d).cuda()
    out = torch.zeros_like(dd)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert probe.run_recip(_p(dd), _p(out), ctypes.c_int(d.size), _p(flag), ctypes.c_int(0)) == 0
    assert flag.item() == 0
    assert np.abs(out.cpu().numpy().view(np.int64) - (1.0 / d).view(np.int64)).max() <= 1
    d = d[(d > 1e-140) & (d < 1e140)][: 32 * 4096].reshape(-1, 32)
    W = np.zeros((d.shape[0], 32, 32))
    W[:, np.arange(32), np.arange(32)] = d
    X, root = _chol(probe, W, 256, 32, exact=0)
    assert np.abs(root.view(np.int64) - np.sqrt(d).view(np.int64)).max() <= 2
    exact = 1.0 / np.sqrt(d.astype(np.longdouble))
    assert np.abs((X[:, np.arange(32), np.arange(32)] - exact) / exact).max() <= 2.0 ** -52
