"""The serial part of every panel on its own: pivot reciprocals against IEEE
division, bit for bit, over random mantissas, the mantissas where the FP32 seed or
a rounding can go wrong (zeros, ones, within 2^30 of either end, the seed's
rounding boundaries) and binary exponents at both ends of the integer range and
beyond it."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "chol32.cuh"
using namespace sldqmc;
__global__ void k_recip(const double *d, double *out, int n, int *flag)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double x = d[i];
    out[i] = chol_reciprocal(x, true, flag);
}
extern "C" int run_recip(const double *d, double *out, int n, int *flag)
{
    k_recip<<<(n + 255) / 256, 256>>>(d, out, n, flag);
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
    assert probe.run_recip(_p(dd), _p(out), ctypes.c_int(d.size), _p(flag)) == 0
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
        assert probe.run_recip(_p(dd), _p(out), ctypes.c_int(1), _p(flag)) == 0
        assert flag.item() == 1 and out.item() == 1.0
