"""The integer reciprocal of a pivot for every FP32 seed that the approximate
reciprocal may give: 1/f to within one unit in the last place (its documented
accuracy), so also just below 1/2 and just above 1.  Compiled for the host from
the same source as the kernels; compared with exact rationals' nearest double."""
import ctypes
import subprocess

import numpy as np
import pytest

SRC = r"""
#include <stdint.h>
#include "chol32.cuh"
extern "C" void recip_bits(const long long *u, const int *ulp, long long *out, int n)
{
    for (int i = 0; i < n; ++i) {
        const uint32_t fb = sldqmc::chol_seed_bits(u[i]);
        float f, r;
        memcpy(&f, &fb, 4);
        r = (float)(1.0 / (double)f);
        uint32_t rb;
        memcpy(&rb, &r, 4);
        out[i] = sldqmc::chol_reciprocal_bits(u[i], (uint32_t)((int)rb + ulp[i]));
    }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    from paper_1612_03804_gb300 import build
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("seed")
    (d / "seed.cu").write_text("#include <string.h>\n" + SRC)
    lib = str(d / "seed.so")
    r = subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-shared", str(d / "seed.cu"), "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)


def _pivots():
    rng = np.random.default_rng(8)
    m = np.concatenate([rng.integers(0, 2 ** 52, 1 << 18), np.arange(4096), 2 ** 52 - 1 - np.arange(4096),
                        rng.integers(0, 2 ** 31, 1 << 15), 2 ** 52 - 1 - rng.integers(0, 2 ** 31, 1 << 15)]).astype(np.int64)
    ef = np.where(np.arange(m.size) % 3 == 0, 1023, np.where(np.arange(m.size) % 3 == 1, 523, 1522)).astype(np.int64)
    return (ef << 52) | m


def _units_off(host, u, ulp):
    """How far 1/d is from the division's, in units in the last place, with seeds ulp units off."""
    shift = np.full(u.size, ulp, dtype=np.int32)
    if ulp == -2:  # two units below 1/2 are one of the binade above
        shift[(u & (2 ** 52 - 1)) < 2 ** 52 - 2 ** 29] = -1
    out = np.zeros_like(u)
    host.recip_bits(*(a.ctypes.data_as(ctypes.c_void_p) for a in (u, shift, out)), ctypes.c_int(u.size))
    return np.abs(out - (1.0 / u.view(np.float64)).view(np.int64))


def test_reciprocal_of_every_allowed_seed(host):
    u = _pivots()
    for ulp in (-2, -1, 0, 1):
        assert _units_off(host, u, ulp).max() <= 1


def test_reciprocal_is_the_division_whatever_the_seed(host):
    u = _pivots()
    for ulp in (-2, -1, 0, 1):
        assert _units_off(host, u, ulp).max() == 0
