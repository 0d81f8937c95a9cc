"""Local-flip decisions where the two parts of the bare weight's change, space and
time, are large and nearly cancel: a decision taken in fewer bits must leave room
for the rounding of each part, not of their difference.  h = 1e-300 makes the
time coupling 346; J is set so that the first site of an ordered field is decided
by a log ratio that lies a few 1e-5 on either side of log u, less than the FP32
rounding of the parts (up to 1.2e-4) and far more than the margin of 1e-8.  Spins
and flip counts are those of the FP64 oracle, in each of the kernels: G in shared
memory (4 x 4), G in global memory (14 x 8), blocks of 32 sites (12 x 12)."""
import math

import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

DTAU, M, XI = 0.1, 4, 1.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


def _model(Lx, Ly, J, h):
    return O.Model(Lx, Ly, mu=-0.5, xi=XI, beta=M * DTAU, dtau=DTAU, n_wrap=M, J=J, h=h)


def _tuned(Lx, Ly, seed, h):
    """J for which the first site's log ratio is log u + delta, delta half the FP32
    rounding of the bare part and of the other sign; (None, 0) if that is small."""
    m = _model(Lx, Ly, 1.0, h)
    s = np.ones((M, m.N), dtype=np.int8)
    fermion = 0.0
    for eta in (1, -1):
        _, _, G = O.weight(m, s, eta, tau0=1, want_G=True)
        g = (O.build_E(m, -1.0) @ G @ O.build_E(m, 1.0))[0, 0]
        fermion += 2.0 * math.log(abs(1.0 + (math.exp(-2.0 * eta * DTAU * XI) - 1.0) * (1.0 - g)))
    lu = math.log(O.uniform(seed, 0, 0, 0, 1))
    Kt = -0.5 * math.log(math.tanh(DTAU * h))
    f = np.float32

    def J_of(delta):  # -2 (4 dtau J + 2 Kt) + fermion = lu + delta
        return ((fermion - lu - delta) / 2.0 - 2.0 * Kt) / 4.0 / DTAU

    dtauJ = DTAU * J_of(0.0)
    rounding = float(f(-2.0) * (f(dtauJ) * f(4) + f(Kt) * f(2))) - (-2.0 * (4.0 * dtauJ + 2.0 * Kt))
    return (J_of(-0.5 * rounding), rounding) if abs(rounding) >= 4e-5 else (None, rounding)


def _cases(Lx, Ly, want):
    out, seed = [], 100
    while len(out) < want:
        J, rounding = _tuned(Lx, Ly, seed, 1e-300 * (1.0 + 0.013 * (seed - 100)))
        if J is not None:
            out.append((seed, 1e-300 * (1.0 + 0.013 * (seed - 100)), J, rounding))
        seed += 1
    return out


@pytest.mark.parametrize("Lx,Ly,want", [(4, 4, 6), (14, 8, 4), (12, 12, 4)])
def test_cancelling_bare_terms_decide_as_fp64(Lx, Ly, want):
    from paper_1612_03804_gb300 import sldqmc
    cases = _cases(Lx, Ly, want)
    assert {r > 0 for _, _, _, r in cases} == {True, False}  # wrong acceptances and wrong rejections
    for seed, h, J, _ in cases:
        m = _model(Lx, Ly, J, h)
        s = np.ones((M, m.N), dtype=np.int8)
        with sldqmc.Context(Lx, Ly, mu=-0.5, xi=XI, beta=m.beta, dtau=DTAU, n_wrap=M, J=J, h=h, max_batch=1) as ctx:
            out, st = ctx.local_sweep(s, seed, 0, 1)
        ref, so = O.local_sweep(m, s, seed, 0, 1)
        assert so["margin_events"] == 0 and st["margin_events"] == 0
        assert st["accepted"] == so["accepted"]
        np.testing.assert_array_equal(out, ref)
