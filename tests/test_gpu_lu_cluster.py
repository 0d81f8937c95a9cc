"""LU panels factored by clusters of CTAs: log|det|, sign and G against the
FP64 oracle at the sizes where a panel's split can go wrong: rows that divide
evenly and not, a ragged last panel, panels that shrink from several CTAs to
one, one item and several; and the tall panels of 36 x 36 and 52 x 52 (two and
four CTAs at least) against the uniform field's closed form.  Bars: the FP64
parity tests' 1e-9 (log|det| relative, G absolute)."""
import math

import numpy as np
import pytest

from paper_1612_03804_gb300.inputs import batch_uniform

pytestmark = pytest.mark.gpu

TOL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("Lx,Ly,B", [(16, 8, 1), (10, 15, 2), (19, 21, 1), (16, 16, 3), (12, 12, 80)])
def test_lu_cluster_against_oracle(Lx, Ly, B):
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    M, N = 6, Lx * Ly
    m = O.Model(Lx, Ly, t=1.0, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=3)
    s = batch_uniform(240 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=3, max_batch=B) as ctx:
        d_s = torch.from_numpy(s).cuda()
        ld = torch.zeros(B, dtype=torch.float64, device="cuda")
        sg = torch.zeros(B, dtype=torch.int32, device="cuda")
        G = torch.zeros((B, N, N), dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, -1, 2, G, ld, sg)
        ctx.sync()
        for b in sorted({0, B // 2, B - 1}):
            ref, rs, Gr = O.weight(m, s[b], -1, tau0=2, want_G=True)
            assert int(sg[b]) == rs
            assert abs(float(ld[b]) - ref) <= TOL * abs(ref)
            assert np.abs(G[b].cpu().numpy() - Gr).max() < TOL


@pytest.mark.parametrize("L,B", [(36, 2), (52, 1)])
def test_lu_cluster_tall_panels_closed_form(L, B):
    import torch
    from paper_1612_03804_gb300 import sldqmc
    M, N, mu, dtau = 6, L * L, -0.5, 0.1
    with sldqmc.Context(L, L, mu=mu, xi=1.0, beta=M * dtau, dtau=dtau, n_wrap=3, max_batch=B) as ctx:
        s = torch.ones((B, M, N), dtype=torch.int8, device="cuda")
        ld = torch.zeros(B, dtype=torch.float64, device="cuda")
        sg = torch.zeros(B, dtype=torch.int32, device="cuda")
        ctx.weight_batch_dev(s, -1, ld, sg)
        ctx.sync()
    k = 2.0 * np.pi * np.arange(L) / L
    eps = -2.0 * (np.cos(k)[:, None] + np.cos(k)[None, :]) - (mu - 1.0)
    ref = float(np.sum(np.log1p(np.exp(-M * dtau * eps))))
    assert sg.cpu().tolist() == [1] * B
    assert all(abs(v - ref) <= TOL * abs(ref) for v in ld.cpu().tolist()), (ld, ref)
    assert math.isfinite(ref)
