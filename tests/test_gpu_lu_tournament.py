"""LU panels taller than a cluster of CTAs holds (12800 rows) choose their pivots
by tournament: 128 x 102 (N = 13056), whose first eight panels do, M = 2, FP64
mode.  The uniform field's log|det| against its closed form (LU without a
right-hand side); for a seeded random field the particle-hole identity
ld_eta(s; mu) - ld_-eta(s; -mu) = beta N mu + eta dtau xi sum s, and G (LU with
a right-hand side) by G (1 + B_2 B_1) v = v for random vectors v, the slice
matrices applied as the two ring propagators they factor into.  Bars: the FP64
parity tests' 1e-9 (log|det| relative; G v relative to the largest |v|)."""
import numpy as np
import pytest

from paper_1612_03804_gb300.inputs import uniform_field

pytestmark = pytest.mark.gpu

LX, LY, M, DTAU, MU, XI = 128, 102, 2, 0.1, -0.5, 1.0
N = LX * LY
TOL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _ctx(mu):
    from paper_1612_03804_gb300 import sldqmc
    return sldqmc.Context(LX, LY, mu=mu, xi=XI, beta=M * DTAU, dtau=DTAU, n_wrap=M, max_batch=1)


def _ring(L):
    """e^{dtau A} of a ring of L sites."""
    k = 2.0 * np.pi * np.arange(L) / L
    row = np.real(np.fft.ifft(np.exp(2.0 * DTAU * np.cos(k))))
    return np.stack([np.roll(row, i) for i in range(L)])


def test_tournament_panels():
    import torch
    s = uniform_field(128, M, N)
    d_s = torch.from_numpy(s[None]).cuda()
    ld = torch.zeros(1, dtype=torch.float64, device="cuda")
    sg = torch.zeros(1, dtype=torch.int32, device="cuda")
    with _ctx(MU) as ctx:
        u = torch.ones((1, M, N), dtype=torch.int8, device="cuda")
        ctx.profile(True)
        ctx.weight_batch_dev(u, -1, ld, sg)
        sites = ctx.profile_read_sites()
        ctx.profile(False)
        ctx.sync()
        assert sites["lu_panel_tournament"]["launches"] == 8
        kx, ky = (2.0 * np.pi * np.arange(L) / L for L in (LX, LY))
        eps = -2.0 * (np.cos(ky)[:, None] + np.cos(kx)[None, :]) - (MU - XI)
        ref = float(np.sum(np.log1p(np.exp(-M * DTAU * eps))))
        assert sg.item() == 1 and abs(ld.item() - ref) <= TOL * abs(ref), (ld.item(), ref)
        G = torch.zeros((1, N, N), dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, 1, 0, G, ld, sg)
        ctx.sync()
    a, sa = ld.item(), sg.item()
    Ex, Ey = (torch.from_numpy(_ring(L)).cuda() for L in (LX, LY))
    v = torch.from_numpy(np.random.default_rng(9).standard_normal((N, 4))).cuda()
    w = v.clone()
    for tau in range(M):
        w = torch.exp(DTAU * XI * d_s[0, tau].double())[:, None] * w
        w = np.exp(DTAU * MU) * torch.einsum("yq,qpc,xp->yxc", Ey, w.reshape(LY, LX, 4), Ex).reshape(N, 4)
    err = float((G[0] @ (v + w) - v).abs().max() / v.abs().max())
    print(f"128x102: max |G (1 + B_2 B_1) v - v| / max |v| = {err:.2e}")
    assert err < TOL
    del G
    torch.cuda.empty_cache()
    with _ctx(-MU) as ctx:
        ctx.weight_batch_dev(d_s, -1, ld, sg)
        ctx.sync()
    rhs = M * DTAU * N * MU + DTAU * XI * float(s.astype(np.int64).sum())
    assert sg.item() == sa
    assert abs((a - ld.item()) - rhs) <= 2 * TOL * max(abs(a), abs(ld.item())), (a - ld.item(), rhs)
