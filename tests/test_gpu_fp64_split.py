"""FP64 mode on lattices of 128 sites and more: slice products, wraps, fresh
Green's functions and rank-32 corrections run by digit splitting on the
tensor cores.  Weights, Green's functions and local sweeps against the FP64
oracle at the sizes where tiles can go wrong: exactly one 128-row tile, one
row more than a multiple of 32, several items per tile with a ragged last
one, more than one exactly accumulated K-chunk (N > 384), and fewer
configurations than the context's capacity.  The bars are those of the FP64
parity tests (1e-9 relative on log|det|, 1e-9 on G, spins equal)."""
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


def _model(Lx, Ly, M, n_wrap=5):
    from oracle import oracle as O
    return O.Model(Lx, Ly, t=1.0, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=n_wrap)


@pytest.mark.parametrize("Lx,Ly,B,cap", [(16, 8, 1, 1), (43, 3, 3, 4), (12, 12, 5, 5), (19, 21, 2, 3)])
def test_fp64_weight_and_green(Lx, Ly, B, cap):
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    M, N = 13, Lx * Ly
    m = _model(Lx, Ly, M)
    s = batch_uniform(40 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, max_batch=cap) as ctx:
        d_s = torch.from_numpy(s).cuda()
        ld = torch.zeros(B, dtype=torch.float64, device="cuda")
        sg = torch.zeros(B, dtype=torch.int32, device="cuda")
        G = torch.zeros((B, N, N), dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, -1, 7, G, ld, sg)
        ctx.sync()
        for b in range(B):
            ref, rs, Gr = O.weight(m, s[b], -1, tau0=7, want_G=True)
            assert int(sg[b]) == rs
            assert abs(float(ld[b]) - ref) <= TOL * abs(ref)
            assert np.abs(G[b].cpu().numpy() - Gr).max() < TOL


@pytest.mark.parametrize("Lx,Ly,rank", [(16, 8, 1), (43, 3, 32), (13, 12, 9)])
def test_fp64_local_sweep(Lx, Ly, rank):
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    import torch
    M, N, B = 7, Lx * Ly, 2
    m = _model(Lx, Ly, M)
    s = batch_uniform(60 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, max_batch=B) as ctx:
        ctx.set_local_update_rank(rank)
        d_s = torch.from_numpy(s).cuda()
        stats = ctx.local_sweep_batch_dev(d_s, 71, 0, 1)
        out = d_s.cpu().numpy()
    for b in range(B):
        so, st = O.local_sweep(m, s[b], 71 + (b << 32), 0, 1)
        assert stats[b]["margin_events"] == 0
        np.testing.assert_array_equal(out[b], so)
        assert stats[b]["max_drift"] < TOL


# Up to 64 sites the slice products of a block run in one launch of 128-row
# CTAs; from there to 127 sites per slice, and wraps at all sizes, once there is
# enough work.  Sizes: one column group and its edges (16, 17 sites), a ragged
# last group (49, 63), exactly 64; rows that end inside a CTA and inside an
# item; one and several CTAs; 81 sites on either side of the rule's line.
@pytest.mark.parametrize("Lx,Ly,B", [(2, 2, 3), (4, 4, 1), (17, 1, 9), (7, 7, 3), (9, 7, 5), (8, 8, 1), (8, 8, 35),
                                     (9, 9, 2), (9, 9, 40)])
def test_fp64_small_weight_and_green(Lx, Ly, B):
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    M, N = 13, Lx * Ly
    m = _model(Lx, Ly, M)
    s = batch_uniform(140 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, max_batch=B) as ctx:
        d_s = torch.from_numpy(s).cuda()
        ld = torch.zeros(B, dtype=torch.float64, device="cuda")
        sg = torch.zeros(B, dtype=torch.int32, device="cuda")
        G = torch.zeros((B, N, N), dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, 1, 9, G, ld, sg)
        ctx.sync()
        for b in sorted({0, 1 % B, B // 2, B - 1}):
            ref, rs, Gr = O.weight(m, s[b], 1, tau0=9, want_G=True)
            assert int(sg[b]) == rs
            assert abs(float(ld[b]) - ref) <= TOL * max(1.0, abs(ref))
            assert np.abs(G[b].cpu().numpy() - Gr).max() < TOL


@pytest.mark.parametrize("Lx,Ly,B", [(4, 4, 3), (9, 7, 2), (8, 8, 40), (9, 9, 12), (8, 8, 80)])
def test_fp64_small_local_sweep(Lx, Ly, B):
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    import torch
    M, N = 7, Lx * Ly
    m = _model(Lx, Ly, M)
    s = batch_uniform(160 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, max_batch=B) as ctx:
        d_s = torch.from_numpy(s).cuda()
        stats = ctx.local_sweep_batch_dev(d_s, 71, 0, 1)
        out = d_s.cpu().numpy()
    for b in sorted({0, 1, B - 1}):
        so, st = O.local_sweep(m, s[b], 71 + (b << 32), 0, 1)
        assert stats[b]["margin_events"] == 0
        np.testing.assert_array_equal(out[b], so)
        assert stats[b]["max_drift"] < TOL


# Up to 25 sites, and to 32 with few configurations, a whole weight runs in one
# CTA; 27 and 32 sites with a capacity beyond that take the launches.
@pytest.mark.parametrize("Lx,Ly,B,cap", [(1, 1, 2, 2), (3, 1, 3, 3), (5, 5, 3, 3), (9, 3, 2, 2), (9, 3, 2, 512), (8, 4, 3, 3),
                                         (8, 4, 3, 400), (11, 3, 2, 2)])
def test_fp64_one_cta_weight(Lx, Ly, B, cap):
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    M, N = 11, Lx * Ly
    m = _model(Lx, Ly, M, n_wrap=4)
    s = batch_uniform(180 + N, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=4, max_batch=cap) as ctx:
        d_s = torch.from_numpy(s).cuda()
        G = torch.zeros((B, N, N), dtype=torch.float64, device="cuda")
        ld = torch.zeros(B, dtype=torch.float64, device="cuda")
        sg = torch.zeros(B, dtype=torch.int32, device="cuda")
        lw = torch.zeros(B, dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, -1, 6, G, ld, sg)
        ctx.log_weight_batch_dev(d_s, lw)
        ctx.sync()
        for b in range(B):
            ref, rs, Gr = O.weight(m, s[b], -1, tau0=6, want_G=True)
            assert int(sg[b]) == rs
            assert abs(float(ld[b]) - ref) <= TOL * max(1.0, abs(ref))
            assert np.abs(G[b].cpu().numpy() - Gr).max() < TOL
            both = 2.0 * (O.weight(m, s[b], 1)[0] + O.weight(m, s[b], -1)[0]) + ctx.log_bare_weight(s[b])
            assert abs(float(lw[b]) - both) <= TOL * max(1.0, abs(both))
