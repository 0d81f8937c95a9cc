"""Local sweeps on the kernels between the resident one (up to 111 sites) and
the blocks of 32 sites on the tensor cores (from 128 on): 112, 121 and 127 sites
with immediate updates in global memory (rank 1) and with delayed ones (ranks 8
and 32, the last block ragged), against the FP64 oracle; rank 1 against rank 32
on 16 chains; and 144 sites in a context too large for the digit planes, whose
flips, wraps and Green's functions stay on the FP64 pipe.  Spins and accept
counts equal, G and log|det| to the FP64 parity bars (1e-9)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1612_03804_gb300.inputs import batch_uniform

pytestmark = pytest.mark.gpu

TOL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


def _model(Lx, Ly, M):
    return O.Model(Lx, Ly, t=1.0, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, J=1.0, h=2.774)


def _ctx(m, B):
    from paper_1612_03804_gb300 import sldqmc
    return sldqmc.Context(m.Lx, m.Ly, mu=m.mu, xi=m.xi, beta=m.beta, dtau=m.dtau, n_wrap=m.n_wrap, J=m.J, h=m.h, max_batch=B)


def _sweep_against_oracle(ctx, m, fields, seed):
    import torch
    d_s = torch.from_numpy(fields).cuda()
    st = ctx.local_sweep_batch_dev(d_s, seed, 0, 1)
    out = d_s.cpu().numpy()
    for b in range(len(fields)):
        so, ref = O.local_sweep(m, fields[b], seed + (b << 32), 0, 1)
        assert ref["margin_events"] == 0 and st[b]["margin_events"] == 0
        assert st[b]["accepted"] == ref["accepted"] and st[b]["proposed"] == ref["proposed"]
        np.testing.assert_array_equal(out[b], so)
        assert st[b]["max_drift"] < TOL


@pytest.mark.parametrize("rank", [1, 8, 32])
@pytest.mark.parametrize("Lx,Ly,B", [(14, 8, 2), (11, 11, 3), (127, 1, 1)])
def test_flips_in_global_memory(Lx, Ly, B, rank):
    m = _model(Lx, Ly, 7)
    fields = batch_uniform(2900 + m.N, B, m.M, m.N)
    with _ctx(m, B) as ctx:
        ctx.set_local_update_rank(rank)
        _sweep_against_oracle(ctx, m, fields, 515)


def test_delayed_equals_immediate_at_121_sites():
    import torch
    m = _model(11, 11, 20)
    B = 16
    fields = batch_uniform(2710, B, m.M, m.N)
    outs = []
    for k in (1, 32):
        with _ctx(m, B) as ctx:
            ctx.set_local_update_rank(k)
            ctx.profile(True)
            d_s = torch.from_numpy(fields).cuda()
            st = ctx.local_sweep_batch_dev(d_s, 99, 0, 2)
            sites = ctx.profile_read_sites()
            ctx.profile(False)
            assert ("local_flips" in sites) == (k == 1) and "flip_block" not in sites
            outs.append((d_s.cpu().numpy(), [x["accepted"] for x in st]))
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    assert outs[0][1] == outs[1][1]


@pytest.mark.parametrize("rank", [1, 32])
def test_without_room_for_the_digit_planes(rank):
    """A workspace for 80000 configurations of 144 sites (133 GB) leaves the planes
    more than a third of what is free, so the context does without them."""
    import torch
    from paper_1612_03804_gb300 import sldqmc
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 240e9:
        pytest.skip("needs 240 GB of free device memory")
    m = _model(12, 12, 7)
    fields = batch_uniform(2800, 2, m.M, m.N)
    with _ctx(m, 80000) as ctx:
        ctx.profile(True)
        d_s = torch.from_numpy(fields).cuda()
        ld = torch.zeros(2, dtype=torch.float64, device="cuda")
        sg = torch.zeros(2, dtype=torch.int32, device="cuda")
        G = torch.zeros((2, m.N, m.N), dtype=torch.float64, device="cuda")
        ctx.green_batch_dev(d_s, -1, 3, G, ld, sg)
        ctx.sync()
        prof = ctx.profile_read()
        assert prof["gemm_oz"]["launches"] == 0 and prof["gemm_f64"]["launches"] > 0
        ctx.profile(False)
        for b in range(2):
            ref, rs, Gr = O.weight(m, fields[b], -1, tau0=3, want_G=True)
            assert int(sg[b]) == rs
            assert abs(float(ld[b]) - ref) <= TOL * abs(ref)
            assert np.abs(G[b].cpu().numpy() - Gr).max() < TOL
        ctx.set_local_update_rank(rank)
        _sweep_against_oracle(ctx, m, fields, 516)
