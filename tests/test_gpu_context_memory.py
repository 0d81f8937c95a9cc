"""Device memory of a mixed-mode context: the work buffers, the split operands, two
buffers of eight digit planes, the planes of the 32 x 32 inverse blocks and the
per-configuration vectors, and nothing else that grows with the lattice: what the
rank-32 updates need lies in work buffers that are idle then, so that the
largest max_batch that fits the GPU stays what it was.  And that sharing does no
harm: a ragged last panel (N = 141) with G, sweeps and weights in turn on one context."""
import numpy as np
import pytest

from paper_1612_03804_gb300.inputs import batch_uniform

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


def test_mixed_mode_context_takes_its_layout():
    import torch
    from paper_1612_03804_gb300 import sldqmc
    N, M, B = 128, 4, 4000
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    with sldqmc.Context(16, 8, beta=M * 0.1, dtau=0.1, n_wrap=2, prec="3xtf32", max_batch=B):
        taken = before - torch.cuda.mem_get_info()[0]
    per = 8 * 10 * N * N                                # work buffers
    per += 4 * 2 * 2 * N * N                            # two TF32 parts of two buffers (128 is a multiple of 64)
    per += 2 * 8 * 2 * N * N + 2 * 8 * 32 * 32          # digit planes, inverse blocks
    per += 4 * (5 * N + 32)                             # row exponents
    per += 8 * 2 * N + 4 * 2 * N + 2 * M * N + 4 * 24 * 32 + 256  # D, permutations, fields, pivot candidates, scalars
    assert taken <= 1.01 * per * B + 32 * 2 ** 20, (taken, per * B)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-9), ("3xtf32", 1e-6)])
def test_ragged_panels_in_turn(prec, tol):
    import torch
    from oracle import oracle as O
    from paper_1612_03804_gb300 import sldqmc
    Lx, Ly, M, B, cap = 47, 3, 8, 2, 3
    N = Lx * Ly
    m = O.Model(Lx, Ly, t=1.0, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=4, J=1.0, h=2.774)
    s = batch_uniform(311, B, M, N)
    with sldqmc.Context(Lx, Ly, mu=-0.5, xi=1.0, beta=m.beta, dtau=0.1, n_wrap=4, prec=prec, max_batch=cap) as ctx:
        for turn in range(2):
            d_s = torch.from_numpy(s).cuda()
            ld = torch.zeros(B, dtype=torch.float64, device="cuda")
            sg = torch.zeros(B, dtype=torch.int32, device="cuda")
            G = torch.zeros((B, N, N), dtype=torch.float64, device="cuda")
            ctx.green_batch_dev(d_s, -1, 3, G, ld, sg)
            l2 = torch.zeros(B, dtype=torch.float64, device="cuda")
            ctx.weight_batch_dev(d_s, 1, l2)
            ctx.sync()
            for b in range(B):
                ref, rs, Gr = O.weight(m, s[b], -1, tau0=3, want_G=True)
                assert int(sg[b]) == rs and abs(float(ld[b]) - ref) <= tol * abs(ref)
                assert np.abs(G[b].cpu().numpy() - Gr).max() < 10 * tol
                ref = O.weight(m, s[b], 1)[0]
                assert abs(float(l2[b]) - ref) <= tol * abs(ref)
            if prec == "fp64":
                ctx.local_sweep_batch_dev(d_s, 5, turn, 1)
                out = d_s.cpu().numpy()
                for b in range(B):
                    so, st = O.local_sweep(m, s[b], 5 + (b << 32), turn, 1)
                    assert st["margin_events"] == 0
                    np.testing.assert_array_equal(out[b], so)
                s = out
