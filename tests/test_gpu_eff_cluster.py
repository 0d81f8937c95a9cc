"""Effective-model sweeps with a chain spread over a cluster of CTAs: spins and
flip counts bit for bit those of the FP64 oracle, for few chains (clusters of
up to eight CTAs) and many (one CTA per chain), where the split can go wrong:
a field whose size is no multiple of 16 bytes (chains start unaligned), colours
that leave the last CTAs without a site, colours of several passes per CTA, and
four and sixteen classes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1612_03804_gb300 import effmodel as E
from paper_1612_03804_gb300.inputs import batch_uniform

pytestmark = pytest.mark.gpu

J = {4: np.array([-0.06, -0.01, -0.005, -0.4]),
     16: np.concatenate([[-0.06, -0.01], -0.4 * 0.6 ** np.arange(10), [-0.01, -0.004, -0.003, -0.001]])}
CLS = {4: E.CLASSES_4, 16: E.paper_classes()}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("Lx,Ly,M,classes,B", [(8, 8, 20, 4, 2), (9, 7, 21, 16, 3), (13, 11, 25, 4, 40), (24, 24, 20, 16, 16),
                                               (24, 24, 20, 16, 60), (32, 32, 80, 4, 2), (32, 32, 160, 16, 1), (9, 7, 21, 4, 170)])
def test_eff_sweeps_bit_exact_at_any_split(Lx, Ly, M, classes, B):
    import torch
    from paper_1612_03804_gb300 import sldqmc
    m = O.Model(Lx, Ly, beta=M * 0.05, dtau=0.05)
    fields = batch_uniform(77 + M, B, M, m.N)
    seed, step, nsw = 91, 6, 2
    with sldqmc.Context(Lx, Ly, t=m.t, mu=m.mu, xi=m.xi, beta=m.beta, dtau=m.dtau, n_wrap=10, J=m.J, h=m.h,
                        max_batch=1) as ctx:
        ctx.set_effective_model(CLS[classes], J[classes])
        d_s = torch.from_numpy(fields).cuda()
        d_acc = torch.zeros(B, dtype=torch.int64, device="cuda")
        ctx.eff_sweeps_batch_dev(d_s, nsw, seed, step, -1, d_acc)
        ctx.sync()
        out, acc = d_s.cpu().numpy(), d_acc.cpu().numpy()
    for b in sorted({0, B // 2, B - 1}):
        key = seed + (b << 32)
        direction = int(O.lib().or_random_word(key, 0, 0, step, 3)) & 1
        so, na, mg = O.eff_sweeps(m, fields[b], CLS[classes], J[classes], nsw, seed=key, step=step, direction=direction)
        assert mg == 0
        np.testing.assert_array_equal(out[b], so)
        assert acc[b] == na
