"""Effective-model sweeps with one launch per colour over all SMs, spins in
global memory: spins and flip counts bit for bit those of the FP64 oracle.  A
chain above 200 KB always takes this path (50 x 41 x 101: an odd number of
spins, so the second chain starts unaligned and every colour ends in a ragged
block); 48 x 48 x 80 takes it for its large colours."""
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


@pytest.mark.parametrize("Lx,Ly,M,classes,B", [(50, 41, 101, 4, 2), (50, 41, 101, 16, 2), (48, 48, 80, 4, 4)])
def test_colours_over_all_sms_bit_exact(Lx, Ly, M, classes, B):
    import torch
    from paper_1612_03804_gb300 import sldqmc
    m = O.Model(Lx, Ly, beta=M * 0.05, dtau=0.05)
    fields = batch_uniform(33 + M, B, M, m.N)
    seed, step, nsw = 92, 7, 2
    with sldqmc.Context(Lx, Ly, t=m.t, mu=m.mu, xi=m.xi, beta=m.beta, dtau=m.dtau, n_wrap=10, J=m.J, h=m.h,
                        max_batch=1) as ctx:
        ctx.set_effective_model(CLS[classes], J[classes])
        d_s = torch.from_numpy(fields).cuda()
        d_acc = torch.zeros(B, dtype=torch.int64, device="cuda")
        before = ctx.kernel_launches()
        ctx.eff_sweeps_batch_dev(d_s, nsw, seed, step, -1, d_acc)
        assert ctx.kernel_launches() - before >= nsw * O.coloring(m, CLS[classes])[0]
        ctx.sync()
        out, acc = d_s.cpu().numpy(), d_acc.cpu().numpy()
    for b in range(B):
        key = seed + (b << 32)
        direction = int(O.lib().or_random_word(key, 0, 0, step, 3)) & 1
        so, na, mg = O.eff_sweeps(m, fields[b], CLS[classes], J[classes], nsw, seed=key, step=step, direction=direction)
        assert mg == 0
        np.testing.assert_array_equal(out[b], so)
        assert acc[b] == na
