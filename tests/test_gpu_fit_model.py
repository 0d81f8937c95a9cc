"""The model that a fit leaves in the context: its classes with the fitted
couplings, so that effective sweeps, features and a second fit in the same
context are those of the fitted model ("The fitted model becomes the context's
effective model").  Spins and flip counts bit for bit those of the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1612_03804_gb300 import effmodel as E
from paper_1612_03804_gb300.inputs import domain_field, uniform_field

pytestmark = pytest.mark.gpu

CLASSES = {4: E.CLASSES_4, 16: E.paper_classes()}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n_class,L,n_cfg", [(4, 4, 40), (16, 6, 60)])
def test_fitted_model_drives_the_sweeps(n_class, L, n_cfg):
    from paper_1612_03804_gb300 import sldqmc
    classes = CLASSES[n_class]
    m = O.Model(L, L, mu=0.0, xi=1.0, beta=2.0, dtau=0.1, n_wrap=10)
    cfgs = np.stack([domain_field(500 + k, m.M, L, L, corr=2) for k in range(n_cfg)])
    # ln omega of a known model with a little noise: the fit is a fit, and no weight is needed
    rng = np.random.default_rng(3)
    F = np.array([O.features(m, c, classes) for c in cfgs], dtype=np.float64)
    logw = F @ (0.05 / (1 + np.arange(n_class))) + 1e-3 * rng.standard_normal(n_cfg)
    with sldqmc.Context(L, L, mu=0.0, xi=1.0, beta=m.beta, dtau=m.dtau, n_wrap=10, max_batch=8) as ctx:
        ctx.set_effective_model(classes, np.zeros(n_class))
        J, _, _ = ctx.fit_effective_action(cfgs, logw)
        s = uniform_field(11, m.M, m.N)
        for direction in (0, 1):
            out, acc = ctx.eff_sweeps(s, 3, seed=77, step=5, direction=direction)
            ref, na, mg = O.eff_sweeps(m, s, classes, J, 3, seed=77, step=5, direction=direction)
            assert mg == 0
            np.testing.assert_array_equal(out, ref)
            assert acc == na
        np.testing.assert_array_equal(ctx.features(cfgs[:3]), F[:3].astype(np.int64))
        J2, _, _ = ctx.fit_effective_action(cfgs, logw)  # the classes are still there
        np.testing.assert_array_equal(J2, J)
