"""A local sweep captured in a CUDA graph by a context whose sweep buffers are
already there (a Green's function was asked for before): nothing may be allocated
under capture, in the mixed modes as in FP64, and the replayed sweep is the
sweep that runs uncaptured."""
import numpy as np
import pytest

from paper_1612_03804_gb300.inputs import batch_uniform

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    from paper_1612_03804_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("prec", ["fp64", "3xtf32"])
def test_first_sweep_under_capture(prec):
    import torch
    from paper_1612_03804_gb300 import sldqmc
    L, M, B, seed = 12, 8, 2, 61
    fields = batch_uniform(810, B, M, L * L)
    kw = dict(mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=4, prec=prec, max_batch=B)
    with sldqmc.Context(L, L, **kw) as ctx:
        d_s = torch.from_numpy(fields).cuda()
        ctx.local_sweep_batch_dev(d_s, seed, 3, 1)
        ref = d_s.cpu().numpy()
    side = torch.cuda.Stream()
    with sldqmc.Context(L, L, stream=side.cuda_stream, **kw) as ctx:
        ctx.green(fields[0], 1, 0)
        d_s = torch.from_numpy(fields).cuda()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            ctx.local_sweep_batch_dev(d_s, seed, 3, 1, want_stats=False)
        np.testing.assert_array_equal(d_s.cpu().numpy(), fields)  # captured, not run
        g.replay()
        torch.cuda.synchronize()
        ctx.sync()
        np.testing.assert_array_equal(d_s.cpu().numpy(), ref)
        del g
