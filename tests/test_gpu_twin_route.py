"""The exact log weight is bit for bit 2 ld(+1) + 2 ld(-1) + log phi of the
single-flavour calls, also for an FP64 context made while there was no room for its
digit planes: the second workspace, made later with room to spare, takes the
context's way of every product."""
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


@pytest.mark.parametrize("room", [True, False])
def test_log_weight_takes_the_contexts_way(room):
    import torch
    from paper_1612_03804_gb300 import sldqmc
    L, M, B, cap = 12, 20, 3, 2000
    fields = batch_uniform(821, B, M, L * L)
    hog = None
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    if not room:  # 3.3 GB of work buffers, 1.8 GB of planes: leave 6.5 GB
        hog = torch.empty(torch.cuda.mem_get_info()[0] - int(6.5e9), dtype=torch.uint8, device="cuda")
    with sldqmc.Context(L, L, mu=-0.5, xi=1.0, beta=M * 0.1, dtau=0.1, n_wrap=5, max_batch=cap) as ctx:
        del hog
        torch.cuda.empty_cache()
        d_s = torch.from_numpy(fields).cuda()
        lw, ldp, ldm = (torch.zeros(B, dtype=torch.float64, device="cuda") for _ in range(3))
        ctx.profile(True)
        ctx.weight_batch_dev(d_s, 1, ldp)
        prof = ctx.profile_read()
        ctx.profile(False)
        assert (prof["gemm_oz"]["launches"] > 0) == room
        ctx.weight_batch_dev(d_s, -1, ldm)
        ctx.log_weight_batch_dev(d_s, lw)
        ctx.sync()
        bare = np.array([ctx.log_bare_weight(f) for f in fields])
        lw, ldp, ldm = lw.cpu().numpy(), ldp.cpu().numpy(), ldm.cpu().numpy()
    np.testing.assert_array_equal(lw, (2.0 * ldp + 2.0 * ldm) + bare)
