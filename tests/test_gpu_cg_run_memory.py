"""A mean solve whose hand-over slots find no memory runs by launches per step, as it did
without them: same bits."""
import numpy as np
import pytest

from synth import make_catalogue
from test_gpu_tc64_fallback import _Pool

pytestmark = pytest.mark.gpu


def test_no_memory_for_the_slots(monkeypatch):
    import torch
    import paper_1708_09705_gb300 as gm
    from paper_1708_09705_gb300 import gmead as g
    cat = make_catalogue("c1_plain_400", n=600, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP32, cg_tol=1e-6)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    size, out = (3 * blocks + 1) * 16, []
    for refuse in ((), (size,)):
        pool = _Pool()
        pool.refuse = refuse
        monkeypatch.setattr(g, "_torch_allocator", pool.allocator)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.profile(True)
            ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            out.append(ctx.get_posterior())
            assert ("k_cg_run" in ctx.kernel_times()) == (not refuse)
        assert refuse == () and size in pool.sizes or pool.refused > 0
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
