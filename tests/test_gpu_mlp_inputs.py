"""Surrogate inference from device arrays at addresses that its loads cannot use: the
arrays are copied first, and the values are those of aligned ones."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [4, 1])
def test_misaligned_device_arrays(shift):
    import torch
    import paper_1708_09705_gb300 as gm
    n, rng = 1000, np.random.default_rng(shift)
    flat = np.concatenate([np.concatenate([W.ravel(), b])
                           for W, b in M.init_params(3)]).astype(np.float32)
    si = np.exp(rng.uniform(np.log(60.0), np.log(5000.0), n))
    x = [si, si + 10.0, rng.uniform(0, 0.01, n)]
    raw = []
    for v in x:
        t = torch.zeros(8 * n + 8, dtype=torch.uint8, device="cuda")
        t[shift:shift + 8 * n] = torch.tensor(v.view(np.uint8), device="cuda")
        raw.append(t)
    torch.cuda.synchronize()
    y, e = (torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(2))
    one = np.array([500.0])
    with gm.ep_init(gm.default_config(precision=gm.PREC_FP32), 0 * one, 0 * one, one, 0 * one + 0.5,
                    0 * one + 0.05) as ctx:
        ctx.surrogate_set_params(flat)
        want = ctx.surrogate_eval(*x, 1.3, 17.0)
        st = gm.lib().gm_surrogate_eval(ctx._h, n, *(t.data_ptr() + shift for t in raw), 1.3, 17.0,
                                        y.data_ptr(), e.data_ptr())
    assert st == 0
    np.testing.assert_array_equal(y.cpu().numpy(), want[0])
    np.testing.assert_array_equal(e.cpu().numpy(), want[1])
