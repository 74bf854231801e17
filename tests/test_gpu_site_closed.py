"""The allocation-free site update of the Gaussian likelihood in ln A (closed form)
against the formula in numpy, up to the largest count it takes: sites, the maximum
change over all blocks, the skipped stars.  A dozen FP64 operations a star, and
1 / v - tau_c loses at most two digits here: 1e-12."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 129, 4097, 300001, 1048576])
@pytest.mark.parametrize("damping", [1.0, 0.6])
def test_closed_form(n, damping):
    import torch
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    var = rng.uniform(0.05, 0.4, n) ** 2
    mu, sig = rng.uniform(-2.0, 1.0, n), rng.uniform(0.02, 0.3, n)
    obs = mu + sig * rng.standard_normal(n)
    tau = 0.5 * rng.uniform(0, 1, n) / var
    tau[::97] = 2.0 / var[::97]                  # cavity precision < 0: skipped
    nu = tau * mu
    d = [torch.tensor(v, device="cuda") for v in (mu, var, obs, sig, tau, nu)]
    delta, skipped = C.c_double(), C.c_int64()
    for _ in range(2):                            # counters and maximum start clean
        d[4].copy_(torch.tensor(tau))
        d[5].copy_(torch.tensor(nu))
        st = gm.lib().gm_site_update_noalloc(
            n, *(x.data_ptr() for x in d), 1, damping, 1e-8,
            C.c_void_p(torch.cuda.current_stream().cuda_stream), C.byref(delta), C.byref(skipped))
        assert st == 0
    ok = 1 / var - tau > 0
    want_t = np.where(ok, (1 - damping) * tau + damping / sig ** 2, tau)
    want_n = np.where(ok, (1 - damping) * nu + damping * obs / sig ** 2, nu)
    got_t, got_n = d[4].cpu().numpy(), d[5].cpu().numpy()
    scale = 1 / sig ** 2 + 1 / var
    assert np.max(np.abs(got_t - want_t) / scale) < 1e-12
    assert np.max(np.abs(got_n - want_n) / (4 * scale)) < 1e-12
    assert skipped.value == np.count_nonzero(~ok)
    dl = np.maximum(np.abs(got_t - tau) / (1 + np.abs(tau)), np.abs(got_n - nu) / (1 + np.abs(nu)))
    assert delta.value == pytest.approx(dl.max(), rel=1e-12)
