"""The site update's lanes per star change with the number of stars: every
split against the oracle's tilted moments at and beside the sizes where it
changes (152 SMs), both likelihoods, damped and not.  The moments carry ~1e-13,
and 1/v - tau_c loses at most two digits on these cavities: rtol 1e-10."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 33, 608, 609, 1217, 2433, 4865, 21889, 21890])
@pytest.mark.parametrize("lik", [0, 1])
def test_site_update_splits(n, lik):
    import torch
    import oracle as O
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    sd = rng.uniform(0.05, 0.4, n)
    mu = rng.uniform(-2.0, 1.0, n)
    A = np.exp(mu + sd * rng.standard_normal(n))
    obs = A + 0.05 * rng.standard_normal(n) if lik == 0 else np.log(A)
    sig = np.full(n, 0.05) if lik == 0 else 0.05 / A
    tau = 0.5 * rng.uniform(0, 1, n) / sd ** 2
    tau[n // 2] = 2.0 / sd[n // 2] ** 2          # cavity precision < 0: skipped
    nu = tau * mu
    damping = 0.7
    d = [torch.tensor(v, dtype=torch.float64, device="cuda")
         for v in (mu, sd ** 2, obs, sig, tau, nu)]
    delta, skipped = C.c_double(), C.c_int64()
    for _ in range(2):                            # the counters start clean each call
        d[4].copy_(torch.tensor(tau))
        d[5].copy_(torch.tensor(nu))
        st = gm.lib().gm_site_update_noalloc(
            n, *(x.data_ptr() for x in d), lik, damping, 1e-8,
            C.c_void_p(torch.cuda.current_stream().cuda_stream), C.byref(delta), C.byref(skipped))
        assert st == 0
    want_t, want_n, skip = tau.copy(), nu.copy(), 0
    # the oracle loops in Python: all stars of small calls, the ends of large ones
    idx = np.arange(n) if n < 700 else np.r_[0:120, n // 2 - 3:n // 2 + 3, n - 120:n]
    for i in idx:
        tc, nc = 1 / sd[i] ** 2 - tau[i], mu[i] / sd[i] ** 2 - nu[i]
        if not tc > 0:
            skip += 1
            continue
        f = O.tilted_moments_gauss_in_a if lik == 0 else O.tilted_moments_gauss_in_lna
        mh, vh = f(nc / tc, 1 / tc, obs[i], sig[i] ** 2)[:2]
        if 1 / vh - tc < 0:
            skip += 1
            continue
        want_t[i] = 0.3 * tau[i] + 0.7 * (1 / vh - tc)
        want_n[i] = 0.3 * nu[i] + 0.7 * (mh / vh - nc)
    got_t, got_n = d[4].cpu().numpy(), d[5].cpu().numpy()
    scale = np.maximum(np.abs(want_t), 1 / sd ** 2)
    assert np.max(np.abs(got_t - want_t)[idx] / scale[idx]) < 1e-10
    assert np.max(np.abs(got_n - want_n)[idx] / (scale * 2.0)[idx]) < 1e-10
    if n < 700:
        assert skipped.value == skip
    dl = np.maximum(np.abs(got_t - tau) / (1 + np.abs(tau)), np.abs(got_n - nu) / (1 + np.abs(nu)))
    assert delta.value == pytest.approx(dl.max(), rel=1e-12)
