"""The few-lanes-per-sightline sampler on values far from one, whose squares leave the
range of floats in its screening of the walls: bit for bit the one-thread kernel, and
every sample non-decreasing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-26, 1e-19, 1e-14, 1e14, 1e19, 1e26])
@pytest.mark.parametrize("m", [5, 16, 24])
def test_scales(m, scale, monkeypatch):
    import paper_1708_09705_gb300 as gm
    rng, nsl = np.random.default_rng(m), 9
    x = np.linspace(0.0, 1.0, m)
    S = (0.05 * np.exp(-np.abs(x[:, None] - x[None, :]) / 0.4) + 1e-4 * np.eye(m)) * scale ** 2
    S = np.repeat(S[None], nsl, 0)
    mu = np.cumsum(rng.normal(0.02, 0.08, (nsl, m)), axis=1) * scale
    mu[0] = 0.0
    mom = rng.standard_normal((nsl, 30, m))
    one, res = np.array([500.0]), {}
    for mode in (None, "0"):
        if mode is None:
            monkeypatch.delenv("GM_HMC_WARP", raising=False)
        else:
            monkeypatch.setenv("GM_HMC_WARP", mode)
        with gm.ep_init(gm.default_config(), 0 * one, 0 * one, one, 0 * one + 0.5,
                        0 * one + 0.05) as ctx:
            res[mode] = ctx.monotone_sample(mu, S, mom, 3)
    np.testing.assert_array_equal(res[None][1], res["0"][1])
    np.testing.assert_array_equal(res[None][0], res["0"][0])
    assert res[None][1].sum() > 0
