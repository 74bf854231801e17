"""The few-lanes-per-sightline sampler against the one-thread kernel at the point
counts where its layout changes (ragged counts among them), with one sightline,
a ragged last warp, many sightlines, a sightline without a Cholesky factor and
one whose upper triangle holds garbage (only the lower one is read).  Both run
the same expressions, so samples and wall hits are equal bit for bit (a chain
that starts in a narrow wedge amplifies a last bit by 1e8: nothing weaker
would do)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,nsl", [(1, 3), (2, 1), (3, 5), (8, 7), (9, 4), (15, 6), (16, 9),
                                   (16, 8193), (17, 3), (31, 5), (32, 2), (33, 2)])
def test_group_sampler(m, nsl, monkeypatch):
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(100 * m + nsl)
    burn, ns = 3, 9
    s = np.linspace(0.0, 1.0, m)
    S = (0.02 + 0.05 * rng.random(nsl))[:, None, None] * np.exp(
        -np.abs(s[:, None] - s[None, :]) / 0.4) + 1e-4 * np.eye(m)
    mu = np.cumsum(rng.normal(0.0, 0.08, (nsl, m)), axis=1) - 1.0
    mom = rng.standard_normal((nsl, burn + ns, m))
    S[0][np.triu_indices(m, 1)] = 7.0
    bad = S.copy()
    bad[nsl - 1, 0, 0] = -1.0
    one = np.array([500.0])
    res = {}
    for mode in (None, "0"):
        if mode is None:
            monkeypatch.delenv("GM_HMC_WARP", raising=False)
        else:
            monkeypatch.setenv("GM_HMC_WARP", mode)
        with gm.ep_init(gm.default_config(), 0 * one, 0 * one, one, 0 * one + 0.5,
                        0 * one + 0.05) as ctx:
            res[mode] = ctx.monotone_sample(mu, S, mom, burn)
            empty, h0 = ctx.monotone_sample(mu, S, mom, burn + ns)   # burn-in only
            assert empty.shape == (nsl, 0, m) and np.array_equal(h0, res[mode][1])
            with pytest.raises(gm.GmError) as e:
                ctx.monotone_sample(mu, bad, mom, burn)
            assert e.value.status == 4
    np.testing.assert_array_equal(res[None][1], res["0"][1])
    np.testing.assert_array_equal(res[None][0], res["0"][0])
