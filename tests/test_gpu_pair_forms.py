"""The two forms of the FP64 node sums, pairs of floats and FP64 instructions
(GM_QUAD=fp64), on the same entries: both read the same cubic table, and differ by the
float pairs' 2^-47 a term and the table's third and fourth coefficients (1e-13 of g),
so 1e-12 relative to the entry; and the range of sigma2 that FP64 contexts take, up to
the end of the FP64 table (about 520), against the sum written out."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


def _entries(cat, i, j, q, **kw):
    import paper_1708_09705_gb300 as gm
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, quad_rule=gm.QUAD_GL, **kw)
    cfg.taper = 1                                    # K = log1p(R) as it is
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.profile(True)
        ctx.build_cov()
        K = ctx.get_entries(i, j)
        times = ctx.kernel_times()
        ctx.set_sites(np.zeros(len(cat["s"])), np.zeros(len(cat["s"])))
        return K, ctx.predict(*q)[1], times


@pytest.mark.parametrize("Q", [2, 31, 32, 33, 64, 100, 128])
@pytest.mark.parametrize("form", [0, 1])
def test_forms_agree(Q, form, monkeypatch):
    cat = make_catalogue("c1_plain_400", n=150, truth="mean")
    cat["l"][:12] = cat["l"][0]                      # one sightline
    cat["b"][:12] = cat["b"][0]
    cat["s"][12:16] = cat["s"][16:20] * (1 + 1e-9)   # nearly equal distances
    i, j = np.triu_indices(150)
    q = cat["l"][:20] + 1e-5, cat["b"][:20], cat["s"][:20] * 1.01
    monkeypatch.delenv("GM_QUAD", raising=False)
    K, v, t = _entries(cat, i, j, q, n_nodes=Q, form=form)
    assert "k_pair_quad" in t and "k_pair_quad_fp64" not in t
    monkeypatch.setenv("GM_QUAD", "fp64")
    K64, v64, t = _entries(cat, i, j, q, n_nodes=Q, form=form)
    assert "k_pair_quad_fp64" in t
    np.testing.assert_array_equal(K == 0, K64 == 0)
    np.testing.assert_allclose(K, K64, rtol=1e-12)
    np.testing.assert_allclose(v, v64, rtol=1e-12)


@pytest.mark.parametrize("n", [700, 1300])
def test_forms_agree_in_batches(n, monkeypatch):
    """Lists long enough for several entries a warp (44,000 and 160,000; the forms take
    batches of different sizes), every entry once: no gaps, no doubles, symmetric."""
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    out = []
    for mode in ("", "fp64"):
        monkeypatch.setenv("GM_QUAD", mode)
        cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, n_nodes=8)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.build_cov()
            out.append(ctx.get_csr() + ctx.get_prior())
    for a, b in zip(*out):
        np.testing.assert_allclose(a, b, rtol=1e-12)
    rp, col, val = out[0][:3]
    K = np.zeros((n, n))
    K[np.repeat(np.arange(n), np.diff(rp)), col] = val
    np.testing.assert_array_equal(K, K.T)
    assert np.all(val > 0) and np.all(np.diag(K) > 0)


@pytest.mark.parametrize("sigma2", [1e-12, 1e-8, 60.0, 75.0, 100.0, 500.0])
def test_range_of_sigma2(sigma2):
    """One star: R = sum over both nodes of w w' g, g = expm1(sigma2 phi), from the
    kernel's definition (the table, 3 parts in 1e12 of g at sigma2 <= 1, worse as g
    steepens, and its clamp at x = 2^-100: 1e-10 sigma2 of the diagonal's exponent)."""
    import paper_1708_09705_gb300 as gm
    from scipy.special import gamma, kv
    Q, L0, s = 16, 20.0, np.array([900.0, 300.0])
    z, w = np.polynomial.legendre.leggauss(Q)
    z, w = (z + 1) / 2, w / 2
    ref = []
    for A in s / L0:
        r = np.abs(A * (z[:, None] - z[None, :]))
        np.fill_diagonal(r, 1e-15)
        phi = 2 ** (2 / 3) / gamma(1 / 3) * np.cbrt(r) * kv(1 / 3, r)
        np.fill_diagonal(phi, 1.0)
        e = np.log(w[:, None] * w[None, :]) + sigma2 * phi
        top = e.max()
        # log1p(sum w w' expm1) without overflow
        if sigma2 > 1:
            ref.append(top + np.log(np.exp(e - top).sum()))
        else:
            ref.append(np.log1p((w[:, None] * w[None, :] * np.expm1(sigma2 * phi)).sum()))
    cfg = gm.default_config(sigma2=sigma2, outer_scale_pc=L0, cutoff_pc=60.0, n_nodes=Q,
                            quad_rule=gm.QUAD_GL, precision=gm.PREC_FP64)
    one = np.ones(2)
    with gm.ep_init(cfg, np.array([0.0, 0.1]), 0 * one, s, one, 0.1 * one) as ctx:
        ctx.build_cov()
        kd = ctx.get_prior()[1]
    np.testing.assert_allclose(kd, ref, rtol=1e-9 * max(1.0, sigma2), atol=0)
