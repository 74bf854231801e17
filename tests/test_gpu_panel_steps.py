"""FP32 variance panels against the dense FP64 formula at panel shapes that take each
form of the X / R step: one and two rows a warp and group, more, groups that do not
fill a block, narrow panels, with the deflation on the tensor cores, on the CUDA cores
and off."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,panel,deflate,core", [(40, 0, 0, ""), (333, 32, 0, ""), (1301, 0, 64, ""),
                                                  (1301, 96, 64, "0"), (1500, 0, 0, ""),
                                                  (4001, 0, 0, ""), (4001, 0, 64, "0")])
def test_panel_variances(n, panel, deflate, core, monkeypatch):
    import paper_1708_09705_gb300 as gm
    if core:
        monkeypatch.setenv("GM_DEFLATE_TC", core)
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    f = max(1.0, np.sqrt(n / 400.0))                 # the density of 400 stars
    l = cat["l"].mean() + (cat["l"] - cat["l"].mean()) * f
    b = cat["b"].mean() + (cat["b"] - cat["b"].mean()) * f
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    tau[::9] = 0.0
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP32, rhs_panel=panel, deflate=deflate)
    with gm.ep_init(cfg, l, b, cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        rp, col, val = ctx.get_csr()
        perm = ctx.get_perm()
        ctx.set_sites(tau, tau * np.log(A))
        var = ctx.get_posterior()[1]
    K = np.zeros((n, n))
    K[perm[np.repeat(np.arange(n), np.diff(rp))], perm[col]] = val
    V = np.sqrt(tau)[:, None] * K
    B = np.eye(n) + V * np.sqrt(tau)[None, :]
    ref = np.diag(K) - np.einsum("ij,ij->j", V, np.linalg.solve(B, V))
    # a column stops at ||r|| <= 1e-5 ||v|| and B >= 1, so its variance is within 1e-5
    # ||v||^2; FP32 vectors, products and their sums: as much again and 1e-5 K_ii
    tol = 2e-5 * np.einsum("ij,ij->j", V, V) + 1e-5 * np.diag(K)
    assert np.all(np.abs(var - ref) <= tol)
