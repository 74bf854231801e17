"""The FP64 tensor-core panel product (integer digits, exact sums) against the
CUDA-core FP64 product (GM_SPMM=simt): posteriors and predictions agree to the
solves' tolerance, at star counts beside the tile's 128 rows, the panel's 32 / 64
columns and the read-out period (128 union columns), with zero and tiny site
precisions (columns of very different scale), several panels and probing."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,panel,probe", [(256, 0, 0.0), (257, 0, 0.0), (300, 96, 0.0),
                                           (385, 32, 0.0), (640, 0, 2.0), (1100, 0, 0.0)])
def test_tc64_product_matches_fp64_units(n, panel, probe, monkeypatch):
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    # tolerance: both solves stop at a relative residual of 1e-13 (the panels go
    # on to 1e-16 of it), amplified by K_ii / Sigma_ii <= 1e4 in the variances
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, cg_tol=1e-13, rhs_panel=panel,
                                   probe_factor=probe)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    tau[::7] = 0.0
    tau[3::11] *= 1e-9
    res = {}
    for mode in ("simt", "tc"):
        monkeypatch.setenv("GM_SPMM", mode)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            mu, var = ctx.get_posterior()
            assert (ctx.stats()["tile_ksteps"] > 0) == (mode == "tc")
            res[mode] = (mu, var) + ctx.predict(cat["l"][:70], cat["b"][:70], cat["s"][:70] + 3.0)
            ctx.build_cov()                       # a second build rebuilds the tiles
            ctx.set_sites(tau, tau * np.log(A))
            np.testing.assert_array_equal(ctx.get_posterior()[1], var)
    for a, b in zip(res["simt"], res["tc"]):
        np.testing.assert_allclose(b, a, rtol=1e-9, atol=1e-11)
