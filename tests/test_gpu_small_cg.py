"""FP64 solves with one block per column (few stored entries) against the panel
passes (GM_SPMM=simt pins them): posteriors, warm-started EP sweeps, probing and
predictions agree to the solves' tolerance, at star counts beside the slices of 32
rows, the groups of four slices, 512 and 1,024 threads and the largest count taken."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,panel,probe", [(1, 0, 0.0), (31, 0, 0.0), (33, 0, 2.0), (129, 64, 0.0),
                                           (400, 0, 0.0), (513, 0, 2.0), (1025, 0, 2.0),
                                           (2048, 32, 2.0), (2049, 32, 2.0)])
def test_columns_in_blocks_match_panels(n, panel, probe, monkeypatch):
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    # beyond 400 stars the field grows with them, so that rows stay short
    f = max(1.0, np.sqrt(n / 400.0)) * (3.0 if n > 1000 else 1.0)
    l = cat["l"].mean() + (cat["l"] - cat["l"].mean()) * f
    b = cat["b"].mean() + (cat["b"] - cat["b"].mean()) * f
    # tolerance: both solves stop below a relative residual of 1e-13, amplified by
    # K_ii / Sigma_ii <= 1e4 in the variances
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, cg_tol=1e-13, rhs_panel=panel,
                                   probe_factor=probe)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    tau[1::7] = 0.0
    tau[3::11] *= 1e-9
    q = np.arange(min(n, 70))
    res = {}
    for mode in ("simt", ""):
        if mode:
            monkeypatch.setenv("GM_SPMM", mode)
        else:
            monkeypatch.delenv("GM_SPMM")
        with gm.ep_init(cfg, l, b, cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.profile(True)
            nnz = ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            out = ctx.get_posterior() + ctx.predict(l[q], b[q], cat["s"][q] + 3.0)
            assert ctx.stats()["cg_iters_mean"] > 0
            ran = "k_cg_columns" in ctx.kernel_times()
            assert ran == (mode == "" and n <= 2048 and nnz < 130e3)
            ctx.ep_sweep(2)                       # the second sweep starts warm
            res[mode] = out + ctx.get_posterior()
    for a, b_ in zip(res["simt"], res[""]):
        np.testing.assert_allclose(b_, a, rtol=1e-9, atol=1e-11)
