"""The way out of a bounded device wait that runs out (GM_WAIT_EXPIRES makes one
thread group take a completed wait for an expired one): the call ends with
GM_E_TIMEOUT whatever the other groups of the block are doing, again and again, and
the context stays usable."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu
TIMEOUT = 7


@pytest.mark.parametrize("n", [100, 128 * 152 * 4 + 5, 400003])
def test_surrogate_groups_leave_together(n, monkeypatch):
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    flat = np.concatenate([np.concatenate([W.ravel(), b])
                           for W, b in M.init_params(3)]).astype(np.float32)
    si = np.exp(rng.uniform(np.log(60.0), np.log(5000.0), n))
    sj, ch = si + 10.0, rng.uniform(0, 0.01, n)
    one = np.array([500.0])
    with gm.ep_init(gm.default_config(precision=gm.PREC_FP32), 0 * one, 0 * one, one, 0 * one + 0.5,
                    0 * one + 0.05) as ctx:
        ctx.surrogate_set_params(flat)
        y, e = ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
        for _ in range(20):
            monkeypatch.setenv("GM_WAIT_EXPIRES", "surrogate")
            with pytest.raises(gm.GmError) as err:
                ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
            assert err.value.status == TIMEOUT
            monkeypatch.delenv("GM_WAIT_EXPIRES")
        y2, e2 = ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
    np.testing.assert_array_equal(y, y2)
    np.testing.assert_array_equal(e, e2)


def test_product64_warps_leave_together(monkeypatch):
    """One lane of a read-out warp in the FP64 panel product: the block's other warps
    follow, the solve reports an error (the rows left out may show as a residual that
    is not finite first), and the next one is as if nothing had been."""
    import paper_1708_09705_gb300 as gm
    from synth import make_catalogue
    cat = make_catalogue("c1_plain_400", n=1100, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, cg_tol=1e-12, warm_start=0)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    monkeypatch.setenv("GM_SPMM", "tc")
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        ctx.set_sites(tau, tau * np.log(A))
        var = ctx.get_posterior()[1]
        assert ctx.stats()["tile_ksteps"] > 9 * 8          # more than one read-out a block
        for _ in range(3):
            monkeypatch.setenv("GM_WAIT_EXPIRES", "product64")
            ctx.set_sites(tau, tau * np.log(A))
            with pytest.raises(gm.GmError) as err:
                ctx.get_posterior()
            assert err.value.status in (TIMEOUT, 4, 6)
            monkeypatch.delenv("GM_WAIT_EXPIRES")
            ctx.set_sites(tau, tau * np.log(A))
            np.testing.assert_array_equal(ctx.get_posterior()[1], var)
