"""The single-right-hand-side solve in one cooperative launch against its launches per
step (GM_CG=launches): bit for bit, for both precisions, star counts beside a block's
256 vector threads and beyond one pass of the grid, an iteration cap between two checks
(the refinement goes on behind it) and several fields."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,fp32,cap", [(1, True, 0), (255, True, 0), (257, False, 0), (1500, False, 0),
                                        (1500, True, 13), (6000, True, 0)])
def test_whole_solve_keeps_the_bits(n, fp32, cap, monkeypatch):
    import paper_1708_09705_gb300 as gm
    monkeypatch.setenv("GM_SPMM", "simt")         # FP64: no per-column blocks
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP32 if fp32 else gm.PREC_FP64,
                                   cg_tol=1e-8 if fp32 else 1e-12, deflate=0, probe_factor=2.0)
    if cap:
        cfg.cg_max_iter = cap
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    res = []
    for mode in ("launches", "one"):
        monkeypatch.setenv("GM_CG", mode)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.profile(True)
            ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            mu = ctx.get_posterior()[0]
            res.append((mu, ctx.stats()["cg_iters_mean"]))
            assert ("k_cg_run" in ctx.kernel_times()) == (mode == "one")
            assert ("k_apply_B" in ctx.kernel_times()) == (mode != "one")
    np.testing.assert_array_equal(res[0][0], res[1][0])
    assert res[0][1] == res[1][1] > 0


def test_fields_keep_the_bits(monkeypatch):
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=900, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP32, probe_factor=2.0)
    field = (np.arange(900) % 3).astype(np.int32)
    res = []
    for mode in ("launches", "one"):
        monkeypatch.setenv("GM_CG", mode)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"],
                        field_id=field, field_L0=np.array([10.0, 20.0, 15.0]),
                        field_cutoff=np.array([30.0, 60.0, 45.0])) as ctx:
            ctx.build_cov()
            ctx.ep_sweep(1)
            res.append(ctx.get_posterior())
    for a, b in zip(*res):
        np.testing.assert_array_equal(a, b)
