"""The undeflated FP32 variance panels write the BF16 planes of the asynchronous
tile product from their update; the other product variants split the FP32 panel
themselves.  Same split, same sums: equal bit for bit, at star counts beside the
tile's 128 rows and the panel's 32 columns, for the stars' and the queries'
panels, with columns that freeze early and more panels than one."""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,panel", [(33, 0), (128, 0), (129, 64), (301, 0), (517, 96)])
def test_planes_equal_panel_split(n, panel, monkeypatch):
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP32, cg_tol=1e-6, rhs_panel=panel)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    tau[::5] = 0.0                                   # right-hand sides that converge at once
    res = {}
    for v in ("1", "4"):
        monkeypatch.setenv("GM_TC_PREFETCH", v)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            res[v] = ctx.get_posterior() + ctx.predict(cat["l"][:50], cat["b"][:50],
                                                       cat["s"][:50] + 1.0)
    for a, b in zip(res["1"], res["4"]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("probe", [0.0, 2.0])
def test_packed_planes_equal_panel_split(probe, monkeypatch):
    """The packed panels of several fields: sizes beside a row segment (64), a
    tile block (128) and one star; the planes written by the direction update
    against the split of the FP32 panel, bit for bit."""
    import paper_1708_09705_gb300 as gm
    cats = [make_catalogue("c1_plain_400", n=k, seed=f, truth="mean")
            for f, k in enumerate((1, 63, 65, 128, 200, 257))]
    cat = {k: np.concatenate([c[k] for c in cats]) for k in ("l", "b", "s", "A_obs", "A_sigma")}
    fid = np.repeat(np.arange(len(cats)), [len(c["s"]) for c in cats])
    L0 = np.linspace(15.0, 30.0, len(cats))
    cfg = gm.config_from_catalogue(cats[0], precision=gm.PREC_FP32, cg_tol=1e-6,
                                   probe_factor=probe)
    res = {}
    for v in ("1", "4"):
        monkeypatch.setenv("GM_TC_PREFETCH", v)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"],
                        field_id=fid, field_L0=L0, field_cutoff=3 * L0) as ctx:
            ctx.build_cov()
            ctx.ep_sweep(2)
            res[v] = ctx.get_posterior()
    for a, b in zip(res["1"], res["4"]):
        np.testing.assert_array_equal(a, b)
