"""Band-rule assembly at the geometries where its panel bookkeeping can go
wrong, against the oracle's band rule: distances shorter than the first panel,
beyond the truncation at 40 outer scales, equal distances (the kink at zero),
pairs on one sightline (chord 0), duplicated stars; and list lengths around
the batches a warp takes.  Tolerances as for the band rule's parity test."""
import numpy as np
import pytest

from oracle import band as Bd
from synth import make_catalogue

pytestmark = pytest.mark.gpu
RULE = dict(n=6, h0=1e-3, q=3.0, m0=0.25, K=40.0)


def _catalogue(kind, n):
    r = np.random.default_rng(n)
    if kind == "field":
        return make_catalogue("c1_plain_400", n=n, truth="mean")
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    s = {"near": np.exp(r.uniform(np.log(0.005), np.log(70.0), n)),
         "far": r.uniform(780.0, 830.0, n),
         "sightline": np.exp(r.uniform(np.log(20.0), np.log(2500.0), n))}[kind]
    cat["s"] = s
    if kind == "sightline":
        cat["l"], cat["b"] = np.full(n, 0.01), np.full(n, 0.01)
        cat["s"][n // 2:] = cat["s"][:n - n // 2]        # duplicates, equal distances
    elif kind == "far":
        cat["s"][::3] = 800.0                             # s = 40 outer scales exactly
    return cat


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind,n", [("field", 1), ("field", 2), ("field", 33), ("field", 90),
                                    ("near", 40), ("far", 24), ("sightline", 40)])
def test_band_edges(prec, kind, n):
    import paper_1708_09705_gb300 as gm
    cat = _catalogue(kind, n)
    ref = Bd.build_cov_band(cat, **RULE)
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64 if prec == "fp64" else gm.PREC_FP32,
                                   quad_rule=gm.QUAD_BAND)
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        i, j = np.nonzero(ref["K"])
        got = ctx.get_entries(i, j)
        kd = ctx.get_prior()[1]
    tol = 1e-9 if prec == "fp64" else 2e-5
    np.testing.assert_allclose(got, ref["K"][i, j], rtol=tol, atol=1e-12 if prec == "fp64" else 1e-9)
    np.testing.assert_allclose(kd, ref["diag"], rtol=tol)
