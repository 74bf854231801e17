"""Covariance entries of the Q-node rule at node counts around the lanes (1, 2 or
4 nodes a lane) and at geometries with coinciding nodes (one sightline, equal
distances, duplicated stars) and separations beyond the kernel table, FP64
(1e-9, the table's error) and FP32 (2e-5), against the oracle."""
import numpy as np
import pytest

import oracle as O
from synth import make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("Q", [2, 31, 32, 33, 64, 65, 100, 128])
def test_entries(prec, Q):
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=60, truth="mean")
    cat["n_nodes"] = Q
    cat["s"][:4] = [3.0, 3.0, 2900.0, 2950.0]
    for k in ("l", "b"):
        cat[k][:12] = cat[k][0]                   # one sightline
    cat["s"][12:16] = cat["s"][16:20]             # equal distances
    for k in ("l", "b", "s"):
        cat[k][20:22] = cat[k][22:24]             # duplicates
    ref = O.build_cov(cat)
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64 if prec == "fp64" else gm.PREC_FP32)
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        i, j = np.nonzero(ref["K"])
        got = ctx.get_entries(i, j)
        m, kd = ctx.get_prior()
    tol = 1e-9 if prec == "fp64" else 2e-5
    np.testing.assert_allclose(got, ref["K"][i, j], rtol=tol, atol=1e-12 if prec == "fp64" else 1e-9)
    np.testing.assert_allclose(kd, np.diag(ref["K"]), rtol=tol)
    # the prior mean carries half of the diagonal's error, whatever its own size
    np.testing.assert_allclose(m + 0.5 * kd, np.log(cat["rho_bar"] * cat["s"]), rtol=1e-13, atol=1e-13)
