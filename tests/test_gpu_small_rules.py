"""Where FP64 solves run one block per column: a mean solve by its stored entries, the
columns by the share of an SM, neither when the sliced rows do not fit the memory or
the product is pinned to simt or tc.  Same posteriors either way (both solves stop at a
relative residual of 1e-13, amplified by K_ii / Sigma_ii <= 1e4: rtol 1e-9)."""
import numpy as np
import pytest

from synth import make_catalogue
from test_gpu_tc64_fallback import _Pool, _posterior, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,columns,mean", [(400, True, "block"), (513, True, "launch"),
                                            (700, False, "launch")])
def test_rules(n, columns, mean, monkeypatch):
    """12,964 entries; 24,023 (4 columns a SM: 9.6e4); 44,000 x 5: 2.2e5."""
    import paper_1708_09705_gb300 as gm
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, cg_tol=1e-13)
    res = {}
    for mode in ("simt", "auto", ""):
        monkeypatch.setenv("GM_SPMM", mode)
        with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
            ctx.profile(True)
            ctx.build_cov()
            ctx.set_sites(tau, tau * np.log(A))
            res[mode] = ctx.get_posterior()
            ran = ctx.kernel_times()
        pinned = mode == "simt"
        assert ("k_cg_run" in ran) == (pinned or mean == "launch")
        blocks = 0 if pinned else int(columns) + (mean == "block")
        assert ran.get("k_cg_columns", (0,))[0] == blocks
    for mode in ("auto", ""):
        for a, b in zip(res["simt"], res[mode]):
            np.testing.assert_allclose(b, a, rtol=1e-9, atol=1e-11)


def test_no_memory_for_the_sliced_rows(monkeypatch):
    cat = make_catalogue("c1_plain_400", n=400, truth="mean")
    base, free, short = _Pool(), _Pool(), _Pool()
    monkeypatch.setenv("GM_SPMM", "simt")
    want = _posterior(base, monkeypatch, cat)[0]
    monkeypatch.delenv("GM_SPMM")
    _same(_posterior(free, monkeypatch, cat)[0], want)
    short.limit = base.peak + 16384                 # the sliced rows take 160 KB at least
    assert free.peak > short.limit
    _same(_posterior(short, monkeypatch, cat)[0], want)
    assert short.refused > 0
