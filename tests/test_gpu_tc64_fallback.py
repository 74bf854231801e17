"""FP64 panel products go without the tensor cores' tiles where these do not fit the
memory or hold too few entries: same posteriors as with the FP64 units pinned, no error.
(Both solves stop at a relative residual of 1e-13, amplified by K_ii / Sigma_ii <= 1e4
in the variances: rtol 1e-9.)"""
import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


class _Pool:
    """torch's caching allocator with a limit on the live bytes and refused sizes."""

    def __init__(self):
        self.live, self.peak, self.sizes, self.limit, self.refuse = {}, 0, [], None, ()
        self.refused = 0

    def allocator(self, device):
        import torch
        from paper_1708_09705_gb300 import gmead as g

        def alloc(n, stream, user):
            used = sum(self.live.values())
            if n in self.refuse or (self.limit is not None and used + n > self.limit):
                self.refused += 1
                return None
            p = int(torch.cuda.caching_allocator_alloc(max(int(n), 1), device=device,
                                                       stream=int(stream or 0)))
            self.live[p] = n
            self.sizes.append(n)
            self.peak = max(self.peak, used + n)
            return p

        def free(p, n, stream, user):
            del self.live[p]
            torch.cuda.caching_allocator_delete(int(p))

        fa, ff = g._ALLOC_FN(alloc), g._FREE_FN(free)
        return g.Allocator(fa, ff, None), (fa, ff)


def _posterior(pool, monkeypatch, cat, **kw):
    import paper_1708_09705_gb300 as gm
    from paper_1708_09705_gb300 import gmead as g
    monkeypatch.setattr(g, "_torch_allocator", pool.allocator)
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, cg_tol=1e-13, **kw)
    A = np.maximum(cat["A_obs"], 0.02)
    tau = (A / cat["A_sigma"]) ** 2
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        out = []
        for _ in range(2):                         # the second keeps the first's decision
            ctx.set_sites(tau, tau * np.log(A))
            out.append(ctx.get_posterior())
        st = ctx.stats()
    assert not pool.live
    return out, st


def _same(a, b):
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            np.testing.assert_allclose(u, v, rtol=1e-9, atol=1e-11)


@pytest.mark.parametrize("what", ["images", "planes", "budget"])
def test_no_memory_for_the_tiles(what, monkeypatch):
    cat = make_catalogue("c1_plain_400", n=1400, truth="mean")
    base, free = _Pool(), _Pool()
    monkeypatch.setenv("GM_SPMM", "simt")
    want, st = _posterior(base, monkeypatch, cat)
    assert st["tile_ksteps"] == 0
    monkeypatch.delenv("GM_SPMM")
    got, st = _posterior(free, monkeypatch, cat)
    assert st["tile_ksteps"] > 0
    _same(got, want)
    short = _Pool()
    if what == "images":
        short.refuse = (st["tile_ksteps"] * 32768,)
    elif what == "planes":
        short.refuse = (1400 * 1408 * 16,)
    else:
        short.limit = base.peak + 65536             # what the FP64 units need
    assert what == "budget" or short.refuse[0] in free.sizes
    got, st = _posterior(short, monkeypatch, cat)
    assert short.refused > 0 and st["tile_ksteps"] == 0
    _same(got, want)


@pytest.mark.parametrize("n,side,L0,panel,used", [(2100, 20.0, 5.0, 0, False),
                                                  (12000, 30.0, 5.0, 1024, False),
                                                  (3000, 20.0, 8.0, 0, True)])
def test_sparse_rows_keep_the_fp64_units(n, side, L0, panel, used, monkeypatch):
    """Fills of 0.035 (short rows), 0.07 (counted) and 0.12."""
    import paper_1708_09705_gb300 as gm
    rng, deg = np.random.default_rng(1), np.pi / 180
    l, b = rng.uniform(0, side * deg, n), np.arcsin(rng.uniform(0, np.sin(side * deg), n))
    s = np.exp(rng.uniform(np.log(100), np.log(3000), n))
    A = 1e-3 * s * np.exp(0.3 * rng.standard_normal(n))
    cfg = gm.default_config(outer_scale_pc=L0, cutoff_pc=3 * L0, n_nodes=16, rhs_panel=panel,
                            quad_rule=gm.QUAD_GL, precision=gm.PREC_FP64, cg_tol=1e-6)
    monkeypatch.delenv("GM_SPMM", raising=False)
    with gm.ep_init(cfg, l, b, s, A, np.full(n, 0.05)) as ctx:
        ctx.profile(True)
        ctx.build_cov()
        ctx.set_sites((A / 0.05) ** 2, (A / 0.05) ** 2 * np.log(A))
        ctx.get_posterior()
        ran = ctx.kernel_times()
        assert (ctx.stats()["tile_ksteps"] > 0) == used
    assert ("k_panel_spmm_tc64" in ran) == used and ("k_panel_spmm" in ran) != used
