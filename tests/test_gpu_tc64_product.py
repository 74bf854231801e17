"""The FP64 panel product of the tensor cores (gm::panel_spmm_tc64, Q = P + d o (K PD))
against exact rational arithmetic.  The digits keep 2^-62 of the row's and the column's
largest entry and leave out the products of weight 2^-76 and less: below 2^-57 of the
two maxima per stored entry.  Then the sum is rounded, scaled by d and added to P: four
roundings.  Panel widths of both block shapes, entries and columns of very different
scale, zero columns, a column of subnormal numbers (zero to it), P . Q per block."""
import ctypes as C
from fractions import Fraction as F

import numpy as np
import pytest

from synth import make_catalogue

pytestmark = pytest.mark.gpu


def _product(ctx, n, R, d, P, PD):
    import torch
    import paper_1708_09705_gb300 as gm
    L = gm.lib()
    prepare = getattr(L, "_ZN2gm12tc64_prepareEP6gm_ctxl")
    prepare.argtypes, prepare.restype = [C.c_void_p, C.c_int64], C.c_int
    prod = getattr(L, "_ZN2gm15panel_spmm_tc64EP6gm_ctxliPKdS3_S3_PdS4_")
    prod.argtypes = [C.c_void_p, C.c_int64, C.c_int] + [C.c_void_p] * 5
    prod.restype = C.c_int
    t = [torch.tensor(v, device="cuda") for v in (d, P, PD)]
    Q = torch.full((n, R), np.nan, dtype=torch.float64, device="cuda")
    part = torch.full((-(-n // 128), R), np.nan, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert prepare(ctx._h, R) == 0 and ctx.stats()["tile_ksteps"] > 0
    assert prod(ctx._h, n, R, *(v.data_ptr() for v in t), Q.data_ptr(), part.data_ptr()) == 0
    torch.cuda.synchronize()
    return Q.cpu().numpy(), part.cpu().numpy()


@pytest.mark.parametrize("n,R", [(129, 32), (300, 96), (700, 64), (1400, 2016)])
def test_product_against_exact_sums(n, R, monkeypatch):
    import paper_1708_09705_gb300 as gm
    monkeypatch.setenv("GM_SPMM", "tc")
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64)
    rng = np.random.default_rng(n)
    d = 10.0 ** rng.uniform(-4, 1, n)
    P = rng.standard_normal((n, R))
    PD = rng.standard_normal((n, R)) * 10.0 ** rng.uniform(-9, 0, (n, R))
    PD *= 10.0 ** rng.uniform(-30, 30, R)
    PD[:, 3] = 0.0
    PD[:, 5] = 5e-324 * rng.integers(0, 99, n)
    PD[::2, 7] = 0.0
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], cat["A_obs"], cat["A_sigma"]) as ctx:
        ctx.build_cov()
        rp, col, val = ctx.get_csr()
        Q, part = _product(ctx, n, R, d, P, PD)
    rows = np.unique(np.r_[0, n // 2, n - 1, rng.integers(0, n, 25)])
    cols = np.unique(np.r_[0, 3, 5, 7, 31, R - 1, rng.integers(0, R, 6)])
    for i in rows:
        e = slice(rp[i], rp[i + 1])
        v, j = val[e], col[e]
        rmax = np.abs(v).max()
        for c in cols:
            x = np.where(np.abs(PD[j, c]) < 2.3e-308, 0.0, PD[j, c])
            s = sum((F(float(a)) * F(float(b)) for a, b in zip(v, x)), F(0))
            ref = F(float(P[i, c])) + F(float(d[i])) * s
            cut = len(v) * F(float(rmax)) * F(float(np.abs(PD[:, c]).max())) / 2 ** 57
            tol = F(float(d[i])) * (abs(s) * 3 / 2 ** 53 + cut) + abs(ref) / 2 ** 53
            assert abs(F(float(Q[i, c])) - ref) <= tol, (i, c)
    # every element against the FP64 sum, every block's P . Q
    K = np.zeros((n, n))
    K[np.repeat(np.arange(n), np.diff(rp)), col] = val
    ref = P + d[:, None] * (K @ PD)
    scale = np.abs(P) + d[:, None] * (np.abs(K).max(1)[:, None] * np.abs(PD).max(0))
    assert np.all(np.abs(Q - ref) <= 1e-13 * scale)
    np.testing.assert_allclose(part.sum(0), (P * Q).sum(0), rtol=0,
                               atol=1e-12 * np.abs(P * Q).sum(0).max())
