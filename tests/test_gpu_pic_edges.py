"""PIC posterior and predictive against the oracle's dense conditioning where the
device steps change form: inducing counts and sub-catalogue sizes beside 32 lanes and
beside the largest matrix factorised in shared memory, empty sub-catalogues, queries
beyond the cutoff of every inducing point or of their own sub-catalogue, one query,
both tapers."""
import numpy as np
import pytest

import oracle as O
from oracle import pic as P
from synth import catalogue_subset, make_catalogue

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,sizes,nq,taper", [
    (1, (1, 2, 31), 1, 0), (31, (32, 0, 33), 33, 0), (32, (64, 65), 7, 0),
    (33, (1, 100), 70, 0), (65, (250,), 12, 0), (250, (40,), 5, 0), (2, (40,), 9, 1)])
def test_pic_sizes(R, sizes, nq, taper):
    import paper_1708_09705_gb300 as gm
    n = sum(sizes)
    cat = catalogue_subset(make_catalogue("c1_plain_400", truth="mean"), np.arange(n))
    rng = np.random.default_rng(100 * R + n)
    li = rng.uniform(cat["l"].min(), cat["l"].max(), R)
    bi = rng.uniform(cat["b"].min(), cat["b"].max(), R)
    si = np.exp(rng.uniform(np.log(150), np.log(2500), R))
    ql = rng.uniform(cat["l"].min(), cat["l"].max(), nq)
    qb = rng.uniform(cat["b"].min(), cat["b"].max(), nq)
    qs = np.exp(rng.uniform(np.log(100), np.log(4000), nq))
    ql[0], qb[0], qs[0] = cat["l"][0], cat["b"][0], 0.99 * cat["s"][0]
    union = dict(cat, l=np.concatenate([cat["l"], li, ql]), b=np.concatenate([cat["b"], bi, qb]),
                 s=np.concatenate([cat["s"], si, qs]))
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, likelihood=gm.LIK_GAUSS_IN_LNA)
    cfg.taper = taper
    cv = O.build_cov(union, taper=O.TAPER_HARD if taper else O.TAPER_WENDLAND)
    K, m = cv["K"], cv["m"]
    # a noise that keeps K + noise positive definite under the hard cutoff too
    A = np.clip(cat["A_obs"], 0.02, None)
    atil = np.log(A) + 0.02 * rng.standard_normal(n)
    sig = cat["A_sigma"] / A + (2.0 if taper else 0.0)
    blk = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    rng.shuffle(blk)
    u = np.arange(n, n + R)
    groups = [np.flatnonzero(blk == k) for k in range(len(sizes))]
    blocks = [dict(Kku=K[np.ix_(g, u)], Kkk=K[np.ix_(g, g)], m=m[g], atil=atil[g],
                   sig2=sig[g] ** 2) for g in groups]
    ref_m, ref_c = P.pitc_posterior_direct(K[np.ix_(u, u)], [b for b in blocks if len(b["m"])], m[u])
    qblk = rng.integers(0, len(sizes), nq).astype(np.int32)
    with gm.ep_init(cfg, cat["l"], cat["b"], cat["s"], atil, sig) as ctx:
        ctx.build_cov()
        mean, cov = ctx.pic_posterior(blk, li, bi, si)
        pm, pv = ctx.pic_predict(qblk, ql, qb, qs)
    # the tolerances of the oracle comparison at 300 stars and 40 points
    np.testing.assert_allclose(mean, ref_m, rtol=1e-7, atol=1e-9)
    np.testing.assert_allclose(cov, ref_c, rtol=1e-6, atol=1e-10)
    for q in range(nq):
        k, j = qblk[q], n + R + q
        mm, vv = P.pic_predict(K[np.ix_(u, u)], m[u], ref_m, ref_c, blocks[k],
                               K[np.ix_([j], u)], np.diag(K)[[j]], K[np.ix_([j], groups[k])], m[[j]])
        assert pm[q] == pytest.approx(mm[0], rel=1e-7, abs=1e-9)
        assert pv[q] == pytest.approx(vv[0], rel=1e-6, abs=1e-10)


def test_pic_vectors_beyond_shared_memory():
    """A sub-catalogue whose solve vectors are kept in device memory (3,100 stars):
    the oracle's formulas on the covariance that a context of all points holds."""
    import paper_1708_09705_gb300 as gm
    n, R, nq = 3100, 3, 5
    cat = make_catalogue("c1_plain_400", n=n, truth="mean")
    rng = np.random.default_rng(5)
    f = 6.0                                             # a wide field: a sparse K
    l = cat["l"].mean() + (cat["l"] - cat["l"].mean()) * f
    b = cat["b"].mean() + (cat["b"] - cat["b"].mean()) * f
    j = rng.choice(n, R + nq, replace=False)
    ll, bb, ss = l[j] + 2e-4, b[j] - 1e-4, 0.97 * cat["s"][j]
    atil = np.log(np.clip(cat["A_obs"], 0.02, None))
    sig = cat["A_sigma"] / np.clip(cat["A_obs"], 0.02, None)
    cfg = gm.config_from_catalogue(cat, precision=gm.PREC_FP64, likelihood=gm.LIK_GAUSS_IN_LNA)
    L, B, S = (np.concatenate(x) for x in ((l, ll), (b, bb), (cat["s"], ss)))
    one = np.ones(len(L))
    with gm.ep_init(cfg, L, B, S, one, one) as ctx:
        ctx.build_cov()
        rp, col, val = ctx.get_csr()
        perm, m = ctx.get_perm(), ctx.get_prior()[0]
    K = np.zeros((len(L), len(L)))
    K[perm[np.repeat(np.arange(len(L)), np.diff(rp))], perm[col]] = val
    u, g = np.arange(n, n + R), np.arange(n)
    blocks = [dict(Kku=K[np.ix_(g, u)], Kkk=K[np.ix_(g, g)], m=m[g], atil=atil, sig2=sig ** 2)]
    ref_m, ref_c = P.pitc_posterior_direct(K[np.ix_(u, u)], blocks, m[u])
    with gm.ep_init(cfg, l, b, cat["s"], atil, sig) as ctx:
        ctx.build_cov()
        mean, cov = ctx.pic_posterior(np.zeros(n, np.int32), ll[:R], bb[:R], ss[:R])
        pm, pv = ctx.pic_predict(np.zeros(nq, np.int32), ll[R:], bb[R:], ss[R:])
    np.testing.assert_allclose(mean, ref_m, rtol=1e-7, atol=1e-9)
    np.testing.assert_allclose(cov, ref_c, rtol=1e-6, atol=1e-10)
    q = np.arange(n + R, n + R + nq)
    mm, vv = P.pic_predict(K[np.ix_(u, u)], m[u], ref_m, ref_c, blocks[0], K[np.ix_(q, u)],
                           np.diag(K)[q], K[np.ix_(q, g)], m[q])
    np.testing.assert_allclose(pm, mm, rtol=1e-7, atol=1e-9)
    np.testing.assert_allclose(pv, vv, rtol=1e-6, atol=1e-10)
