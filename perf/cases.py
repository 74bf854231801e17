"""Performance cases of the extinction mapper: the calls a mapping program makes,
over the sizes of the repository's workloads (400-star field in FP64 up to the
20,000-star field in FP32), each through the public binding or C ABI.

A case is a dict of plain values.  prepare() makes the inputs from the seed
alone and the context a program keeps; run() is one pass and returns what the
pass computes; exact() restates the same quantities in FP64 with torch, from
the formulae (no code of the library).  Results of FP32 contexts are returned
in FP32, the precision they are computed in, although the API hands out
doubles.

Catalogues: stars uniform in a square field at b = 0 .. side (as the
workloads), distances log-uniform 100-3000 pc, extinctions the line integrals
of exp(f) for a log-density field f with the model's own spectrum
P(k) ~ (k^2 + k0^2)^(-11/6) (random Fourier modes), 0.05 mag of noise.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1708_09705_gb300 as gm

DEG = math.pi / 180.0
RHO, SIGMA2, NOISE = 1e-3, 1.0, 0.05     # mag/pc, log-density variance, mag
S_LO, S_HI = 100.0, 3000.0               # pc


# --------------------------------------------------------------------- cases
def listed():
    return [
        # The smallest call: the allocation-free site update of a service loop
        # on the 400-star field (latency of a launch and a small read-back).
        dict(name="site_400", kind="site", n=400, lik=0, damping=1.0),
        # The whole plain FP64 run on the 400-star field: assembly, three
        # sweeps, posterior (32 nodes; many small launches).
        dict(name="ep_fp64_400", kind="ep", n=400, side=1.0, L0=20.0, nodes=32, rule="gl",
             prec="fp64", probe=0.0, deflate=0, products=6, sweeps=3, tol=1e-12),
        # Posterior of given sites in FP64 with exact variances (one solve per
        # star) on a field of 2,001 stars: the reference form.
        dict(name="posterior_fp64_2001", kind="posterior", n=2001, side=3.0, L0=20.0, nodes=64,
             rule="gl", prec="fp64", probe=0.0, deflate=0, products=6, tol=1e-12),
        # The plain FP32 form with exact variances at 4,000 stars (the size at
        # which the forms are compared).
        dict(name="posterior_fp32_4000", kind="posterior", n=4000, side=3.0, L0=20.0, nodes=64,
             rule="gl", prec="fp32", probe=0.0, deflate=0, products=6, tol=1e-6),
        # The benchmark's step at one sweep: 20,000 stars, FP32, probed
        # variances, deflated preconditioner; assembly, a sweep, posterior.
        # (Over several sweeps the solves' stopping error, 1e-5 of a residual,
        # travels through the sites, and results say less about a change.)
        dict(name="ep_fp32_20000", kind="ep", n=20000, side=5.0, L0=20.0, nodes=64, rule="gl",
             prec="fp32", probe=2.0, deflate=64, products=6, sweeps=1, tol=1e-6),
        # Assembly alone, 64-node rule, FP32, the 20,000-star field; the
        # program reads the entries of its pair list and the prior.
        dict(name="cov_gl_fp32_20000", kind="cov", n=20000, side=5.0, L0=20.0, nodes=64,
             rule="gl", prec="fp32"),
        # Assembly with the library's default (converged band) rule, FP32.
        dict(name="cov_band_fp32_6000", kind="cov", n=6000, side=5.0, L0=20.0, nodes=64,
             rule="band", prec="fp32"),
        # Batched fields of uneven size (the 256-field workload, a sixteenth
        # of its fields, at the lower end of its star counts): assembly, a
        # sweep, posterior.
        dict(name="fields_fp32_16", kind="fields", fields=16, nmin=500, nmax=2000, nodes=64,
             probe=2.0, sweeps=1, tol=1e-6),
        # Map points: predictive mean and variance at query points from a
        # kept posterior.
        dict(name="predict_fp32_8000x1000", kind="predict", n=8000, side=5.0, L0=20.0, nodes=64,
             rule="gl", prec="fp32", probe=2.0, deflate=64, products=6, tol=1e-6, queries=1000),
        # Samples conditioned on dA/ds >= 0: 16 points per sightline, 20 of
        # 120 steps burnt in.
        dict(name="sampler_4096x16", kind="sampler", sightlines=4096, points=16, steps=120,
             burn=20),
        # PIC posterior and predictive: sub-catalogues of a 6 x 6 grid, 140
        # inducing points, FP64.
        dict(name="pic_fp64_6000", kind="pic", n=6000, side=5.0, L0=20.0, nodes=64, grid=6,
             inducing=140, queries=4000),
        # Covariance surrogate inference on a block of pairs.
        dict(name="surrogate_1m", kind="mlp", n=1000000),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["site", "ep64", "ep32", "post64", "post32", "cov_gl", "cov_band",
                       "cov_gl64", "fields", "predict", "predict64", "sampler", "pic", "mlp"])
    side = rng.choice([1.0, 2.0, 3.0, 5.0])
    L0 = round(rng.uniform(10.0, 25.0), 2)
    if kind == "site":
        return dict(kind="site", n=_logint(rng, 200, 1000000), lik=rng.choice([0, 1]),
                    damping=rng.choice([1.0, 0.7]))
    if kind == "ep64":
        return dict(kind="ep", n=_logint(rng, 150, 1000), side=side, L0=L0,
                    nodes=rng.choice([32, 48, 64]), rule=rng.choice(["gl", "band"]), prec="fp64",
                    probe=rng.choice([0.0, 3.0]), deflate=0, products=6, sweeps=3, tol=1e-12)
    if kind == "ep32":
        return dict(kind="ep", n=_logint(rng, 1000, 14000), side=rng.choice([4.0, 5.0]),
                    L0=round(rng.uniform(10.0, 20.0), 2), nodes=rng.choice([32, 64]),
                    rule=rng.choice(["gl", "band"]), prec="fp32", probe=2.0, deflate=64,
                    products=rng.choice([6, 6, 3]), sweeps=1, tol=1e-6)
    if kind == "post64":
        return dict(kind="posterior", n=_logint(rng, 300, 2200), side=rng.choice([2.0, 3.0, 5.0]),
                    L0=L0, nodes=64, rule=rng.choice(["gl", "band"]), prec="fp64",
                    probe=rng.choice([0.0, 2.0]), deflate=0, products=6, tol=1e-12)
    if kind == "post32":
        return dict(kind="posterior", n=_logint(rng, 500, 6000), side=rng.choice([3.0, 5.0]),
                    L0=L0, nodes=64, rule="gl", prec="fp32", probe=rng.choice([0.0, 2.0]),
                    deflate=rng.choice([0, 64]), products=rng.choice([6, 6, 3]), tol=1e-6)
    if kind == "cov_gl":
        return dict(kind="cov", n=_logint(rng, 500, 16000), side=rng.choice([3.0, 5.0]),
                    L0=round(rng.uniform(10.0, 20.0), 2), nodes=rng.choice([24, 32, 64, 100]),
                    rule="gl", prec="fp32")
    if kind == "cov_band":
        return dict(kind="cov", n=_logint(rng, 300, 6000), side=rng.choice([3.0, 5.0]), L0=L0,
                    nodes=64, rule="band", prec="fp32")
    if kind == "cov_gl64":
        return dict(kind="cov", n=_logint(rng, 200, 3000), side=side, L0=L0,
                    nodes=rng.choice([32, 64]), rule=rng.choice(["gl", "band"]), prec="fp64")
    if kind == "fields":
        lo = rng.choice([200, 500])
        return dict(kind="fields", fields=rng.randint(3, 16), nmin=lo,
                    nmax=rng.choice([1000, 2000]), nodes=64, probe=rng.choice([0.0, 2.0]),
                    sweeps=1, tol=1e-6)
    if kind == "predict":
        return dict(kind="predict", n=_logint(rng, 1000, 10000), side=5.0, L0=L0, nodes=64,
                    rule="gl", prec="fp32", probe=2.0, deflate=64, products=6, tol=1e-6,
                    queries=_logint(rng, 1, 2000))
    if kind == "predict64":
        return dict(kind="predict", n=_logint(rng, 300, 2000), side=rng.choice([2.0, 3.0]), L0=L0,
                    nodes=64, rule=rng.choice(["gl", "band"]), prec="fp64", probe=0.0, deflate=0,
                    products=6, tol=1e-12, queries=_logint(rng, 1, 1500))
    if kind == "sampler":
        m = rng.choice([2, 5, 8, 16, 24, 32, 40])
        return dict(kind="sampler", sightlines=max(1, _logint(rng, 16, 65536) // m), points=m,
                    steps=rng.choice([30, 60, 120]), burn=rng.choice([0, 10, 20]))
    if kind == "pic":
        return dict(kind="pic", n=_logint(rng, 400, 6000), side=rng.choice([3.0, 5.0]), L0=L0,
                    nodes=rng.choice([32, 64]), grid=rng.choice([4, 5, 6]), inducing=_logint(rng, 10, 140),
                    queries=_logint(rng, 50, 4000))
    return dict(kind="mlp", n=_logint(rng, 100, 1000000))


# -------------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _extinctions(rng, l, b, s, L0):
    """Line integrals of exp(f) by 256 midpoints, f from 384 Fourier modes
    drawn from the spectrum (k is a multivariate t with 2/3 degrees of
    freedom in units of k0)."""
    dev, M, T = _dev(), 384, 256
    k = rng.standard_normal((M, 3)) / np.sqrt(2.0 * rng.gamma(1.0 / 3.0, 1.0, (M, 1))) / L0
    ph = torch.tensor(rng.uniform(0, 2 * math.pi, M), dtype=torch.float32, device=dev)
    u = np.stack([np.cos(b) * np.cos(l), np.cos(b) * np.sin(l), np.sin(b)], 1)
    w = torch.tensor(u @ k.T, dtype=torch.float32, device=dev)          # n x M
    st = torch.tensor(s, dtype=torch.float32, device=dev)
    out = torch.empty(len(s), dtype=torch.float64, device=dev)
    mid = (torch.arange(T, device=dev, dtype=torch.float32) + 0.5) / T
    for i0 in range(0, len(s), 512):
        t = st[i0:i0 + 512, None] * mid                                   # stars x T
        f = torch.cos(w[i0:i0 + 512, None, :] * t[:, :, None] + ph).sum(-1)
        f = f * math.sqrt(2.0 * SIGMA2 / M) - 0.5 * SIGMA2
        out[i0:i0 + 512] = (RHO * torch.exp(f)).double().mean(1) * st[i0:i0 + 512].double()
    return out.cpu().numpy()


def _catalogue(rng, n, side, L0, l0=0.0, b0=0.0):
    l = rng.uniform(l0 * DEG, (l0 + side) * DEG, n)
    b = np.arcsin(rng.uniform(math.sin(b0 * DEG), math.sin((b0 + side) * DEG), n))
    s = np.exp(rng.uniform(math.log(S_LO), math.log(S_HI), n))
    A = _extinctions(rng, l, b, s, L0) + NOISE * rng.standard_normal(n)
    return dict(l=l, b=b, s=s, A=A, sig=np.full(n, NOISE))


def _rng(seed):
    return np.random.default_rng([int(seed), 17080970])


def _t(a, dtype=torch.float64):
    return torch.as_tensor(a, dtype=dtype, device=_dev())


def _config(c, **kw):
    f32 = c.get("prec") == "fp32"
    base = dict(sigma2=SIGMA2, outer_scale_pc=c["L0"], rho_bar=RHO, cutoff_pc=3.0 * c["L0"],
                n_nodes=c["nodes"],
                quad_rule=gm.QUAD_BAND if c.get("rule") == "band" else gm.QUAD_GL,
                precision=gm.PREC_FP32 if f32 else gm.PREC_FP64,
                probe_factor=c.get("probe", 0.0), deflate=c.get("deflate", 0),
                tc_products=c.get("products", 6), cg_tol=c.get("tol", 1e-10))
    base.update(kw)
    return gm.default_config(**base)


def _context(c, cat, **kw):
    return gm.ep_init(_config(c, **kw), *(_t(cat[k]) for k in ("l", "b", "s", "A", "sig")))


def _sites(cat):
    """Sites of the observations: ln A with standard deviation sigma / A."""
    A = np.maximum(cat["A"], 0.02)
    tau = (A / cat["sig"]) ** 2
    return tau, tau * np.log(A)


def _pairs(cat, cut, room=0):
    """Unique pairs (i <= j) within the cutoff, on the device; with room, the
    list filled up to that length with the first star's own entry."""
    x = _t(_unit(cat["l"], cat["b"]) * cat["s"][:, None])
    n, out = len(x), []
    for i0 in range(0, n, 1024):
        d2 = sum((x[i0:i0 + 1024, None, k] - x[None, :, k]) ** 2 for k in range(3))
        i, j = torch.nonzero(d2 <= cut * cut, as_tuple=True)
        i = i + i0
        keep = i <= j
        out.append(torch.stack([i[keep], j[keep]]))
    out = torch.cat(out, 1)
    if room:
        out = torch.cat([out, out.new_zeros(2, max(0, room - out.shape[1]))], 1)[:, :room]
    return out.contiguous()


def _room(c):
    """Length of the pair list a program reads: the expected number of pairs
    and a quarter (the number itself depends on the catalogue)."""
    n = c["n"]
    return int(1.25 * 0.5 * n * n * _frac(c["side"], 3.0 * c["L0"])) + 2 * n


def _unit(l, b):
    return np.stack([np.cos(b) * np.cos(l), np.cos(b) * np.sin(l), np.sin(b)], -1)


def _queries(rng, c, n):
    return dict(l=rng.uniform(0, c["side"] * DEG, n), b=rng.uniform(0, c["side"] * DEG, n),
                s=np.exp(rng.uniform(math.log(S_LO), math.log(S_HI), n)))


def _fields(rng, c):
    """Fields as in the batched workload: uneven star counts (the case's),
    sides 1-3 degrees, outer scales 10-40 pc, 5 degrees apart in longitude."""
    out, r = [], np.random.default_rng([c["fields"], c["nmin"], c["nmax"]])
    for f in range(c["fields"]):
        n = int(round(math.exp(r.uniform(math.log(c["nmin"]), math.log(c["nmax"])))))
        side, L0 = rng.uniform(1.0, 3.0), rng.uniform(10.0, 40.0)
        out.append(dict(_catalogue(rng, n, side, L0, 5.0 * f, -side / 2), L0=L0))
    return out


def _sightlines(rng, c):
    """Predictive of the log-extinction along sightlines, 150-2800 pc: spread
    0.3, correlation falling with the ratio of the distances, means near
    ln(rho s) with the scatter that makes the walls matter."""
    n, m = c["sightlines"], c["points"]
    ls = np.log(np.geomspace(150.0, 2800.0, m) if m > 1 else np.array([150.0]))
    sd = rng.uniform(0.1, 0.4, (n, 1, 1))
    cov = sd ** 2 * np.exp(-np.abs(ls[:, None] - ls[None, :]) / 0.5) + 1e-4 * np.eye(m)
    mean = np.log(RHO) + ls + 0.15 * rng.standard_normal((n, m))
    return mean, cov


def _pic_setup(rng, c):
    cat = _catalogue(rng, c["n"], c["side"], c["L0"])
    A = np.maximum(cat["A"], 0.02)
    cat["a"], cat["asig"] = np.log(A), cat["sig"] / A
    g, w = c["grid"], c["side"] * DEG

    def block(l, b):
        return (np.minimum((g * l / w).astype(int), g - 1) * g
                + np.minimum((g * b / w).astype(int), g - 1)).astype(np.int32)

    R = c["inducing"]
    dirs = -(-R // 4)
    u = dict(l=np.repeat(rng.uniform(0, w, dirs), 4)[:R], b=np.repeat(rng.uniform(0, w, dirs), 4)[:R],
             s=np.tile([1000.0, 2000.0, 3000.0, 4000.0], dirs)[:R])
    q = _queries(rng, c, c["queries"])
    blk = block(cat["l"], cat["b"])
    blk[0] = g * g - 1
    return cat, blk, u, q, block(q["l"], q["b"])


def _mlp_setup(rng, n):
    """Weights of a 5-64-64-64-2 network at the scale training leaves them
    (ln K of order -3, log errors of order -5) and neighbour-pair geometry."""
    P = []
    for i, o in ((5, 64), (64, 64), (64, 64), (64, 2)):
        P.append((rng.standard_normal((i, o)) * math.sqrt(2.0 / i) * (0.3 if o == 2 else 1.0),
                  0.1 * rng.standard_normal(o)))
    P[3] = (P[3][0], np.array([-3.0, -5.0]))
    P = [(w.astype(np.float32), b.astype(np.float32)) for w, b in P]
    si = np.exp(rng.uniform(math.log(S_LO), math.log(S_HI), n))
    sj = np.clip(si + rng.uniform(-60.0, 60.0, n), 0.9 * S_LO, None)
    ch = np.minimum(rng.uniform(0.0, 60.0, n) / np.sqrt(si * sj), 0.3)
    return P, si, sj, ch


class _State:
    pass


def prepare(case, seed):
    c, rng, S = case, _rng(seed), _State()
    S.c, k = c, c["kind"]
    if k == "site":
        n = c["n"]
        s = np.exp(rng.uniform(math.log(S_LO), math.log(S_HI), n))
        sd = rng.uniform(0.05, 0.5, n)
        mu = np.log(RHO * s) + 0.3 * rng.standard_normal(n)
        A = np.exp(mu + sd * rng.standard_normal(n))
        obs = A + NOISE * rng.standard_normal(n) if c["lik"] == 0 else np.log(A)
        sig = np.full(n, NOISE) if c["lik"] == 0 else NOISE / A
        S.x = [_t(v) for v in (mu, sd ** 2, obs, sig)]
        S.tau0 = _t(0.5 * rng.uniform(0, 1, n) / sd ** 2)
        S.nu0 = S.tau0 * S.x[0]
        S.tau, S.nu = torch.empty_like(S.tau0), torch.empty_like(S.nu0)
        S.lib = gm.lib()
    elif k in ("ep", "posterior", "cov", "predict"):
        cat = _catalogue(rng, c["n"], c["side"], c["L0"])
        S.ctx = _context(c, cat)
        S.out = (torch.empty(c["n"], dtype=torch.float64, device=_dev()),
                 torch.empty(c["n"], dtype=torch.float64, device=_dev()))
        if k == "ep":
            S.zero = torch.zeros(c["n"], dtype=torch.float64, device=_dev())
        elif k == "cov":
            S.ij = _pairs(cat, 3.0 * c["L0"], _room(c))
            S.K = torch.empty(S.ij.shape[1], dtype=torch.float64, device=_dev())
            S.lib = gm.lib()
        else:
            S.ctx.build_cov()
            S.tau, S.nu = (_t(v) for v in _sites(cat))
            if k == "predict":
                S.ctx.set_sites(S.tau, S.nu)
                S.ctx.get_posterior(out=S.out)
                q = _queries(rng, c, c["queries"])
                S.q = [_t(q[v]) for v in ("l", "b", "s")]
                S.out = tuple(torch.empty(c["queries"], dtype=torch.float64, device=_dev())
                              for _ in range(2))
    elif k == "fields":
        F = _fields(rng, c)
        cat = {v: np.concatenate([f[v] for f in F]) for v in ("l", "b", "s", "A", "sig")}
        fid = np.repeat(np.arange(len(F)), [len(f["s"]) for f in F])
        L0 = np.array([f["L0"] for f in F])
        cfg = _config(dict(c, L0=20.0, prec="fp32"))
        S.ctx = gm.ep_init(cfg, *(_t(cat[v]) for v in ("l", "b", "s", "A", "sig")), field_id=fid,
                           field_L0=L0, field_cutoff=3.0 * L0)
        n = len(fid)
        S.zero = torch.zeros(n, dtype=torch.float64, device=_dev())
        S.out = tuple(torch.empty(n, dtype=torch.float64, device=_dev()) for _ in range(2))
    elif k == "sampler":
        mean, cov = _sightlines(rng, c)
        n, m, T = c["sightlines"], c["points"], c["steps"]
        S.mean, S.cov = _t(mean), _t(cov)
        S.mom = _t(rng.standard_normal((n, T, m)))
        S.samples = torch.empty((n, T - c["burn"], m), dtype=torch.float64, device=_dev())
        S.hits = torch.empty(n, dtype=torch.int64, device=_dev())
        one = _t(np.array([500.0]))
        S.ctx = gm.ep_init(gm.default_config(), 0 * one, 0 * one, one, 0 * one + 0.5, 0 * one + NOISE)
        S.lib = gm.lib()
    elif k == "pic":
        cat, S.blk, S.u, S.q, S.qblk = _pic_setup(rng, c)
        cfg = _config(c, likelihood=gm.LIK_GAUSS_IN_LNA)
        S.ctx = gm.ep_init(cfg, *(_t(cat[v]) for v in ("l", "b", "s", "a", "asig")))
        S.ctx.build_cov()
    else:
        P, si, sj, ch = _mlp_setup(rng, c["n"])
        one = _t(np.array([500.0]))
        S.ctx = gm.ep_init(gm.default_config(precision=gm.PREC_FP32), 0 * one, 0 * one, one,
                           0 * one + 0.5, 0 * one + NOISE)
        S.ctx.surrogate_set_params(np.concatenate([np.concatenate([w.ravel(), b]) for w, b in P]))
        S.x = [_t(v) for v in (si, sj, ch)]
    return S


# ---------------------------------------------------------------------- pass
def _graded(S, ts):
    """FP32 contexts compute in FP32: their results as FP32 values."""
    return [t.float() for t in ts] if S.c.get("prec", "fp32") == "fp32" else list(ts)


def run(S):
    c, k = S.c, S.c["kind"]
    if k == "site":
        S.tau.copy_(S.tau0)
        S.nu.copy_(S.nu0)
        delta, skipped = ctypes.c_double(), ctypes.c_int64()
        st = S.lib.gm_site_update_noalloc(
            c["n"], *(x.data_ptr() for x in S.x), S.tau.data_ptr(), S.nu.data_ptr(), c["lik"],
            c["damping"], 1e-8, torch.cuda.current_stream().cuda_stream, ctypes.byref(delta),
            ctypes.byref(skipped))
        if st != 0:
            raise RuntimeError("site update: status %d" % st)
        return [S.tau, S.nu, delta.value, skipped.value]
    if k in ("ep", "fields"):
        S.ctx.build_cov()
        S.ctx.set_sites(S.zero, S.zero)
        S.ctx.ep_sweep(c["sweeps"], 0.0)
        return _graded(S, S.ctx.get_posterior(out=S.out))
    if k == "posterior":
        S.ctx.set_sites(S.tau, S.nu)
        return _graded(S, S.ctx.get_posterior(out=S.out))
    if k == "cov":
        nnz = S.ctx.build_cov()
        st = S.lib.gm_get_entries(S.ctx._h, S.ij.shape[1], S.ij[0].data_ptr(), S.ij[1].data_ptr(),
                                  S.K.data_ptr())
        if st != 0:
            raise RuntimeError("entries: status %d" % st)
        return _graded(S, (S.K,) + tuple(S.ctx.get_prior(out=S.out))) + [nnz]
    if k == "predict":
        return _graded(S, S.ctx.predict(*S.q, out=S.out))
    if k == "sampler":
        st = S.lib.gm_monotone_sample(
            S.ctx._h, c["sightlines"], c["points"], S.mean.data_ptr(), S.cov.data_ptr(),
            S.mom.data_ptr(), c["burn"], c["steps"] - c["burn"], S.samples.data_ptr(),
            S.hits.data_ptr())
        if st != 0:
            raise RuntimeError("sampler: status %d" % st)
        return [S.samples, S.hits]
    if k == "pic":
        mean, cov = S.ctx.pic_posterior(S.blk, S.u["l"], S.u["b"], S.u["s"])
        qm, qv = S.ctx.pic_predict(S.qblk, S.q["l"], S.q["b"], S.q["s"])
        return [mean, cov, qm, qv]
    return list(S.ctx.surrogate_eval(*S.x, SIGMA2, 20.0))


# ---------------------------------------------------------------------- work
def _frac(side, cut, b0=0.0, n=1500):
    """Fraction of star pairs within the cutoff (a fixed small sample)."""
    r = np.random.default_rng(5)
    l, b = r.uniform(0, side * DEG, n), r.uniform(0, side * DEG, n)
    s = np.exp(r.uniform(math.log(S_LO), math.log(S_HI), n))
    x = _unit(l, b) * s[:, None]
    g = x @ x.T
    q = np.diag(g)
    return float(np.mean(q[:, None] + q[None, :] - 2 * g <= cut * cut))


def _evals(c):
    return 1200.0 if c.get("rule") == "band" else float(c["nodes"]) ** 2


def _colours(n, nnz):
    """Right-hand sides of probed variances at 2 x cutoff: about three times
    the neighbours of a star."""
    return min(n, 3.0 * nnz / n)


def work(case):
    """Bytes and operations of one pass: 13 per node pair of the quadrature,
    2 per stored entry, right-hand side and CG iteration of the solves (at 20
    iterations a refresh)."""
    c, k = case, case["kind"]
    if k == "site":
        return dict(bytes=8.0 * 8 * c["n"], flops=64.0 * 20 * c["n"])
    if k == "mlp":
        return dict(bytes=32.0 * c["n"], flops=2.0 * (5 * 64 + 2 * 64 * 64 + 128) * c["n"])
    if k == "sampler":
        n, m, T = c["sightlines"], c["points"], c["steps"]
        return dict(bytes=8.0 * n * m * (1 + m + 2 * T - c["burn"]), flops=1.0 * n * T * m * (m + 30))
    if k == "fields":
        n = (c["nmax"] - c["nmin"]) / math.log(c["nmax"] / c["nmin"])
        nnz = n * n * _frac(2.0, 75.0) + n
        one = 0.5 * nnz * 13.0 * c["nodes"] ** 2 + (c["sweeps"] + 1) * 40.0 * nnz * (
            _colours(n, nnz) if c["probe"] else n)
        return dict(bytes=c["fields"] * (8.0 * nnz + 7 * 8.0 * n), flops=c["fields"] * one)
    n = c["n"]
    nnz = n * n * _frac(c["side"], 3.0 * c["L0"]) + n
    val = 4.0 if c.get("prec") == "fp32" else 8.0
    quad = 0.5 * nnz * 13.0 * _evals(c)
    if k == "cov":
        return dict(bytes=(val + 4.0) * nnz + 8.0 * 7 * n, flops=quad)
    if k == "pic":
        nb, R = c["grid"] ** 2, c["inducing"]
        d = n / nb
        dense = nb * (d ** 3 / 3 + d * d * R + d * R * R) + 4.0 * R ** 3 + n * R * R
        pred = c["queries"] * (d * d + R * R) * 2.0
        return dict(bytes=8.0 * (nb * d * d + 2 * n * R + R * R + 8 * c["queries"]),
                    flops=2.0 * dense + pred)
    if k == "predict":
        q = c["queries"]
        kq = nnz / n * q
        return dict(bytes=(val + 4.0) * (nnz + kq) + 40.0 * q,
                    flops=kq * 13.0 * _evals(c) + 40.0 * nnz * q)
    R = _colours(n, nnz) if c["probe"] else n
    refresh = 40.0 * nnz * R
    times = c["sweeps"] + 1 if k == "ep" else 1
    return dict(bytes=(val + 4.0) * nnz + 8.0 * 9 * n,
                flops=times * refresh + (quad if k == "ep" else 0.0))


# --------------------------------------------------------------------- exact
_G = {}


def _phi(rho):
    """2^(2/3) / Gamma(1/3) rho^(1/3) K_(1/3)(rho), K by the trapezoid rule on
    int exp(-rho cosh t) cosh(t / 3) dt."""
    t = np.arange(0, 2000) * 0.05
    out = np.empty_like(rho)
    w = np.cosh(t / 3.0)
    w[0] = 0.5
    ct = np.cosh(t)
    for i0 in range(0, len(rho), 2048):
        r = rho[i0:i0 + 2048, None]
        with np.errstate(over="ignore", under="ignore"):
            out[i0:i0 + 2048] = (np.exp(-r * ct) * w).sum(1) * 0.05
    return 2.0 ** (2.0 / 3.0) / math.gamma(1.0 / 3.0) * np.cbrt(rho) * out


class _Kernel:
    """g(x) = expm1(sigma2 phi(sqrt x)) by degree-6 interpolation on 32
    segments per octave of x, 2^-96 .. 2^12 (0 beyond, held below)."""
    EMIN, EMAX, SEG, D = -96, 12, 32, 6

    def __init__(self):
        node = np.cos((np.arange(self.D + 1) + 0.5) * math.pi / (self.D + 1))
        e = np.arange(self.EMIN, self.EMAX)
        lo = np.ldexp(1.0, e)[:, None] * (1.0 + np.arange(self.SEG) / self.SEG)[None, :]
        h = np.ldexp(1.0 / self.SEG, e)[:, None] + 0 * lo
        x = lo[..., None] + h[..., None] * (node + 1.0) / 2.0
        y = np.expm1(SIGMA2 * _phi(np.sqrt(x).ravel())).reshape(-1, self.D + 1)
        V = np.vander(node, self.D + 1, increasing=True)
        self.c = _t(np.linalg.solve(V, y.T).T.copy())

    def __call__(self, x):
        n = self.c.shape[0]
        x = x.clamp_min(2.0 ** self.EMIN)
        bits = x.view(torch.int64)
        k = (bits >> 47) - ((1023 + self.EMIN) << 5)
        dead = k >= n
        k = k.clamp_max(n - 1)
        v = (bits & ((1 << 47) - 1)).double() * (2.0 ** -46) - 1.0
        c = self.c[k]
        p = c[..., self.D]
        for d in range(self.D - 1, -1, -1):
            p = p * v + c[..., d]
        return torch.where(dead, torch.zeros_like(p), p)


def _g():
    dev = torch.cuda.current_device()
    if dev not in _G:
        _G[dev] = _Kernel()
    return _G[dev]


def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return _t((x + 1) / 2), _t(w / 2)


def _side(D):
    """0, then breakpoints growing threefold from 1e-3, clipped at D (per pair)."""
    b = 1e-3 * (3.0 ** torch.arange(0, 13, device=D.device, dtype=torch.float64) - 1.0) / 2.0
    return torch.minimum(b[None, :], D[:, None])


def _band_R(A, B, c2):
    """R by composite rules in d = t - t', m = (t + t') / 2 (6 nodes a panel)."""
    z, w = _gl(6)
    g, K = _g(), 40.0
    Dp, Dn = A.clamp_max(K), B.clamp_max(K)
    kink = torch.minimum(torch.maximum(A - B, -Dn), Dp)
    bp = torch.cat([-_side(Dn), _side(Dp), kink[:, None]], 1).sort(1).values
    a, h = bp[:, :-1], bp[:, 1:] - bp[:, :-1]
    d = (a[..., None] + h[..., None] * z).flatten(1)
    wd = (h[..., None] * w).flatten(1)
    lo = d.abs() / 2
    hi = torch.minimum(A[:, None] - d / 2, B[:, None] + d / 2)
    c = c2.sqrt()[:, None]
    same = c2[:, None] <= 0
    sc = 1.0 / torch.where(same, torch.ones_like(c), c)
    end = torch.where(same, hi, torch.minimum(hi, lo + K * sc))
    dd = d * d * (1 - 0.25 * c2[:, None])
    tot = torch.zeros_like(d)
    ma, step = lo, 0.25 * sc
    for _ in range(6):
        mb = torch.minimum(ma + step, end)
        ln = (mb - ma).clamp_min(0.0)
        s = 0
        for j in range(6):
            m = ma + ln * z[j]
            s = s + w[j] * g(dd + m * m * c2[:, None])
        tot = tot + ln * s
        ma, step = torch.maximum(ma, mb), step * 3.0
    flat = (hi - lo).clamp_min(0.0) * g(d * d)
    return (wd * torch.where(same, flat, tot)).sum(1) / (A * B)


def _gl_R(A, B, c2, Q):
    z, w = _gl(Q)
    g = _g()
    tp = B[:, None] * z
    out = torch.zeros_like(A)
    for q in range(Q):
        t = (A * z[q])[:, None]
        out = out + w[q] * (g((t - tp) ** 2 + t * tp * c2[:, None]) * w).sum(1)
    return out


def _K(c, si, sj, c2, taper=True):
    """Covariance entries of pairs at distances si, sj and chord^2 c2."""
    L0, band = c["L0"], c.get("rule") == "band"
    R = torch.empty_like(si)
    step = 4000 if band else 60000
    for i0 in range(0, len(si), step):
        sl = slice(i0, i0 + step)
        A, B = si[sl] / L0, sj[sl] / L0
        R[sl] = _band_R(A, B, c2[sl]) if band else _gl_R(A, B, c2[sl], c["nodes"])
    K = torch.log1p(R)
    if taper:
        h = (((si - sj) ** 2 + si * sj * c2).sqrt() / (3.0 * L0)).clamp_max(1.0)
        K = K * (1 - h) ** 4 * (4 * h + 1)
    return K


def _geom(p):
    return _t(_unit(p["l"], p["b"])), _t(p["s"])


def _cross(c, p, q):
    """Dense tapered covariance between two point sets."""
    (up, sp), (uq, sq) = _geom(p), _geom(q)
    K = torch.zeros(len(sp), len(sq), dtype=torch.float64, device=_dev())
    for i0 in range(0, len(sp), 1024):
        u, s = up[i0:i0 + 1024], sp[i0:i0 + 1024]
        c2 = sum((u[:, None, k] - uq[None, :, k]) ** 2 for k in range(3))
        d2 = (s[:, None] - sq) ** 2 + s[:, None] * sq * c2
        i, j = torch.nonzero(d2 <= (3.0 * c["L0"]) ** 2, as_tuple=True)
        K[i0 + i, j] = _K(c, s[i], sq[j], c2[i, j])
    return K


def _star_K(c, cat):
    ij = _pairs(cat, 3.0 * c["L0"])
    u, s = _geom(cat)
    v = _K(c, s[ij[0]], s[ij[1]], ((u[ij[0]] - u[ij[1]]) ** 2).sum(1))
    K = torch.zeros(len(s), len(s), dtype=torch.float64, device=_dev())
    K[ij[0], ij[1]] = v
    K[ij[1], ij[0]] = v
    return K, torch.log(RHO * s) - 0.5 * K.diagonal()


def _solve(K, m, tau, nu):
    """Posterior mean, variances, B's factor, D and alpha for given sites."""
    d = tau.sqrt()
    L = torch.linalg.cholesky(torch.eye(len(m), dtype=K.dtype, device=K.device)
                              + d[:, None] * K * d[None, :])
    b = nu - tau * m
    alpha = b - d * torch.cholesky_solve((d * (K @ b))[:, None], L)[:, 0]
    V = torch.linalg.solve_triangular(L, d[:, None] * K, upper=False)
    return m + K @ alpha, K.diagonal() - (V * V).sum(0), L, d, alpha


def _site(mu, var, obs, sig, tau, nu, lik, damping=1.0, floor=1e-8):
    """Cavity, tilted moments (64-node rule at the mode), matched sites."""
    tc, nc = 1 / var - tau, mu / var - nu
    ok = tc > 0
    tc = torch.where(ok, tc, torch.ones_like(tc))
    mc, vc = nc / tc, (1 / tc).clamp_min(floor)
    s2 = sig * sig
    if lik == 1:
        vh = 1 / (1 / vc + 1 / s2)
        mh = vh * (mc / vc + obs / s2)
    else:
        def f(a):
            return -0.5 * (a - mc) ** 2 / vc - 0.5 * (obs - a.exp()) ** 2 / s2
        lo = obs.clamp_min(1e-300).log()
        pos = obs > 0
        vl = s2 / (obs * obs).clamp_min(1e-300)
        a = torch.where(pos, (mc / vc + lo / vl) / (1 / vc + 1 / vl), mc)
        for _ in range(60):
            e = a.exp()
            gr = -(a - mc) / vc + (obs - e) * e / s2
            H = -1 / vc + (obs * e - 2 * e * e) / s2
            st = torch.where(H < 0, -gr / H, gr * vc).clamp(-1, 1)
            for _ in range(8):
                st = torch.where(f(a + st) < f(a), st / 2, st)
            a = a + st
        e = a.exp()
        H = -1 / vc + (obs * e - 2 * e * e) / s2
        sh = torch.where(H < 0, (-H).clamp_min(1e-300).rsqrt(), vc.sqrt())
        x, w = (_t(v) for v in np.polynomial.hermite.hermgauss(64))
        y = math.sqrt(2.0) * sh[:, None] * x
        A = a[:, None] + y
        lt = (-0.5 * (A - mc[:, None]) ** 2 / vc[:, None]
              - 0.5 * (obs[:, None] - A.exp()) ** 2 / s2[:, None])
        W = (torch.log(w) + x * x + lt - f(a)[:, None]).exp()
        S0 = W.sum(1)
        m1 = (W * y).sum(1) / S0
        mh, vh = a + m1, (W * y * y).sum(1) / S0 - m1 * m1
    tn, nn = 1 / vh - 1 / vc, mh / vh - mc / vc
    ok = ok & (tn >= 0)
    return (torch.where(ok, tau + damping * (tn - tau), tau),
            torch.where(ok, nu + damping * (nn - nu), nu), ok)


def _ep(c, cat):
    K, m = _star_K(c, cat)
    obs, sig = _t(cat["A"]), _t(cat["sig"])
    tau, nu = torch.zeros_like(m), torch.zeros_like(m)
    for _ in range(c["sweeps"]):
        mu, var = _solve(K, m, tau, nu)[:2]
        tau, nu, _ = _site(mu, var, obs, sig, tau, nu, 0)
    return list(_solve(K, m, tau, nu)[:2])


def _mlp(P, si, sj, ch):
    r = np.sqrt(si * sj) / 20.0
    h = _t(np.stack([np.log(r) / 4, np.abs(si - sj) / 60.0, ch * r / 3, 0 * r + SIGMA2, 0 * r], 1))
    for i, (w, b) in enumerate(P):
        h = h @ _t(w) + _t(b)
        if i < 3:
            h = h * torch.sigmoid(h)
    return [h[:, 0].contiguous(), h[:, 1].contiguous()]


def _pic(c, rng):
    cat, blk, u, q, qblk = _pic_setup(rng, c)
    K, m = _star_K(c, cat)
    Kuu = _cross(c, u, u)
    Kau = _cross(c, cat, u)
    us = _t(u["s"])
    mu_u = torch.log(RHO * us) - 0.5 * Kuu.diagonal()
    iK = torch.linalg.inv(Kuu)
    A = Kau @ iK
    a, s2 = _t(cat["a"]), _t(cat["asig"]) ** 2
    P, h, inv = iK.clone(), iK @ mu_u, {}
    for k in range(c["grid"] ** 2):
        i = torch.as_tensor(np.nonzero(blk == k)[0], device=_dev())
        if len(i) == 0:
            continue
        C = K[i][:, i] - A[i] @ Kau[i].T + torch.diag(s2[i])
        L = torch.linalg.cholesky(C)
        P = P + A[i].T @ torch.cholesky_solve(A[i], L)
        h = h + A[i].T @ torch.cholesky_solve((a[i] - m[i] + A[i] @ mu_u)[:, None], L)[:, 0]
        inv[k] = (i, L)
    cov = torch.linalg.inv(P)
    mean = cov @ h
    Kqu, Kqa = _cross(c, q, u), _cross(c, q, cat)
    qs = _t(q["s"])
    kss = _K(c, qs, qs, 0 * qs)
    As = Kqu @ iK
    qm = torch.log(RHO * qs) - 0.5 * kss + As @ (mean - mu_u)
    qv = kss - (As * Kqu).sum(1) + ((As @ cov) * As).sum(1)
    for k, (i, L) in inv.items():
        j = torch.as_tensor(np.nonzero(qblk == k)[0], device=_dev())
        if len(j) == 0:
            continue
        D = Kqa[j][:, i].T - Kau[i] @ As[j].T
        G = torch.cholesky_solve(D, L)
        Lr = As[j] - G.T @ A[i]
        m0 = torch.log(RHO * qs[j]) - 0.5 * kss[j]
        qm[j] = m0 + G.T @ (a[i] - m[i]) + Lr @ (mean - mu_u)
        qv[j] = kss[j] - (As[j] * Kqu[j]).sum(1) - (G * D).sum(0) + ((Lr @ cov) * Lr).sum(1)
    return [mean, cov, qm, qv]


def exact(case, seed):
    c, rng, k = case, _rng(seed), case["kind"]
    if k == "site":
        S = prepare(c, seed)
        mu, var, obs, sig = S.x
        tau, nu, ok = _site(mu, var, obs, sig, S.tau0, S.nu0, c["lik"], c["damping"])
        dl = torch.maximum((tau - S.tau0).abs() / (1 + S.tau0.abs()),
                           (nu - S.nu0).abs() / (1 + S.nu0.abs()))
        return [tau, nu, float(dl.max()), int((~ok).sum())]
    if k == "mlp":
        return _mlp(*_mlp_setup(rng, c["n"]))
    if k == "sampler":
        return None  # a chain of reflections: step by step on the host it would take minutes
    if k == "fields":
        parts = [_ep(dict(c, L0=f["L0"]), f) for f in _fields(rng, c)]
        return [torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])]
    n = c["n"]
    pairs = 0.5 * n * n * _frac(c["side"], 3.0 * c["L0"])
    if pairs * (8000.0 if c.get("rule") == "band" else c["nodes"] ** 2) > 1.6e10 or n > 9000:
        return None  # too long in FP64 with torch
    if k == "pic":
        return _pic(c, rng)
    cat = _catalogue(rng, n, c["side"], c["L0"])
    if k == "cov":
        K, m = _star_K(c, cat)
        ij = _pairs(cat, 3.0 * c["L0"], _room(c))
        return [K[ij[0], ij[1]], m, K.diagonal().clone(), None]
    if k == "ep":
        return _ep(c, cat)
    K, m = _star_K(c, cat)
    tau, nu = (_t(v) for v in _sites(cat))
    mu, var, L, d, alpha = _solve(K, m, tau, nu)
    if k == "posterior":
        return [mu, var]
    q = _queries(rng, c, c["queries"])
    qs = _t(q["s"])
    kss = _K(c, qs, qs, 0 * qs)
    Kq = _cross(c, q, cat)
    V = torch.linalg.solve_triangular(L, d[:, None] * Kq.T, upper=False)
    return [torch.log(RHO * qs) - 0.5 * kss + Kq @ alpha, kss - (V * V).sum(0)]
