"""FP64 entries of the Q-node rule for stars at nearly equal distances, where the
separation of two nodes is a small difference of large numbers and the kernel has a
cusp: against an FP64 evaluation from the same cubic table (so that the table's own
error, 2e-12 of g(0), cancels) with the separations of equal nodes taken from the
difference of the distances.  Float pairs carry 2^-47 a term and the table's third and
fourth coefficients 1e-13 of g: rtol 1e-12."""
import numpy as np
import pytest
from scipy.special import gamma, kv

pytestmark = pytest.mark.gpu
M, EMIN, EMAX = 7, -100, 11


def _phi(x):
    r = np.sqrt(x)
    return 2 ** (2 / 3) / gamma(1 / 3) * np.cbrt(r) * kv(1 / 3, r)


def table_g(x, sigma2):
    """The cubic through four equispaced values of g on each segment of x."""
    x = np.maximum(x, 2.0 ** EMIN)
    m, e = np.frexp(x)
    lo = np.ldexp(np.floor(np.ldexp(2 * m - 1, M)) * 2.0 ** -M + 1, e - 1)
    H = np.ldexp(2.0 ** -M, e - 1)
    v = [np.expm1(sigma2 * _phi(lo + H * q / 3)) for q in range(4)]
    d1, d2, d3 = v[1] - v[0], v[2] - 2 * v[1] + v[0], v[3] - 3 * v[2] + 3 * v[1] - v[0]
    w = 3 * (x - lo) / H
    g = v[0] + w * ((d1 - .5 * d2 + d3 / 3) + w * ((.5 * d2 - .5 * d3) + w * d3 / 6))
    return np.where(x < 2.0 ** EMAX, g, 0.0)


def rule(A, B, c2, Q, sigma2):
    z, w = np.polynomial.legendre.leggauss(Q)
    z, w = (z + 1) / 2, w / 2
    d = A * z[:, None] - B * z[None, :]
    np.fill_diagonal(d, (A - B) * z)
    x = d * d + A * B * c2 * z[:, None] * z[None, :]
    return np.log1p(w @ table_g(x, sigma2) @ w)


@pytest.mark.parametrize("Q", [5, 32, 64, 100])
def test_nearly_equal_distances(Q):
    import oracle as O
    import paper_1708_09705_gb300 as gm
    L0, rng = 10.0, np.random.default_rng(Q)
    # stars 1e-12 .. 1e-4 of the distance behind the first, in its direction and
    # (the last eight) 0.1 degrees away
    gap = np.r_[0.0, 10.0 ** np.linspace(-12, -4, 25) * rng.uniform(1, 3, 25), 3e-9 * np.arange(8)]
    s = 2900.0 * (1 + gap)
    l = np.full(len(s), 0.02)
    l[-8:] += 0.1 * np.pi / 180
    b = np.full(len(s), 0.01)
    cfg = gm.default_config(sigma2=1.0, outer_scale_pc=L0, cutoff_pc=30.0, n_nodes=Q,
                            quad_rule=gm.QUAD_GL, precision=gm.PREC_FP64, taper=1)
    one = np.ones(len(s))
    i, j = np.triu_indices(len(s), 1)
    with gm.ep_init(cfg, l, b, s, one, 0.1 * one) as ctx:
        ctx.build_cov()
        got = ctx.get_entries(i, j)
    u = O.unit_vectors(l, b)
    A = s * (1.0 / L0)
    ref = np.array([rule(A[p], A[q], ((u[p] - u[q]) ** 2).sum(), Q, 1.0) for p, q in zip(i, j)])
    np.testing.assert_allclose(got, ref, rtol=1e-12)
