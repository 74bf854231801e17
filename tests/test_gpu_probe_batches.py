"""The probing colouring in batches of 32 stars: valid and greedy (every star holds
the smallest colour that no star closer than D holds among smaller ones) at counts
around the batch and beyond it, with duplicated stars and separations at the edge
of the single-precision test."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 300, 1500])
def test_batched_colouring_is_greedy(n):
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    s = np.round(rng.uniform(500.0, 618.0, n), 1)      # many pairs at exact differences
    l, b = rng.uniform(0, 0.002, n), rng.uniform(0, 0.002, n)
    if n > 40:
        l[5:20], b[5:20] = l[25:40], b[25:40]
        s[5:12] = s[25:32]
        s[12:20] = s[32:40] + 60.0                       # D apart
    D = 60.0
    cfg = gm.default_config(outer_scale_pc=20.0, cutoff_pc=30.0, probe_factor=2.0,
                            precision=gm.PREC_FP32, quad_rule=gm.QUAD_GL, n_nodes=8)
    with gm.ep_init(cfg, l, b, s, np.ones(n), np.full(n, 0.1)) as ctx:
        ctx.build_cov()
        got = ctx.get_probe_colours()
    u = O.unit_vectors(l, b)
    d2 = (s[:, None] - s[None, :]) ** 2 + s[:, None] * s[None, :] * (
        (u[:, None] - u[None, :]) ** 2).sum(-1)
    near = d2 < D * D
    np.fill_diagonal(near, False)
    for i in range(n):
        held = set(got[near[i]])
        assert got[i] not in held                        # valid
        assert set(range(got[i])) <= held                # smallest free: greedy
