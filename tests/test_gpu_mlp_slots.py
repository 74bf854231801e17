"""Surrogate inference over its tile schedule: one tile, ragged tiles, the first
tile of a block's second group (152 blocks of 4 groups), more tiles than groups;
host and device arrays give the same values, and both the network's FP64 output
within the two-piece BF16 products' error (2^-15 of the largest layer output)."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 129, 128 * 152 + 1, 128 * 152 * 4 + 5, 200003])
def test_forward_schedule(n):
    import torch
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    params = M.init_params(3)
    flat = np.concatenate([np.concatenate([W.ravel(), b]) for W, b in params]).astype(np.float32)
    si = np.exp(rng.uniform(np.log(60.0), np.log(5000.0), n))
    sj = np.clip(si + rng.uniform(-60, 60, n), 30.0, None)
    ch = rng.uniform(0, 60.0, n) / np.sqrt(si * sj)
    one = np.array([500.0])
    with gm.ep_init(gm.default_config(precision=gm.PREC_FP32), 0 * one, 0 * one, one, 0 * one + 0.5,
                    0 * one + 0.05) as ctx:
        ctx.surrogate_set_params(flat)
        y, e = ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
        yd, ed = ctx.surrogate_eval(*(torch.tensor(v, device="cuda") for v in (si, sj, ch)), 1.3, 17.0)
    np.testing.assert_array_equal(y, yd)
    np.testing.assert_array_equal(e, ed)
    p32 = [(W.astype(np.float32).astype(float), b.astype(np.float32).astype(float)) for W, b in params]
    out, cache = M.forward(p32, M.features(si, sj, ch, 1.3, 17.0))
    scale = max(float(np.abs(out).max()), 1.0)
    assert np.abs(y - out[:, 0]).max() < 4 * scale * 2.0 ** -15
    assert np.abs(e - out[:, 1]).max() < 4 * scale * 2.0 ** -15
