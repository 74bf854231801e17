"""The way out of a bounded device wait that runs out (GM_WAIT_EXPIRES makes one
thread group take a completed wait for an expired one): the call ends with
GM_E_TIMEOUT whatever the other groups of the block are doing, again and again, and
the context stays usable."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu
TIMEOUT = 7


@pytest.mark.parametrize("n", [100, 128 * 152 * 4 + 5, 400003])
def test_surrogate_groups_leave_together(n, monkeypatch):
    import paper_1708_09705_gb300 as gm
    rng = np.random.default_rng(n)
    flat = np.concatenate([np.concatenate([W.ravel(), b])
                           for W, b in M.init_params(3)]).astype(np.float32)
    si = np.exp(rng.uniform(np.log(60.0), np.log(5000.0), n))
    sj, ch = si + 10.0, rng.uniform(0, 0.01, n)
    one = np.array([500.0])
    with gm.ep_init(gm.default_config(precision=gm.PREC_FP32), 0 * one, 0 * one, one, 0 * one + 0.5,
                    0 * one + 0.05) as ctx:
        ctx.surrogate_set_params(flat)
        y, e = ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
        for _ in range(20):
            monkeypatch.setenv("GM_WAIT_EXPIRES", "surrogate")
            with pytest.raises(gm.GmError) as err:
                ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
            assert err.value.status == TIMEOUT
            monkeypatch.delenv("GM_WAIT_EXPIRES")
        y2, e2 = ctx.surrogate_eval(si, sj, ch, 1.3, 17.0)
    np.testing.assert_array_equal(y, y2)
    np.testing.assert_array_equal(e, e2)
