"""Values that are not finite in a training call: every parameter that the same
step in fp64 makes NaN is NaN, and no other."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")


@pytest.mark.parametrize("where", ["none", "x", "t", "omega", "beta", "alpha", "gamma", "x_inf", "t_inf"])
@pytest.mark.parametrize("H,m", [(1, 1), (8, 33), (32, 5000)])
def test_nan_reaches_the_parameters_that_it_reaches_in_fp64(where, H, m):
    rng = np.random.default_rng(m)
    x, t = np.sort(rng.random(m)).astype(np.float32), rng.random(m).astype(np.float32)
    theta = rng.normal(size=3 * H + 1).astype(np.float32)
    at = {"omega": 0, "beta": H, "alpha": 2 * H, "gamma": 3 * H}
    if where in at:
        theta[at[where]] = np.nan
    elif where != "none":
        a = x if where[0] == "x" else t
        a[m // 2] = np.inf if where.endswith("inf") else np.nan
    c = vx.vx_open(64 << 20)
    try:
        got, _ = vx.vx_mlp_train(c, theta, H, x, t, 1, 0.01)
    finally:
        vx.vx_close(c)
    th = theta.astype(np.float64)
    m1, m2 = np.zeros_like(th), np.zeros_like(th)
    with np.errstate(all="ignore"):
        _, g = O.mlp_loss_grad(th, H, x, t)
        O.adam_step(th, g, m1, m2, 1)
    assert np.array_equal(np.isnan(got), np.isnan(th))
