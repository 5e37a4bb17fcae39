"""Training steps at the edges of the training kernel's split (32 points a
warp, 448 a block, more points than the resident blocks take at once) and for
every width, against the same steps in fp64.  Tolerance: a parameter moves by
at most lr = 0.01 per Adam step, and a gradient entry that is off by a share of
itself moves the step by that share at most; two percent of lr per step, as for
a single step in test_gpu_learn.py."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")

STEPS, LR = 3, 0.01


@pytest.mark.parametrize("H", [1, 8, 16, 32])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 447, 448, 449, 5000, 70_001, 300_000])
def test_steps_match_fp64(H, m):
    rng = np.random.default_rng(100 * H + m)
    x = np.sort(rng.random(m)).astype(np.float32)
    t = ((np.arange(m) + 0.5) / m).astype(np.float32)
    theta = rng.normal(size=3 * H + 1).astype(np.float32)
    c = vx.vx_open(64 << 20)
    try:
        got, _ = vx.vx_mlp_train(c, theta, H, x, t, STEPS, LR)
        again, _ = vx.vx_mlp_train(c, theta, H, x, t, STEPS, LR)
    finally:
        vx.vx_close(c)
    assert np.array_equal(got, again)  # sums are taken in a fixed order
    th = theta.astype(np.float64)
    m1, m2 = np.zeros_like(th), np.zeros_like(th)
    for k in range(1, STEPS + 1):
        _, g = O.mlp_loss_grad(th, H, x.astype(np.float64), t.astype(np.float64))
        O.adam_step(th, g, m1, m2, k, lr=LR)
    assert np.abs(got - th).max() <= 0.02 * LR * STEPS
