"""The size of the training kernel's gradients.  Adam's first step moves a
parameter by lr g / (|g| + 1e-8), which shows no more than g's sign unless |g| is
near 1e-8, so here it is: output weights (softplus(alpha)) and targets are small
enough that the units' gradients ("units") or the offset's ("offset") are of that
size.  Every point's error has the same sign, so that nothing cancels, and the
last 32 points carry as much of the gradient as all others together: a dropped
point of the ragged tail shows, and so do dropped blocks and sweeps.

Tolerance: a gradient is a sum of positive terms, each right to a few roundings,
in at most 160 + 60 roundings of the longest chain of additions: 2e-5 of itself,
hence 5e-6 lr of the step (g / (g + eps) falls by at most a quarter of what g
does); bias corrections in fp32 add 1e-5.  1e-4 lr per step, and four roundings
of a parameter of up to 16 (4e-6)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")


def _points(which, H, m):
    """theta, x, t as the call takes them."""
    rng = np.random.default_rng(10 * m + H)
    small = 11.0 if which == "units" else 18.5
    theta = np.concatenate([rng.uniform(-1, 3, H), rng.uniform(-1.5, 1.5, H), -small + rng.uniform(-0.5, 0.5, H),
                            [0.0]]).astype(np.float32)
    x = np.sort(rng.random(m)).astype(np.float32)
    t = -(0.5 + rng.random(m)) * (6e-4 if which == "units" else 3e-9)
    t[-32:] *= max(1.0, m / 32)
    return theta, x, t.astype(np.float32)


def _fp64(theta, H, x, t, steps, lr):
    th = theta.astype(np.float64)
    m1, m2 = np.zeros_like(th), np.zeros_like(th)
    for k in range(1, steps + 1):
        _, g = O.mlp_loss_grad(th, H, x, t)
        O.adam_step(th, g, m1, m2, k, lr=lr)
    return th


@pytest.mark.parametrize("which", ["units", "offset"])
@pytest.mark.parametrize("H", [1, 8, 16, 32])
@pytest.mark.parametrize("m", [1, 31, 33, 447, 449, 5000, 65_537, 70_001, 300_000])
def test_step_sizes_match_fp64(which, H, m):
    theta, x, t = _points(which, H, m)
    c = vx.vx_open(64 << 20)
    try:
        for steps, lr in ((1, 1.0), (3, 0.1)):
            got, _ = vx.vx_mlp_train(c, theta, H, x, t, steps, lr)
            want = _fp64(theta, H, x, t, steps, lr)
            assert np.abs(got - want).max() <= 1e-4 * lr * steps + 4e-6
    finally:
        vx.vx_close(c)
