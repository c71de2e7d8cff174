"""The training kernels at the edges of how a tile of 16 samples is split (over four CTAs while
there are at most 76 tiles, beyond not): ragged tiles, the last count that is split, the first
that is not, more tiles than CTAs; and the running powers of beta1, beta2 behind the bias correction
over calls with other betas. Gradients within 1e-4 of the largest entry and losses within 1e-4
(FP32 sums of up to 5000 samples, about 1e-6, and FP32 erf / exp)."""
import numpy as np
import pytest

from oracle import mlp as M
from test_gpu_mlp import lbm, net_with  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2, 5, 1215, 1216, 1217, 4865])
def test_gradient_at_the_edges_of_the_tile_rule(lbm, n):  # noqa: F811
    net, theta, x, y = net_with(lbm, n, seed=60 + n)
    loss, g = net.loss_grad()
    lref, gref = M.loss_and_grad(theta.astype(np.float64), x, y, M.normalisation(x, y), bf16=True)
    assert loss == pytest.approx(lref, rel=1e-4)
    assert np.max(np.abs(g - gref)) <= 1e-4 * np.max(np.abs(gref))
    net.close()


def test_bias_correction_over_calls_with_other_betas(lbm):  # noqa: F811
    n, lr = 300, 1e-3
    net, theta, x, y = net_with(lbm, n, seed=71)
    norm = M.normalisation(x, y)
    th, m, v = theta.astype(np.float64), 0.0, 0.0
    step = 0
    for count, b1, b2 in ((3, 0.9, 0.999), (52, 0.8, 0.99), (2, 0.9, 0.999)):
        net.train(count, lr, b1, b2)
        for _ in range(count):
            step += 1
            _, g = M.loss_and_grad(th, x, y, norm, bf16=True)
            th, m, v = M.adam_step(th, m, v, g, step, lr, b1, b2)
            th = th.astype(np.float32).astype(np.float64)
    d = np.abs(net.params() - th)
    # a wrong power of beta in one of the 57 steps moves every entry by far more than this
    assert np.median(d) < 1e-2 * lr and np.mean(d <= 0.2 * lr) > 0.99
    assert net.steps_done == 57
    net.close()
