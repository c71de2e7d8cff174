"""The warp-per-sample inference kernels (lb_mlp_forward, lb_mlp_invert_kappa) at the edges
of their launch rule: one sample, as many as there are resident warps (two CTAs of four warps
per SM), one more (two samples per warp, the last group ragged) and several rounds of the
grid. Predictions against the FP64 oracle within 2e-4 (64-term FP32 sums, FP32 erf and exp:
about 1e-6, times the output scale); a sample's bits do not depend on the batch it is in."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1306_6445_gb300 import inputs as I
from test_gpu_mlp import lbm, monotone_params  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def counts():
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    warps = sms * 8
    return [1, 3, warps, warps + 1, 2 * warps + 3, 5 * warps + 1]


@pytest.mark.parametrize("which", range(6))
def test_predictions_and_inversions_at_the_edges_of_the_grid(lbm, which):  # noqa: F811
    n = counts()[which]
    x, y = I.mlp_random_data(200, seed=51)
    theta = monotone_params(52)
    norm = M.normalisation(x.astype(np.float64), y.astype(np.float64))
    net = lbm.MLP(200)
    net.set_params(theta)
    net.set_data(x, y)
    q = I.mlp_random_data(n, seed=53)[0]
    got = net.forward(q)
    ref = M.forward(theta.astype(np.float64), q.astype(np.float64), norm)[0]
    assert np.max(np.abs(got / ref - 1)) < 2e-4
    goal = q.copy()
    goal[:, 1] = np.clip(goal[:, 1], 0.05, 0.9)
    sigma = M.forward(theta.astype(np.float64), goal.astype(np.float64), norm)[0][:, 0]
    queries = np.stack([goal[:, 0], goal[:, 2], sigma], axis=1)
    queries[n // 2, 2] *= 1e3 if n > 1 else 1.0     # above the bracket: NaN, its neighbours not
    kappa = net.invert_kappa(queries, 0.0, 0.95)
    inside = np.ones(n, dtype=bool)
    inside[n // 2] = n == 1
    assert np.array_equal(np.isnan(kappa), ~inside)
    # sigma falls by a factor e^-1..e^-2 over the bracket: 2e-4 of sigma moves kappa by < 1e-3
    assert np.max(np.abs(kappa - goal[:, 1])[inside]) < 1e-3
    one = net.forward(q[-1:])
    assert np.array_equal(one[0], got[-1])
    net.close()
