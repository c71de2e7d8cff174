"""max |v| of lb_reduce where |v|^2 is a subnormal FP32 number: FP32 must not rule the larger of two
such speeds out. Every thread meets |v|^2 = 2.6 units of the smallest FP32 number first, 1.4 + 1.4 of
them later (which FP32 rounds to 2, below the 3 of the first)."""
import numpy as np
import pytest

from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_max_speed_of_subnormal_squares(lbm):  # noqa: F811
    nx = ny = 400
    unit = 2.0 ** -149
    f = np.zeros((9, ny, nx))
    f[0] = 1.0                                   # uniform density and potential: v = j
    f[1, :ny // 2] = np.sqrt(2.6 * unit)
    f[1, ny // 2:] = f[2, ny // 2:] = np.sqrt(1.4 * unit)
    lat = lbm.Lattice(nx, ny, lbm.EOSParams(kind="exp"), -40.0, prec="fp64")
    lat.set_populations(f)
    # the squares, their sum and the root are FP64 operations of half an ulp each
    assert lat.reduce()[3] == pytest.approx(np.sqrt(2.8 * unit), rel=1e-15, abs=0)
    lat.close()
