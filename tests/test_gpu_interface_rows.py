"""lb_interface_height at every row that an interface can lie at in lattices whose rows are no multiple
of the scan's segments (64 rows) or of the rows that it loads at a time: the lowest row below rho_mid,
interpolated, as numpy finds it in the same densities."""
import numpy as np
import pytest

from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bc", ["walls", "open"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ny", [3, 4, 5, 61, 64, 66, 131])
def test_first_row_below(lbm, prec, ny, bc):  # noqa: F811
    nx = ny + 3                                  # column x: liquid below row x; columns of one phase
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    rho = np.where(y < x, 400.0, 150.0) + np.random.default_rng(ny).uniform(-20, 20, (ny, nx))
    lat = lbm.Lattice(nx, ny, lbm.EOSParams(kind="exp"), -40.0, prec=prec, walls_y=bc == "walls",
                      open_bc=bc == "open")
    lat.set_rho_u(rho)
    got, rho = lat.interface_height(275.0), lat.rho()
    lat.close()
    first = np.where((rho < 275.0).any(axis=0), (rho < 275.0).argmax(axis=0), -1)
    for c in range(nx):
        if first[c] <= 0:
            assert np.isnan(got[c])
        else:
            a, b = rho[first[c] - 1, c], rho[first[c], c]
            assert got[c] == pytest.approx(first[c] - 1 + (a - 275.0) / (a - b), rel=1e-14)
