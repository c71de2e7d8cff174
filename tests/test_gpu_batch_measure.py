"""The chunked Laplace measurement of a batch (lb_batch_measure) at the edges of its chunks
(whole rows, about 8192 sites): one chunk, exactly one, one row more, many, a lattice of three
columns; masks whose radius falls on a site's distance. Densities and mass against host sums of
the same density field, pressures against lb_measure_droplet of the same state (FP64 sums in
another order: 1e-12 relative)."""
import numpy as np
import pytest

from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import case_params, lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(3, 40), (64, 64), (128, 64), (91, 90), (91, 91), (301, 257), (40, 700)]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["cs", "exp", "piecewise"])
def test_chunked_measurement(lbm, prec, kind):  # noqa: F811
    eos, G, (lo, hi) = case_params(lbm, kind)
    rates = lbm.RateParams.from_viscosity(0.1)
    b = lbm.Batch([lbm.LatticeDesc(nx, ny, eos, G, kappa=0.3, rates=rates) for nx, ny in SIZES],
                  prec=prec)
    rhos = [I.smooth_random_density(np.random.default_rng(nx + ny), nx, ny, lo, hi) for nx, ny in SIZES]
    for i, r in enumerate(rhos):
        b.set_rho_u(i, r)
    b.step(3)
    # radii 2 d with d the distance of a site: r < radius / 2 excludes that site exactly
    radii = np.array([2.0 * np.hypot(0.5 * ((nx + 1) % 2) + 1, 0.5 * ((ny + 1) % 2) + 1) for nx, ny in SIZES])
    radii[-1] = 7.3
    m = b.measure(radii)
    for i, (nx, ny) in enumerate(SIZES):
        rho = b.rho(i)
        y, x = np.mgrid[0:ny, 0:nx]
        r = np.sqrt((x - 0.5 * (nx - 1)) ** 2 + (y - 0.5 * (ny - 1)) ** 2)
        inside, outside = r < 0.5 * radii[i], r > radii[i] + 0.3 * 0.5 * min(nx, ny)
        assert m[i, 6] == pytest.approx(rho.sum(), rel=1e-12)
        assert m[i, 1] == pytest.approx(rho[inside].mean(), rel=1e-12)
        if outside.any():
            assert m[i, 2] == pytest.approx(rho[outside].mean(), rel=1e-12)
        lat = lbm.Lattice(nx, ny, eos, G, kappa=0.3, rates=rates, prec=prec)
        lat.set_populations(b.populations(i))
        one = lat.measure_droplet(float(radii[i]))
        lat.close()
        assert m[i, 4] == pytest.approx(one["p_in"], rel=1e-10, abs=1e-12 * hi)
        if outside.any():
            assert m[i, 5] == pytest.approx(one["p_out"], rel=1e-10, abs=1e-12 * hi)
            # (an interior mask close to the outside one: R and theta of the mass are checked as NaN too)
            assert np.isnan(m[i, 0]) == np.isnan(one["theta"])
        else:
            assert np.isnan(m[i, 2]) and m[i, 7] == 1.0
    assert np.array_equal(m, b.measure(radii), equal_nan=True)
    b.close()
