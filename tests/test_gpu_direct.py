"""The direct step kernels (launch variant 7: one CTA per 64-column tile in FP32 and BF16, a psi
and a collision pass in FP64; variant 8: pipelined tiles) give the bits of the ring kernels
(variant 4) at the edges of their tiles: lattices narrower than a tile, one column short of, exactly and one or two beyond
it, and rows around the tile height, for every boundary, EOS and storage type."""
import numpy as np
import pytest

from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import case_params, lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(3, 3), (5, 4), (63, 5), (64, 8), (65, 7), (66, 3), (127, 12), (128, 9), (130, 17), (257, 4), (66, 21), (70, 22), (192, 19), (700, 401)]


@pytest.mark.parametrize("prec", ["fp32", "fp64", "bf16", "bf16-stochastic"])
@pytest.mark.parametrize("bc", ["periodic", "walls", "open"])
@pytest.mark.parametrize("kind", ["cs", "exp", "piecewise"])
def test_direct_kernels_give_the_ring_kernels_bits(lbm, prec, bc, kind):  # noqa: F811
    if prec.startswith("bf16") and bc == "open":
        pytest.skip("open boundaries are not compiled for BF16 storage")
    eos, G, (lo, hi) = case_params(lbm, kind)
    kw = {"walls_y": bc == "walls", "open_bc": bc == "open"}
    if bc == "open":
        kw["viscosity_switch"] = (0.5 * (lo + hi), 1.1)
    if prec.startswith("bf16"):
        kw.update(storage_shift=0.5 * (lo + hi), stochastic_rounding=prec != "bf16")
    for nx, ny in SIZES:
        rng = np.random.default_rng(nx * 100 + ny)
        rho = I.smooth_random_density(rng, nx, ny, lo, hi)
        ux, uy = I.random_velocity(rng, rho.shape, 1e-3)
        outs = []
        for variant in (4, 7) if prec == "fp64" else (4, 7, 8):
            lat = lbm.Lattice(nx, ny, eos, G, kappa=0.4, sigma_force=0.05,
                              rates=lbm.RateParams.from_viscosity(0.1), prec=prec.split("-")[0], **kw)
            lbm.lb_set_launch(lat.ctx, variant, 0)
            assert lbm.lb_get_launch(lat.ctx)["variant"] == variant
            lat.set_rho_u(rho, ux, uy)
            lat.step(3)
            outs.append(lat.populations())
            lat.close()
        for o in outs[1:]:
            assert np.array_equal(o, outs[0]), (nx, ny)
