"""Several steps of a small FP32 lattice in one launch (the cluster kernel, taken by contexts with
launch variant 7) give the bits of single steps with the staged tiles (variant 8), at the edges of
what the kernel takes: one row per CTA, uneven rows, four columns, two pairs per thread, the
largest lattice; for both boundary kinds and every EOS. The state it writes back (with its ghost
columns) carries on in the other kernels, and the step count and domain errors are those of single
steps."""
import numpy as np
import pytest

from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import case_params, lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(4, 16), (6, 31), (64, 64), (66, 17), (100, 100), (1024, 16), (62, 130), (128, 128), (128, 129), (180, 180)]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("kind", ["cs", "exp", "piecewise"])
def test_many_steps_in_one_launch(lbm, walls, kind):  # noqa: F811
    eos, G, (lo, hi) = case_params(lbm, kind)
    for nx, ny in SIZES:
        rng = np.random.default_rng(nx * 100 + ny)
        rho = I.smooth_random_density(rng, nx, ny, lo, hi)
        ux, uy = I.random_velocity(rng, rho.shape, 1e-3)
        states = []
        for variant in (7, 8):
            lat = lbm.Lattice(nx, ny, eos, G, kappa=0.4, sigma_force=0.05, prec="fp32", walls_y=walls,
                              rates=lbm.RateParams.from_viscosity(0.1))
            lbm.lb_set_launch(lat.ctx, variant, 0)
            lat.set_rho_u(rho, ux, uy)
            out = []

            def keep(call):               # a state off the EOS branch is the same error in both
                try:
                    out.append(call())
                except lbm.LBError as e:
                    out.append(e.status)

            for n in (2, 1, 5):
                if lbm.lb_status_of(lat.ctx) == lbm.LB_OK:
                    for m in [1] * n if variant == 8 else [n]:
                        lat.step(m)
                keep(lat.populations)
            if lbm.lb_status_of(lat.ctx) == lbm.LB_OK:
                if variant == 7:                  # the written state carries on elsewhere
                    lbm.lb_set_launch(lat.ctx, 4, 0)
                lat.step(2)
                assert lat.steps_done == 10
            for call in (lat.populations, lat.rho, lat.reduce):
                keep(call)
            states.append(out)
            lat.close()
        for a, b in zip(*states):
            assert np.array_equal(a, b), (nx, ny)


def test_domain_error_in_one_of_many_steps(lbm):  # noqa: F811
    eos = lbm.cs_eos(0.8)
    lat = lbm.Lattice(64, 64, eos, -1.0, prec="fp32", rates=lbm.RateParams.from_viscosity(0.1))
    rng = np.random.default_rng(3)
    f = I.random_populations(rng, np.full((64, 64), 0.3))
    f[:, 20, 20] = 0.0                            # no density at one site
    lat.set_populations(f)
    lat.step(3)
    with pytest.raises(lbm.LBError) as e:
        lat.sync()
    assert e.value.status == lbm.LB_EDOMAIN
    lat.close()
