"""Several steps of a mid-size FP32 lattice in one launch (the resident kernel, taken by contexts with
their default launch variant) give the bits of single steps: at the edges of how it cuts a lattice
(last tiles of 2, 3, 53 and 64 columns, tiles of 4 to 35 rows, one tile across or up the lattice, a
last tile of one column, which it leaves to single steps), for every boundary kind and EOS, over
several launches and carried on by another kernel."""
import numpy as np
import pytest

from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import case_params, lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(194, 200), (195, 203), (193, 200), (501, 383), (600, 225), (128, 300), (7, 5000), (64, 5000),
         (9000, 4), (8000, 5), (6400, 8), (560, 560)]


def run(lbm, nx, ny, kind, bc, chunks):  # noqa: F811
    eos, G, (lo, hi) = case_params(lbm, kind)
    rng = np.random.default_rng(nx * 100 + ny)
    rho = I.smooth_random_density(rng, nx, ny, lo, hi)
    ux, uy = I.random_velocity(rng, rho.shape, 1e-3)
    kw = {"walls_y": bc == "walls", "open_bc": bc == "open"}
    if bc == "open":
        kw["viscosity_switch"] = (0.5 * (lo + hi), 1.1)
    lat = lbm.Lattice(nx, ny, eos, G, kappa=0.4, sigma_force=0.05, prec="fp32",
                      rates=lbm.RateParams.from_viscosity(0.1), **kw)
    lat.set_rho_u(rho, ux, uy)
    out = []

    def keep():
        try:
            out.append(lat.populations())
        except lbm.LBError as e:              # off the EOS branch: the same error either way
            out.append(e.status)

    for i, m in enumerate(chunks):
        if lbm.lb_status_of(lat.ctx) == lbm.LB_OK:
            lat.step(m)
        if i % 4 == 3:                        # the written state, with its ghost columns
            keep()
    if lbm.lb_status_of(lat.ctx) == lbm.LB_OK:
        assert lat.steps_done == sum(chunks)
        lbm.lb_set_launch(lat.ctx, 4, 0)
        lat.step(2)
    keep()
    lat.close()
    return out


@pytest.mark.parametrize("bc", ["periodic", "walls", "open"])
@pytest.mark.parametrize("kind", ["cs", "exp", "piecewise"])
def test_many_steps_in_one_launch(lbm, bc, kind):  # noqa: F811
    for nx, ny in SIZES:
        many = run(lbm, nx, ny, kind, bc, [2, 3, 1, 2, 6, 2, 1, 3])
        single = run(lbm, nx, ny, kind, bc, [1] * 20)
        for a, b in zip((many[0], many[1], many[2]), (single[1], single[4], single[5])):
            assert np.array_equal(a, b), (nx, ny)


@pytest.mark.parametrize("size", [(64, 64), (200, 160)])   # the cluster kernel, the resident one
def test_captured_launches_replay(lbm, size):  # noqa: F811
    """a captured even number of steps ends in the buffer it starts from, so its replays go on stepping,
    as those of single launches do; a captured odd number leaves the state in the other buffer"""
    eos, G, (lo, hi) = case_params(lbm, "cs")
    nx, ny = size
    rho = I.smooth_random_density(np.random.default_rng(5), nx, ny, lo, hi)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lat, ref = (lbm.Lattice(nx, ny, eos, G, kappa=0.4, prec="fp32",
                                rates=lbm.RateParams.from_viscosity(0.1)) for _ in range(2))
    for x in (lat, ref):
        x.set_rho_u(rho, 0 * rho, 0 * rho)
    lat.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        lat.step(6)
    with torch.cuda.stream(st):
        for _ in range(3):
            graph.replay()
    for _ in range(18):
        ref.step(1)
    assert np.array_equal(lat.populations(), ref.populations())
    for n in (5, 2):
        lat.step(n)
    for _ in range(7):
        ref.step(1)
    assert np.array_equal(lat.populations(), ref.populations())
    lat.close()
    ref.close()
