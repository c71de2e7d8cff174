"""Which lattices take several steps in one launch (the cluster kernel and the resident one), as counted
by lb_step_launches, and what a launch that cannot be made does to the context."""
import threading
import time

import numpy as np
import pytest

import _capture
from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STEPS = 40          # more than the fewest steps that one launch is made for


def lattice(lbm, nx, ny, bc="periodic", prec="fp32"):  # noqa: F811
    """uniform liquid at rest: any number of steps leaves it"""
    lat = lbm.Lattice(nx, ny, lbm.EOSParams(kind="exp"), -40.0, prec=prec, walls_y=bc == "walls",
                      open_bc=bc == "open")
    lat.set_rho_u(np.full((ny, nx), 400.0))
    return lat


def launches(lbm, lat, n):  # noqa: F811
    before = lbm.lb_step_launches(lat.ctx)
    lat.step(n)
    return lbm.lb_step_launches(lat.ctx) - before


# the cluster kernel: even nx >= 4, ny >= 16, at most 512 site pairs per 1/16 of the rows, no open
# sides; the resident kernel: from 32768 sites and 96 tiles on while tiles of 64 x 35 suffice, a last
# tile of two columns at least
MANY = [(4, 16, "periodic"), (64, 64, "periodic"), (66, 17, "walls"), (1024, 16, "periodic"), (128, 128, "walls"),
        (194, 200, "periodic"), (195, 203, "walls"), (501, 383, "periodic"), (600, 225, "open"), (128, 300, "open"),
        (7, 5000, "walls"), (9000, 4, "periodic"), (6400, 8, "walls"), (560, 560, "periodic")]
SINGLE = [(64, 15, "periodic"), (63, 64, "periodic"), (64, 64, "open"), (128, 129, "periodic"), (180, 180, "walls"),
          (193, 200, "periodic"), (5000, 20, "periodic"), (700, 700, "periodic")]


@pytest.mark.parametrize("nx,ny,bc", MANY)
def test_many_steps_are_one_launch(lbm, nx, ny, bc):  # noqa: F811
    lat = lattice(lbm, nx, ny, bc)
    assert launches(lbm, lat, 1) == 1
    assert launches(lbm, lat, STEPS) == 1
    assert launches(lbm, lat, 1024 + STEPS) == 2
    lat.sync()
    assert lat.steps_done == 1 + STEPS + 1024 + STEPS
    lat.close()


@pytest.mark.parametrize("nx,ny,bc", SINGLE)
def test_other_lattices_take_single_launches(lbm, nx, ny, bc):  # noqa: F811
    lat = lattice(lbm, nx, ny, bc)
    assert launches(lbm, lat, STEPS) == STEPS
    lat.close()


@pytest.mark.parametrize("prec,per_step", [("fp64", 2), ("bf16", 1)])
def test_other_types_take_single_launches(lbm, prec, per_step):  # noqa: F811
    lat = lattice(lbm, 64, 64, prec=prec)
    assert launches(lbm, lat, STEPS) == STEPS * per_step
    lat.close()


@pytest.mark.parametrize("nx,ny", [(64, 64), (200, 200)])
def test_a_launch_that_fails_is_reported_and_changes_nothing(lbm, nx, ny):  # noqa: F811
    """A call that waits inside a capture is an error and spoils the capture, so the steps after it
    fail too: that is reported, and the context takes its steps together again afterwards."""
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lat = lattice(lbm, nx, ny)
    lat.sync()
    _capture.begin(st.cuda_stream)
    with pytest.raises(lbm.LBError):
        lat.sync()
    with pytest.raises(lbm.LBError) as e:
        lat.step(STEPS)
    assert e.value.status == lbm.LB_ECUDA
    assert _capture.end(st.cuda_stream) is None
    assert launches(lbm, lat, STEPS) == 1
    lat.sync()
    assert lat.steps_done == STEPS
    lat.close()


@pytest.mark.parametrize("sizes", [((4, 16), (128, 128)), ((195, 200), (560, 560))])
def test_lattices_of_different_size_step_side_by_side(lbm, sizes):  # noqa: F811
    """Two host threads step a small and a large lattice, which one kernel takes with different amounts
    of shared memory: neither loses its launches of many steps."""
    lats = []
    for size in sizes:
        with torch.cuda.stream(torch.cuda.Stream()):
            lats.append(lattice(lbm, *size))
    calls = 2000
    before = [lbm.lb_step_launches(lat.ctx) for lat in lats]

    def work(lat):
        for i in range(calls):
            lat.step(STEPS)
            if i % 50 == 0:
                lat.sync()
        lat.sync()

    threads = [threading.Thread(target=work, args=(lat,)) for lat in lats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [lbm.lb_step_launches(lat.ctx) - b for lat, b in zip(lats, before)] == [calls, calls]
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("nx,ny,bc", [(64, 64, "walls"), (200, 200, "periodic"), (600, 225, "open")])
def test_autotuning(lbm, nx, ny, bc):  # noqa: F811
    """The launch of single steps is chosen by trials (each takes a microsecond a step at the very
    least), also where many steps go together, which they do afterwards whatever was chosen."""
    lat = lattice(lbm, nx, ny, bc)
    lbm.lb_set_launch(lat.ctx, 4, 0)
    lat.step(2)
    before = lat.populations()
    t = time.perf_counter()
    variant, _ = lat.autotune(3000)
    assert time.perf_counter() - t > 2 * 3 * 3000 * 1e-6
    assert variant in (7, 8) and lbm.lb_get_launch(lat.ctx)["variant"] == variant
    assert np.array_equal(lat.populations(), before) and lat.steps_done == 2
    assert launches(lbm, lat, 1) == 1 and launches(lbm, lat, STEPS) == 1
    lbm.lb_debug_stall_row(lat.ctx, 3)      # (a test hook that renews the launch)
    lbm.lb_debug_stall_row(lat.ctx, -2**31)
    assert launches(lbm, lat, STEPS) == 1
    lat.sync()
    lat.close()
