"""The bounded waits of the staged tiles and of the resident kernel, made to run out by the test hook (a
load that is never issued, an exchange word that is never published): the call that synchronises
reports LB_ETIMEOUT, the context stays poisoned, and a fresh context of the same lattice steps as if
nothing had happened. (The ring kernels' waits: test_gpu_parity.)"""
import numpy as np
import pytest

from test_gpu_many_steps import STEPS, launches
from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

INT_MIN = -2**31


def lattice(lbm, nx, ny, bc, prec):  # noqa: F811
    lat = lbm.Lattice(nx, ny, lbm.EOSParams(kind="exp"), -40.0, prec=prec, walls_y=bc == "walls",
                      open_bc=bc == "open", storage_shift=400.0 if prec == "bf16" else 0.0)
    rng = np.random.default_rng(1)
    lat.set_rho_u(400.0 * (1 + 0.01 * rng.standard_normal((ny, nx))))
    return lat


def times_out(lbm, lat, n):  # noqa: F811
    lat.step(n)
    with pytest.raises(lbm.LBError) as e:
        lat.sync()
    assert e.value.status == lbm.LB_ETIMEOUT
    with pytest.raises(lbm.LBError) as e:
        lat.step(n)
    assert e.value.status == lbm.LB_ETIMEOUT == lbm.lb_status_of(lat.ctx)
    lat.close()


def steps_as_before(lbm, args, n, expected):  # noqa: F811
    lat = lattice(lbm, *args)
    lat.step(n)
    assert np.array_equal(lat.populations(), expected)
    lat.close()


def after(lbm, args, n):  # noqa: F811
    lat = lattice(lbm, *args)
    lat.step(n)
    out = lat.populations()
    lat.close()
    return out


# a row of the first staged tile, of an inner one, of the last
@pytest.mark.parametrize("args,row", [((70, 64, "periodic", "bf16"), 2), ((70, 64, "walls", "bf16"), 31),
                                      ((70, 61, "open", "fp32"), 60), ((130, 64, "periodic", "fp32"), 61)])
def test_staged_tile(lbm, args, row):  # noqa: F811
    good = after(lbm, args, 3)
    lat = lattice(lbm, *args)
    lbm.lb_set_launch(lat.ctx, 8, 0)
    lbm.lb_debug_stall_row(lat.ctx, row)
    assert lbm.lb_get_launch(lat.ctx)["variant"] == 8
    times_out(lbm, lat, 1)
    steps_as_before(lbm, args, 3, good)


def test_rows_that_no_staged_tile_loads(lbm):  # noqa: F811
    lat = lattice(lbm, 70, 64, "periodic", "bf16")
    lbm.lb_debug_stall_row(lat.ctx, 0)
    assert lbm.lb_get_launch(lat.ctx)["variant"] == 4
    times_out(lbm, lat, 1)


# border and inner rows of a tile, the seam, a lattice of one tile column
@pytest.mark.parametrize("args,row", [((200, 200, "periodic", "fp32"), 0), ((200, 200, "walls", "fp32"), 100),
                                      ((600, 225, "open", "fp32"), 7), ((64, 5000, "periodic", "fp32"), 4999)])
def test_resident_kernel(lbm, args, row):  # noqa: F811
    good = after(lbm, args, STEPS)
    lat = lattice(lbm, *args)
    lbm.lb_debug_stall_row(lat.ctx, row)
    before = lbm.lb_step_launches(lat.ctx)
    lat.step(STEPS)
    assert lbm.lb_step_launches(lat.ctx) - before == 1
    with pytest.raises(lbm.LBError) as e:
        lat.sync()
    assert e.value.status == lbm.LB_ETIMEOUT
    lat.close()
    steps_as_before(lbm, args, STEPS, good)


@pytest.mark.parametrize("args", [(64, 64, "periodic", "fp32"), (200, 200, "periodic", "fp32"),
                                  (70, 64, "periodic", "bf16"), (70, 64, "periodic", "fp64")])
def test_hook_switched_off(lbm, args):  # noqa: F811
    """the launch is what it was, for one step and for many; a launch chosen while the hook is on is
    taken when it is off"""
    good = after(lbm, args, STEPS)
    lat = lattice(lbm, *args)
    shape, n = lbm.lb_get_launch(lat.ctx), launches(lbm, lat, STEPS)
    lat.close()
    lat = lattice(lbm, *args)
    lbm.lb_debug_stall_row(lat.ctx, 20)
    lbm.lb_set_launch(lat.ctx, 7, 0)
    assert lbm.lb_get_launch(lat.ctx)["variant"] == 4
    lbm.lb_set_launch(lat.ctx, shape["variant"], 0)
    lbm.lb_debug_stall_row(lat.ctx, INT_MIN)
    assert lbm.lb_get_launch(lat.ctx) == shape and launches(lbm, lat, STEPS) == n
    assert np.array_equal(lat.populations(), good)
    lat.close()
