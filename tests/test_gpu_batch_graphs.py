"""Batches of several groups of lattices: their steps are queued as graphs once the first 512 have been
launched one by one, and give the bits of the ring kernel's single launch per step over blocks of
groups, from either buffer, after a change of the active lattices and inside a capture. The calling
thread is not held while the GPU works."""
import threading
import time

import numpy as np
import pytest

import _capture
from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def batch(lbm, sides, stream=None):  # noqa: F811
    eos = lbm.cs_eos(0.8)
    rv, rl, _ = lbm.lb_maxwell(eos, -1.0)
    b = lbm.Batch([lbm.LatticeDesc(s, s + 1, eos, -1.0, kappa=0.3, sigma_force=0.05,
                                   rates=lbm.RateParams.from_viscosity(0.1)) for s in sides], stream=stream)
    for i, s in enumerate(sides):
        b.set_rho_u(i, I.droplet_density(s, s + 1, 0.2 * s + 0.01 * i, rl, rv))
    return b


# 2 groups, 3, 4 (15 lattices each), 12 (graphs of 32 steps), 50 (of 16, the second block has two), 49
# (the second block has one)
@pytest.mark.parametrize("sides", [[256] * 2, [512, 511, 301], [128] * 60, [512] * 12, [511] * 50, [512] * 49])
def test_bits_of_single_launches(lbm, sides):  # noqa: F811
    a, b = batch(lbm, sides), batch(lbm, sides)
    b.set_launch(4, 16)
    active = np.ones(len(sides), np.uint8)
    pick = sorted({0, 1, len(sides) // 2, len(sides) - 1})

    def same():
        for i in pick:
            assert np.array_equal(a.populations(i), b.populations(i)), i
        assert a.steps_done == b.steps_done

    for x in (a, b):
        x.step(500)                # one by one
        x.step(150)                # the last of these, then graphs
        x.step(16)
    same()
    for x in (a, b):
        x.step(1)                  # from the other buffer
        x.step(135)
    same()
    active[0] = 0
    for x in (a, b):
        x.set_active(active)
        x.step(513 + 133)
    same()
    a.close()
    b.close()


@pytest.mark.parametrize("warm", [False, True])
def test_captured_steps(lbm, warm):  # noqa: F811
    """recorded by the caller, before and after the batch has graphs of its own"""
    st = torch.cuda.Stream()
    sides = [512, 511, 301]
    a, b = batch(lbm, sides, st.cuda_stream), batch(lbm, sides)
    if warm:
        a.step(640)
        b.step(640)
    a.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        a.step(70)
    with torch.cuda.stream(st):
        for _ in range(2):
            graph.replay()
    a.sync()
    b.step(140)
    for i in range(3):
        assert np.array_equal(a.populations(i), b.populations(i))
    a.close()
    b.close()


def test_the_calling_thread_is_not_held(lbm):  # noqa: F811
    b = batch(lbm, [128] * 60)
    b.step(512)
    b.step(64)                     # the graphs are made
    held, whole = [], []
    for _ in range(5):
        b.sync()
        t = time.perf_counter()
        b.step(640)
        held.append(time.perf_counter() - t)
        b.sync()
        whole.append(time.perf_counter() - t)
    assert sorted(held)[2] < 0.5 * sorted(whole)[2], (held, whole)
    b.close()


def test_every_group_has_the_priority_of_the_stream(lbm):  # noqa: F811
    st = torch.cuda.Stream(priority=-1)
    assert st.priority < 0
    b = batch(lbm, [512, 511, 301], st.cuda_stream)
    b.sync()
    _capture.begin(st.cuda_stream)
    b.step(2)
    graph = _capture.end(st.cuda_stream)
    assert _capture.kernel_priorities(graph) == [st.priority] * 6
    _capture.destroy(graph)
    b.close()


@pytest.mark.parametrize("variant,partly", [(8, False), (8, True), (4, True)])
def test_steps_that_fail(lbm, variant, partly):  # noqa: F811
    """A capture that is spoilt while the steps are being recorded: some lattices have moved on and
    others not, so the batch refuses everything afterwards. Spoilt before, nothing has happened."""
    st = torch.cuda.Stream()
    b = batch(lbm, [512, 511, 301], st.cuda_stream)
    b.set_launch(variant, 16)
    b.sync()
    _capture.begin(st.cuda_stream)

    def spoil():                   # waiting for a stream that is being captured
        if partly:
            time.sleep(0.01)
        st.synchronize()

    t = threading.Thread(target=lambda: pytest.raises(RuntimeError, spoil))
    t.start()
    if not partly:
        t.join()
    with pytest.raises(lbm.LBError) as e:
        b.step(100000)             # far longer than the wait
    assert e.value.status == lbm.LB_ECUDA
    t.join()
    assert _capture.end(st.cuda_stream) is None
    if partly:
        for call in (lambda: b.step(1), b.sync, lambda: b.measure([50.0] * 3), lambda: b.populations(0)):
            with pytest.raises(lbm.LBError) as e:
                call()
            assert e.value.status == lbm.LB_ECUDA
    else:
        b.step(2)
        b.sync()
        assert b.steps_done == 2
    b.close()


def step_us(b, calls=40):
    t = []
    for _ in range(7):
        b.sync()
        a = time.perf_counter()
        for _ in range(calls):
            b.step(1)
        b.sync()
        t.append((time.perf_counter() - a) / calls * 1e6)
    return sorted(t)[3]


def test_single_steps_of_a_tuned_batch(lbm):  # noqa: F811
    """A batch tuned for many steps takes single ones no slower than its fastest ring launch, with the
    bits of any other launch, also after a change of the active lattices."""
    sides = [1024, 1000]
    a, b = batch(lbm, sides), batch(lbm, sides)
    a.autotune(8)
    assert a.launch()["variant"] == 8 and a.steps_done == 0
    ring = 1e9
    for variant in range(7):
        for rows in (8, 16, 24):
            b.set_launch(variant, rows)
            ring = min(ring, step_us(b))
    assert step_us(a) < 1.1 * ring
    a.close()
    a = batch(lbm, sides)
    a.autotune(8)
    b.close()
    b = batch(lbm, sides)
    b.set_launch(4, 16)
    for x in (a, b):
        for n in (1, 2, 64, 3, 4, 1, 1):
            x.step(n)
    for i in range(2):
        assert np.array_equal(a.populations(i), b.populations(i))
    for x in (a, b):
        x.set_active(np.array([0, 1], np.uint8))
        for n in (1, 17, 2, 4):
            x.step(n)
    for i in range(2):
        assert np.array_equal(a.populations(i), b.populations(i)) and a.lattice_steps(i) == b.lattice_steps(i)
    a.close()
    b.close()


@pytest.mark.parametrize("sides,before", [([64] * 3, 2), ([512, 511, 301], 512)])   # 1 and 3 groups
def test_steps_beside_a_capture_of_another_stream(lbm, sides, before):  # noqa: F811
    """The thread records into a stream of its own while the batch, whose graphs are not made yet, steps
    in another: the steps are taken, and the recording is not spoilt."""
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = batch(lbm, sides, st.cuda_stream), batch(lbm, sides)
    a.step(before)
    b.step(before)
    a.sync()
    _capture.begin(other.cuda_stream)
    a.step(128)
    graph = _capture.end(other.cuda_stream)
    assert graph is not None
    _capture.destroy(graph)
    b.step(128)
    for i in range(3):
        assert np.array_equal(a.populations(i), b.populations(i))
    a.close()
    b.close()
