"""Making and freeing a context costs less than one page-locked allocation; what the kernels write into
its host words (error bits, sums) arrives whatever the order in which contexts come and go."""
import ctypes as C
import time

import numpy as np
import pytest

from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def median(call, n=31):
    t = []
    for _ in range(n):
        torch.cuda.synchronize()
        a = time.perf_counter()
        call()
        t.append(time.perf_counter() - a)
    return sorted(t)[n // 2]


def test_cost(lbm):  # noqa: F811
    driver, p = C.CDLL("libcuda.so.1"), C.c_void_p()
    torch.zeros(1, device="cuda")

    def locked():
        assert driver.cuMemHostAlloc(C.byref(p), C.c_size_t(4096), 0) == 0
        assert driver.cuMemFreeHost(p) == 0

    def context():
        lbm.Lattice(64, 64, lbm.EOSParams(kind="exp"), -40.0, prec="fp32").close()

    context()
    assert median(context) < median(locked)


def test_words_of_contexts_that_come_and_go(lbm):  # noqa: F811
    lats = []
    for i in range(40):
        lat = lbm.Lattice(8 + i, 9, lbm.EOSParams(kind="exp"), -40.0, prec="fp64")
        lat.set_rho_u(np.full((9, 8 + i), 100.0 + i))
        lats.append(lat)
        if i % 3 == 2:
            lats.pop(0).close()
    for lat in lats[::2]:
        f = lat.populations()
        f[:, 4, 4] = 0.0
        lat.set_populations(f)
    for lat in lats:
        lat.step(1)
    for i, lat in enumerate(lats):
        if i % 2 == 0:
            with pytest.raises(lbm.LBError) as e:
                lat.reduce()
            assert e.value.status == lbm.LB_EDOMAIN
        else:
            rho = 100.0 + lat.nx - 8
            assert lat.reduce()[0] == pytest.approx(rho * lat.nx * 9, rel=1e-13)
        lat.close()
