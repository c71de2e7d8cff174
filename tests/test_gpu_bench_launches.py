"""bench.py's count of kernel launches is what the library queued: one for the steps of a lattice that
takes them together, one each where the lattice is too large for one kernel and too small for the
other, and one each where another launch variant was chosen."""
import pytest

from test_bench_host import bench  # noqa: F401
from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,variant,per_chunk", [(64, 64, 7, 1), (180, 160, 7, 40), (64, 64, 4, 40)])
def test_launch_count(bench, lbm, nx, ny, variant, per_chunk):  # noqa: F811
    from paper_1306_6445_gb300 import inputs

    launches = bench.time_precision(lbm, torch, inputs, "fp32", nx, ny, 40, 2, 1, None, launch=(variant, 0))[2]
    assert launches == 2 * (per_chunk + 2)      # two chunks, each with a reduction of two kernels
