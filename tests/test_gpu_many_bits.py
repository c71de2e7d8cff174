"""Many steps in one launch (the cluster kernel and the resident one, from the fewest steps that they take
on) give the bits of single steps: over several launches mixed with single steps, at the edges of what
the two kernels take, for every boundary kind and EOS, carried on by another kernel, and replayed from
a capture."""
import numpy as np
import pytest

from paper_1306_6445_gb300 import inputs as I
from test_gpu_cluster import SIZES as CLUSTER
from test_gpu_many_steps import lattice, launches
from test_gpu_parity import case_params, lbm  # noqa: F401
from test_gpu_resident import SIZES as RESIDENT
from test_gpu_resident import run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,least", [(64, 64, 7), (200, 200, 10)])
def test_fewest_steps(lbm, nx, ny, least):  # noqa: F811
    lat = lattice(lbm, nx, ny)
    for n in range(1, least):
        assert launches(lbm, lat, n) == n
    assert launches(lbm, lat, least) == launches(lbm, lat, 1024) == 1
    assert launches(lbm, lat, 1024 + least) == 2
    assert launches(lbm, lat, 1024 + least - 1) == 1 + least - 1
    lat.close()


# run() keeps the state after every fourth chunk and at the end
@pytest.mark.parametrize("sizes,bcs,chunks", [
    (CLUSTER, ("periodic", "walls"), [7, 8, 1, 12, 9, 2, 17, 12]),
    (RESIDENT, ("periodic", "walls", "open"), [10, 11, 1, 10, 13, 12, 1, 10])])
@pytest.mark.parametrize("kind", ["cs", "exp", "piecewise"])
def test_bits_of_single_steps(lbm, kind, sizes, bcs, chunks):  # noqa: F811
    first, both = sum(chunks[:4]), sum(chunks)
    for bc in bcs:
        for nx, ny in sizes:
            many = run(lbm, nx, ny, kind, bc, chunks)
            single = run(lbm, nx, ny, kind, bc, [1] * both)
            for a, b in zip(many, (single[first // 4 - 1], single[both // 4 - 1], single[-1])):
                assert np.array_equal(a, b), (bc, nx, ny)


@pytest.mark.parametrize("size", [(64, 64), (210, 160)])
def test_captured_launches_replay(lbm, size):  # noqa: F811
    """a captured even number of steps ends in the buffer it starts from, so its replays go on stepping"""
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
        assert launches(lbm, lat, 12) == 1
    with torch.cuda.stream(st):
        for _ in range(3):
            graph.replay()
    for _ in range(36):
        ref.step(1)
    assert np.array_equal(lat.populations(), ref.populations())
    for n in (11, 10):
        assert launches(lbm, lat, n) == 1
    for _ in range(21):
        ref.step(1)
    assert np.array_equal(lat.populations(), ref.populations())
    lat.close()
    ref.close()


@pytest.mark.parametrize("size", [(64, 64), (200, 200)])
def test_domain_error_in_one_of_many_steps(lbm, size):  # noqa: F811
    nx, ny = size
    lat = lbm.Lattice(nx, ny, lbm.cs_eos(0.8), -1.0, prec="fp32", rates=lbm.RateParams.from_viscosity(0.1))
    f = I.random_populations(np.random.default_rng(3), np.full((ny, nx), 0.3))
    f[:, 20, 20] = 0.0                            # no density at one site
    lat.set_populations(f)
    assert launches(lbm, lat, 12) == 1
    with pytest.raises(lbm.LBError) as e:
        lat.sync()
    assert e.value.status == lbm.LB_EDOMAIN
    lat.close()
