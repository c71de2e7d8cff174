"""lb_get_launch reports the resident CTAs per SM of the kernel that the context's steps are, as the
occupancy calculator has it: what the tile kernels are compiled for (65536 registers by threads of at
most 80 registers for the direct tiles, 64 for the staged ones, 128 with stochastic rounding) up to one
more CTA where fewer registers are used, and for FP64 the fewer of its two kernels."""
import pytest

from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,stochastic,variant,least,most", [
    ("fp32", False, 7, 6, 16), ("fp32", False, 8, 8, 13), ("bf16", False, 8, 8, 16), ("bf16", True, 8, 4, 7),
    ("bf16", True, 7, 4, 7), ("fp64", False, 7, 1, 31)])
def test_resident_ctas(lbm, prec, stochastic, variant, least, most):  # noqa: F811
    lat = lbm.Lattice(70, 64, lbm.cs_eos(0.8), -1.0, prec=prec,
                      **({"storage_shift": 0.02, "stochastic_rounding": stochastic} if prec == "bf16" else {}))
    lbm.lb_set_launch(lat.ctx, variant, 0)
    shape = lbm.lb_get_launch(lat.ctx)
    assert shape["variant"] == variant and least <= shape["ctas_per_sm"] <= most
    lat.close()
