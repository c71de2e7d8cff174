"""An error of the runtime is reported once: by the call that met it, not again by the next one of the
same thread, whichever object that is of."""
import numpy as np
import pytest

import _capture
from paper_1306_6445_gb300 import inputs as I
from test_gpu_parity import lbm  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def lattice(lbm, stream):  # noqa: F811
    with torch.cuda.stream(stream):
        return lbm.Lattice(16, 16, lbm.EOSParams(kind="exp"), -40.0)


def batch(lbm, stream):  # noqa: F811
    return lbm.Batch([lbm.LatticeDesc(16, 16, lbm.EOSParams(kind="exp"), -40.0)], stream=stream.cuda_stream)


def network(lbm, stream):  # noqa: F811
    return lbm.MLP(16, stream=stream.cuda_stream)


@pytest.mark.parametrize("make,call", [(lattice, lambda x: x.sync()), (batch, lambda x: x.sync()),
                                       (network, lambda x: x.params())])
def test_reported_once(lbm, make, call):  # noqa: F811
    st = torch.cuda.Stream()
    x = make(lbm, st)
    st.synchronize()
    _capture.begin(st.cuda_stream)
    with pytest.raises(lbm.LBError) as e:
        call(x)                    # waits for a stream that is being captured
    assert e.value.status == lbm.LB_ECUDA
    assert _capture.end(st.cuda_stream) is None

    lat = lattice(lbm, torch.cuda.Stream())
    lat.set_rho_u(np.full((16, 16), 400.0))
    lat.step(1)
    assert lat.reduce()[0] == pytest.approx(400.0 * 256)
    b = batch(lbm, torch.cuda.Stream())
    b.set_rho_u(0, np.full((16, 16), 400.0))
    b.step(1)
    b.sync()
    net = network(lbm, torch.cuda.Stream())
    net.set_params(I.mlp_init(1))
    for y in (x, lat, b, net):
        y.close()
