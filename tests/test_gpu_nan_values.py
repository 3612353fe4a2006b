"""A NaN pre-activation (a parameter that became NaN) spreads to the values of
the layers behind it: its sign entry is +, so it is an active input, and a
caller sees it in values() and in the gradient instead of finite numbers.

The NaN sits in the bias of the first layer's last neuron, so that every
vertex of the first layer's complex has it; each layer product is taken (float64,
tensor cores with rows of 4 floats and others, SIMT, wider than 128)."""
import numpy as np
import pytest

from paper_2306_07212_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _net(widths):
    net = wl.he_normal_mlp(widths, seed=4).rounded_to_fp32()
    b = [x.copy() for x in net.b]
    b[0][-1] = np.nan
    return wl.Net(widths, net.W, b), wl.Box.cube(widths[0])


@pytest.fixture(scope="module")
def Extractor():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    return Extractor


@pytest.mark.parametrize("kw", [{"precision": "fp64"}, {"precision": "mixed"}, {"precision": "mixed", "gemm": "simt"},
                                {"precision": "fp32"}], ids=["fp64", "mixed", "simt", "fp32"])
@pytest.mark.parametrize("widths", [[2, 8, 8, 2], [2, 7, 9, 1], [2, 140, 6, 1]])
def test_values_are_nan(Extractor, widths, kw):
    net, box = _net(widths)
    with Extractor(**kw) as ex:
        ex.extract(net, box)
        Z = ex.values()
    assert len(Z) > 10 and np.isnan(Z).all()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_gradient_is_nan(Extractor, precision):
    import torch
    net, box = _net([2, 8, 8, 1])
    with Extractor(precision=precision, keep_tape=True) as ex:
        ex.extract(net, box)
        c = ex.counts()
        g = torch.ones((c["D"], c["nV"]), dtype=torch.float64, device="cuda")
        out = torch.zeros(net.flat_params().size, dtype=torch.float64, device="cuda")
        ex.backward(g, out)
    dW2 = out.cpu().numpy()[24:88].reshape(8, 8)
    assert np.isnan(dW2[:, -1]).all()
