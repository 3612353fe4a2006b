"""The adjoint of networks whose parameters are not float32 (after one optimiser
step none is): the layer products take the weights' remainders too.

Sums of float pairs carry about 44 bits (6e-14) and the crossings amplify an
error by up to about 1e4 (edges of 1e-4 of the box, in the quotient form):
6e-10 of the largest component, so 1e-9.  Weights rounded to float32 instead
are off by 3e-8 each."""
import numpy as np
import pytest

import oracle
from paper_2306_07212_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[2, 15, 17, 1], [3, 16, 32, 1], [2, 33, 9, 20, 2]])
def test_gradient_matches_the_oracle(widths):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    from paper_2306_07212_gb300.autograd import extract_vertices
    net = wl.he_normal_mlp(widths, seed=8)
    assert not np.array_equal(net.flat_params(), net.rounded_to_fp32().flat_params())
    box = wl.Box.cube(widths[0])
    theta = torch.tensor(net.flat_params(), dtype=torch.float64, device="cuda", requires_grad=True)
    with Extractor(precision="fp64", keep_tape=True) as ex:
        X = extract_vertices(theta, ex, net, box)
        (X.sin() * X).sum().backward()
    ref = oracle.extract(net, box)
    g = oracle.grad(net, ref, np.sin(ref.X) + ref.X * np.cos(ref.X))
    err = np.max(np.abs(theta.grad.cpu().numpy() - g)) / np.max(np.abs(g))
    print(f"\n{widths}: {err:.2e}")
    assert err <= 1e-9
