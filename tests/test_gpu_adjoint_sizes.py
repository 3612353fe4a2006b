"""The adjoint's products at the edges of their tiles: layer widths around 16,
32 and 33, more than one output, fewer vertices than a tile, against the
oracle's implicit-function gradient (float64).

The adjoint's sums carry about 44 bits; an ill-conditioned crossing (edge
length 1e-4 of the box) amplifies them by up to ~1e8 in dt/da, of which the
quotient form loses the square root: 1e-7 of the largest component bounds what
is left with a wide margin, and a wrong index in any kernel is off by the order
of the components themselves."""
import numpy as np
import pytest

import oracle
from paper_2306_07212_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[1, 5, 1], [2, 3, 2], [2, 15, 17, 1], [2, 31, 33, 2], [3, 16, 32, 1], [2, 64, 9, 40, 1],
                                    [4, 7, 8, 1], [2, 129, 6, 1]])
def test_gradient_matches_the_oracle(widths):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    from paper_2306_07212_gb300.autograd import extract_vertices
    net = wl.he_normal_mlp(widths, seed=8).rounded_to_fp32()
    box = wl.Box.cube(widths[0])
    theta = torch.tensor(net.flat_params(), dtype=torch.float64, device="cuda", requires_grad=True)
    with Extractor(precision="fp64", keep_tape=True) as ex:
        X = extract_vertices(theta, ex, net, box)
        (X.sin() * X).sum().backward()  # every vertex, whatever its number
    ref = oracle.extract(net, box)
    g = oracle.grad(net, ref, np.sin(ref.X) + ref.X * np.cos(ref.X))
    assert np.max(np.abs(theta.grad.cpu().numpy() - g)) <= 1e-7 * np.max(np.abs(g))
