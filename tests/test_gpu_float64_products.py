"""The float64 layer products at the edges of their tiles: widths around 16, 32
and 64 outputs, odd and one-neuron layers, up to the widest layer, and fewer
vertices than a tile.  Every last-layer value must be the network's at the
vertex (float64 forward pass by numpy on the vertex's own piece), off by at most
1e-9 of the sum of |terms|: crossings interpolate with a few roundings of 2^-53
each, amplified by short edges (1e-4 of the box at the worst here)."""
import numpy as np
import pytest

from paper_2306_07212_gb300 import workloads as wl
from _util import unpack_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[1, 3, 1], [2, 15, 16, 17, 1], [2, 31, 33, 2], [3, 20, 3, 1], [2, 63, 65, 1],
                                    [2, 64, 64, 3], [2, 129, 7, 1], [2, 256, 5, 1], [2, 9, 200, 1]])
def test_values_are_the_networks(widths):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net, box = wl.he_normal_mlp(widths, seed=2), wl.Box.cube(widths[0])
    with Extractor(precision="fp64") as ex:
        ex.extract(net, box)
        X, S, Z = ex.vertices(), unpack_codes(ex.sign_words(), ex.counts()["P"]), ex.values()
    a, at = X, 2 * widths[0]
    for W, b in zip(net.W, net.b):
        z, terms = a @ W.T + b, np.abs(a) @ np.abs(W).T + np.abs(b)
        a, at = np.where(S[:, at:at + len(b)] > 0, z, 0.0), at + len(b)
    assert Z.shape == z.shape and np.max(np.abs(Z - z) / terms) <= 1e-9
