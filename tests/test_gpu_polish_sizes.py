"""The coordinate polish at the sizes where its kernel takes another path: layer
widths around its passes (8 or 16 lanes, up to 8 outputs each), input
dimensions around its record sizes, networks whose weights fit in shared memory
or not, with and without float32 remainders.

With a negligible tolerance every vertex with a coordinate error estimate is
moved.  Its zero entries, evaluated in float64 at the result, must then vanish:
the values are evaluated in float-float (about 2^-44 of the sum of |terms|) and
the step solved in float32 removes all but ~1e-6 of a residual of ~1e-7 of that
sum, so 1e-9 of the sum leaves three orders of margin and is two below what the
FP32 coordinates give."""
import numpy as np
import pytest

from paper_2306_07212_gb300 import workloads as wl
from _util import unpack_codes

pytestmark = pytest.mark.gpu

NETS = [[1, 5, 1], [2, 7, 9, 1], [2, 63, 65, 1], [2, 64, 64, 1], [2, 72, 80, 3], [2, 127, 129, 1], [2, 136, 8, 1],
        [2, 200, 16, 1], [2, 256, 9, 1], [3, 24, 17, 1], [4, 10, 11, 1], [5, 9, 8, 1], [6, 8, 7, 1], [7, 7, 8, 1],
        [8, 8, 9, 1]]


@pytest.mark.parametrize("widths", NETS)
@pytest.mark.parametrize("rounded", [True, False])
def test_polished_vertices_lie_on_their_zero_sets(widths, rounded):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net = wl.he_normal_mlp(widths, seed=5)
    if rounded:
        net = net.rounded_to_fp32()
    box = wl.Box.cube(widths[0])
    with Extractor(precision="mixed", polish_tol=1e-30) as ex:
        ex.extract(net, box)
        X, S = ex.vertices(), unpack_codes(ex.sign_words(), ex.counts()["P"])
        polished, exc = ex.diagnostics()["polished"], ex.error_estimates()[1]
    assert polished == int((exc > 0).sum()) > 0
    m = 2 * widths[0]
    a, at = X, m
    worst = 0.0
    for W, b in zip(net.W, net.b):
        z, terms = a @ W.T + b, np.abs(a) @ np.abs(W).T + np.abs(b)
        s = S[:, at:at + len(b)]
        worst = max(worst, float(np.max(np.abs(z) / terms, initial=0.0, where=s == 0)))
        a, at = np.where(s > 0, z, 0.0), at + len(b)
    assert worst <= 1e-9
    facets = np.stack([X - box.lo, box.hi - X], axis=2).reshape(len(X), m)
    assert float(np.max(np.abs(facets), initial=0.0, where=S[:, :m] == 0)) <= 1e-9
