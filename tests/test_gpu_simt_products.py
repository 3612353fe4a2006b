"""The SIMT layer product at the edges of its tiles (rows of fewer than 32 inputs,
one chunk, remainders, 16 outputs and others, wider than the tensor cores
take): the oracle's complex, and the last layer's values against a float64
forward pass at the vertices.  K float32 multiply-adds and float32-accurate
crossings: 1e-4 of the largest value, as for the other products; a row or
column out of place is off by the order of the values."""
import numpy as np
import pytest

import oracle
from paper_2306_07212_gb300 import workloads as wl
from _util import assert_same_complex, forward_all, unpack_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[2, 15, 16, 17], [2, 31, 33, 5], [2, 32, 32, 1], [2, 33, 63, 16], [3, 64, 15, 1],
                                    [2, 130, 97, 2]])
def test_product_at_its_edges(widths):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net = wl.he_normal_mlp(widths, seed=6).rounded_to_fp32()
    box = wl.Box.cube(widths[0], 1.0 if widths[0] == 2 else 0.3)
    ref = oracle.extract(net, box)
    with Extractor(precision="mixed", gemm="simt") as ex:
        ex.extract(net, box)
        X, Z = ex.vertices(), ex.values()
        got = X, unpack_codes(ex.sign_words(), ex.counts()["P"]), ex.edges()
    tol = 1e-6 * float(np.linalg.norm(box.hi - box.lo))
    assert_same_complex(got, (ref.X, ref.S, ref.E), coord_tol=tol, what=str(widths))
    z = forward_all(net, X)[:, -widths[-1]:]
    assert np.max(np.abs(Z - z)) <= 1e-4 * np.max(np.abs(z))
