"""More intersecting edges than a generic input has: the appends stay inside
the edge capacity.

Step (5) pairs a 2-face at its second occurrence.  The capacity check of a
step counts two occurrences per 2-face (Section 4.2); a neuron whose values are
float32 rounding noise (a_1 - 3 a_2 of two units with a_2 = a_1 / 3) gives the
vertices of a 2-face alternating signs, so many 2-faces occur four times and
their later occurrences pair too: 11 % more edges than the check counts.  With
the capacity set to exactly what it asks for, these edges do not fit.  The
extraction must end in PC_ERR_PAIRING, and the context must stay usable.  The
noise neuron is followed by others of its layer, or is the last one."""
import numpy as np
import pytest

import oracle
from paper_2306_07212_gb300 import workloads as wl
from _util import assert_same_complex, unpack_codes

pytestmark = pytest.mark.gpu


def _first_layer():
    w = np.array([0.3, -0.2, 0.1])  # |w x| <= 0.6: units 0 and 1 stay active on the box
    base = wl.he_normal_mlp([3, 48, 1], seed=0).rounded_to_fp32()
    return np.vstack([w, w / 3, base.W[0]]), np.concatenate([[10.0, 10.0 / 3], base.b[0]])


def _pairs(codes, edges, m):
    """(2-faces' occurrences beyond the first, summed, split edges) for split edges between codes' rows."""
    p, q = edges[:, 0], edges[:, 1]
    faces = {}
    for row in np.where(codes[p] != 0, codes[p], codes[q]):
        for z in np.flatnonzero(row == 0):
            for sign in (1, -1) if z >= m else (1,):
                f = row.copy()
                f[z] = sign
                faces[f.tobytes()] = faces.get(f.tobytes(), 0) + 1
    return sum(k - 1 for k in faces.values())


@pytest.mark.parametrize("more", [3, 0])
def test_appends_stay_inside_the_edge_capacity(more):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    from paper_2306_07212_gb300.binding import PcError
    W1, b1 = _first_layer()
    box, n = wl.Box.cube(3), len(b1)
    with Extractor(precision="fp32", gemm="simt") as ex:
        ex.extract(wl.Net([3, n], [W1], [b1]), box)
        c, Z, E = ex.counts(), ex.values(), ex.edges()
        codes = unpack_codes(ex.sign_words(), c["P"])
    # the noise neuron's value as the product forms it: one rounding per input, the others' weights are 0
    z = (Z[:, 0].astype(np.float64) - 3.0 * Z[:, 1].astype(np.float64)).astype(np.float32)
    minus = z < 0
    cut = E[minus[E[:, 0]] != minus[E[:, 1]]]
    ecap = (c["nE"] + 3 * len(cut) + 63) // 64 * 64  # what the step asks for
    pairs = _pairs(codes, cut, 6)
    assert c["nE"] + len(cut) + pairs > ecap + 1000  # the input does what this test is about
    W2 = np.zeros((1 + more, n))
    W2[0, :2] = 1.0, -3.0
    b2 = np.zeros(1 + more)
    rng = np.random.default_rng(1)
    W2[1:, 2:] = rng.normal(0, 0.2, (more, n - 2))
    net = wl.Net([3, n, 1 + more], [W1, W2], [b1, b2])
    with Extractor(precision="fp32", gemm="simt", init_ecap=ecap) as ex:
        with pytest.raises(PcError) as err:
            ex.extract(net, box)
        assert err.value.status == 5, str(err.value)
        d = ex.diagnostics()
        assert d["ecap"] == ecap, d  # the step ran at this capacity
        ok, obox = wl.small_d2()
        ref = oracle.extract(ok, obox)
        ex.extract(ok, obox)
        got = (ex.vertices(), unpack_codes(ex.sign_words(), ex.counts()["P"]), ex.edges())
        assert_same_complex(got, (ref.X, ref.S, ref.E), coord_tol=1e-5, what="after")
