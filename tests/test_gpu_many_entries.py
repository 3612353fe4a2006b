"""Sign vectors of more than 512 entries (two words per lane in the neuron loop):
float64 and inline pairing against the oracle, in both executions.  (Mixed
precision with fingerprints at this size is in the filter audit.)"""
import numpy as np
import pytest

import oracle
from paper_2306_07212_gb300 import workloads as wl
from _util import assert_same_complex, unpack_codes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[[2] + [52] * 10 + [1], [3, 250, 255, 20, 1]], ids=["2d", "3d"])
def case(request):
    widths = request.param
    net = wl.he_normal_mlp(widths, seed=2).rounded_to_fp32()
    box = wl.Box.cube(widths[0], 0.4 if widths[0] == 2 else 0.012)
    assert 2 * widths[0] + net.n_neurons > 512
    ref = oracle.extract(net, box)
    assert ref.status == 0
    return net, box, ref


@pytest.mark.parametrize("kw", [{"precision": "fp64"}, {"precision": "fp64", "pairing": "inline"},
                                {"precision": "mixed", "pairing": "inline"},
                                {"precision": "fp64", "pairing": "inline", "execution": "stepwise"}],
                         ids=["fp64", "fp64-inline", "mixed-inline", "fp64-inline-stepwise"])
def test_more_than_512_entries(case, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net, box, ref = case
    with Extractor(**kw) as ex:
        ex.extract(net, box)
        got = ex.vertices(), unpack_codes(ex.sign_words(), ex.counts()["P"]), ex.edges()
    tol = 1e-6 * float(np.linalg.norm(box.hi - box.lo))
    assert_same_complex(got, (ref.X, ref.S, ref.E), coord_tol=tol, what=str(kw))
