"""Stepwise extraction without a server: a layer runs as one cluster while few
vertices are expected, else as a launch per step and neuron over the whole GPU
(a cluster is 8 or 16 of its 152 SMs: a 4-12x4-1 net took twice as long in
one).  Both forms give the persistent extraction's complex, and a context keeps
to the rule after a larger network has grown it."""
import pytest

from paper_2306_07212_gb300 import workloads as wl
from _util import assert_same_complex, unpack_codes

pytestmark = pytest.mark.gpu


def _triple(ex):
    return ex.vertices(), unpack_codes(ex.sign_words(), ex.counts()["P"]), ex.edges()


def _launches(ex, net, box):
    ex.extract(net, box)  # grows what it needs
    before = ex.diagnostics()["launches"]
    ex.extract(net, box)
    return ex.diagnostics()["launches"] - before


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_form_follows_the_size(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    small, large = [2] + [24] * 4 + [1], [4] + [12] * 4 + [1]  # 3.7e3 and 2.1e5 vertices
    with Extractor(precision=precision, execution="stepwise") as ex:
        for widths, cluster in ((small, True), (large, False), (small, True)):
            net, box = wl.he_normal_mlp(widths, seed=1).rounded_to_fp32(), wl.Box.cube(widths[0])
            n = _launches(ex, net, box)
            assert (n < net.n_neurons) == cluster, (widths, n, net.n_neurons)
            got = _triple(ex)
            with Extractor(precision=precision) as other:
                other.extract(net, box)
                assert_same_complex(got, _triple(other), coord_tol=1e-12, what=f"{widths} {precision}")
