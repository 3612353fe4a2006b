"""Pruned extraction in mixed precision gives float64's pruned complex: the signs
of future neurons are those at the exact vertices.  The torus net on the box of
its workload, jittered or cut, where signs taken at the float32-accurate
coordinates dropped an edge that a later neuron crosses (PC_ERR_PAIRING) for
four boxes in ten; the whole extraction in stepwise execution too, and with
inline pairing."""
import numpy as np
import pytest

from paper_2306_07212_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _box(k):
    _, box = wl.torus_d3()
    if k == "cut":
        return wl.Box(0.7 * box.lo, 0.7 * box.hi)
    return wl.Box(box.lo + np.random.default_rng(k).uniform(-.02, .02, 3),
                  box.hi + np.random.default_rng(100 + k).uniform(-.02, .02, 3))


@pytest.mark.parametrize("k,kw", [(3, {}), (4, {}), (5, {"execution": "stepwise"}), (6, {"pairing": "inline"}), ("cut", {})])
def test_same_complex_as_float64(k, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net, box = wl.torus_d3()[0], _box(k)
    got = []
    for precision, more in (("fp64", {}), ("mixed", kw)):
        with Extractor(precision=precision, prune=True, canonical=True, **more) as ex:
            ex.extract(net, box)
            got.append((ex.sign_words(), ex.edges(), ex.vertices()))
    (S, E, X), (Sm, Em, Xm) = got
    assert np.array_equal(S, Sm) and np.array_equal(E, Em)
    assert np.max(np.abs(X - Xm)) <= 1e-6 * float(np.linalg.norm(box.hi - box.lo))
