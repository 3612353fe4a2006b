"""Canonical order at the sizes where its sort takes another path: ranks by
direct counting up to 16384 vertices, radix levels above, one or several
levels by how long equal prefixes are; D = 1 (one word, two edges per
vertex) and more facets and neurons than one level's key holds.  The sorted
arrays must be the unsorted extraction's, put in order by numpy."""
import numpy as np
import pytest

from paper_2306_07212_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (net, vertices): below and above 16384, long equal prefixes, several words
NETS = [([1, 8, 8, 1], "he"), ([2, 40, 40, 40, 1], "he"), ([2, 64, 64, 64, 1], "he"), ([2, 128, 128, 1], "he"),
        ([2, 128, 128, 128, 1], "he"), ([3, 24, 24, 1], "he"), ([3, 32, 32, 32, 1], "he"),
        ([5, 20, 20, 20, 20, 1], "uniform"), ([8, 10, 10, 10, 10, 1], "uniform"), ([4, 9, 7, 11, 2], "he")]


@pytest.mark.parametrize("widths,init", NETS)
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_sorted_arrays_equal_the_unsorted_ones_in_order(widths, init, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2306_07212_gb300 import Extractor
    net = (wl.he_normal_mlp if init == "he" else wl.default_uniform_mlp)(widths, seed=3)
    box = wl.Box.cube(widths[0])
    with Extractor(precision=precision) as ex:
        ex.extract(net, box)
        X0, W0, E0, Z0 = ex.vertices(), ex.sign_words(), ex.edges().astype(np.int64), ex.values()
    with Extractor(precision=precision, canonical=True) as ex:
        ex.extract(net, box)
        X, W, E, Z = ex.vertices(), ex.sign_words(), ex.edges(), ex.values()
    perm = np.lexsort(W0[::-1])  # word 0 most significant
    rank = np.empty(len(perm), np.int64)
    rank[perm] = np.arange(len(perm))
    assert np.array_equal(W, W0[:, perm])
    assert np.array_equal(X, X0[perm]) and np.array_equal(Z, Z0[perm])
    e = np.sort(rank[E0], axis=1)
    assert np.array_equal(E, e[np.lexsort((e[:, 1], e[:, 0]))])
