"""Sort and leaf tiles on both sides of the sizes at which their width changes
(two, four or eight keys and one or two particles per thread; lanes of the FP64
kernels): the neighbour lists of every particle, which need every particle in
exactly one leaf, against a k-d tree of the same points.  Whole numbers,
identical; no pair of these points lies within rounding of the radius."""
import numpy as np
import pytest

from paper_1709_04488_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [(8000, "fp64"), (8001, "fp64"), (65536, "mixed"), (65537, "mixed"),
                                    (131072, "mixed"), (131073, "mixed"), (196608, "mixed"), (196609, "mixed")])
def test_lists_at_the_edges_of_the_tile_sizes(n, prec):
    spatial = pytest.importorskip("scipy.spatial")
    from paper_1709_04488_gb300 import sph as S
    a, p = ics.random_cloud(n, n % 97, periodic=False)
    h = np.full(n, 0.6 / n ** (1 / 3))
    R = 2.0 * h[0]
    x = np.stack([a[c] for c in "xyz"], 1)
    i, j = spatial.cKDTree(x).query_pairs(R * (1 + 1e-12), output_type="ndarray").T
    r = np.sqrt(((x[i] - x[j]) ** 2).sum(1))
    assert np.abs(r / R - 1).min() > 1e-14
    i, j = np.concatenate([i, j]), np.concatenate([j, i])
    order = np.lexsort((j, i))
    off_r = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=n))])
    prob = S.Problem(a, S.make_params(S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED, **p))
    off, idx = prob.neighbours(1, h=h)
    assert np.array_equal(off.cpu().numpy(), off_r)
    assert np.array_equal(idx.cpu().numpy(), j[order])
    prob.close()
