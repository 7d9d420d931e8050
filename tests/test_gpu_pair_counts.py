"""The pairs the density and force passes count, against the exact neighbour
lists at the h they return: equal in FP64, and in mixed precision between the
lists at h (1 - 2e-6) and h (1 + 2e-6), which brackets the FP32 rounding of
r / h (offset, shift, their difference, the three squares and their sum, the
product with 1 / h: under 1e-6 together; coordinates of a leaf's size, as the
staged ones are).  A pair lost by a node test or a candidate test shows here,
where its share of rho or a would not."""
import numpy as np
import pytest

from paper_1709_04488_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_04488_gb300 import build as b
    b.build()
    from paper_1709_04488_gb300 import sph
    return sph


@pytest.mark.parametrize("shift", [0.0, 7.0, -300.0])
@pytest.mark.parametrize("kind", ["periodic", "thin", "isolated", "m6"])
@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_counts_match_the_lists(S, shift, kind, lanes, prec):
    if prec == "fp64" and lanes not in (2, 4):
        pytest.skip("the FP64 kernels run two or four lanes")
    if kind == "thin":
        a, p = ics.sod(left=(96, 12, 12), right=(48, 6, 6), length=0.75, width=0.09375, jitter=0.05)
    elif kind == "isolated":
        a, p = ics.cloud(3000, seed=9)
    else:
        a, p = ics.lattice(14, seed=9)
    kw = {}
    if kind == "m6":
        kw = dict(kernel=1, eta=1.0)
        a["h"] = a["h"] / 1.2
    for c in "xyz":
        a[c] = a[c] + shift
    p = dict(p)
    if p["periodic"]:
        p["box_lo"] = tuple(v + shift for v in p["box_lo"])
    prob = S.Problem(a, S.make_params(S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED, **p, lanes_per_particle=lanes, **kw))
    prob.density_h()
    prob.forces()
    d = prob.diagnostics()
    h = prob.numpy("h")["h"]
    e = 0.0 if prec == "fp64" else 2e-6
    n = len(h)
    for k, got in ((0, round(d.ngb_mean * n)), (1, d.force_pairs)):
        few, many = (len(prob.neighbours(k, h=h * (1 + s * e))[1]) for s in (-1, 1))
        assert few <= got <= many, (k, few, got, many)
        assert many - few < 1e-3 * many
    prob.close()
