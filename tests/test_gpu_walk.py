"""The tree walk's node tests where the coordinates are large against the
smoothing lengths (the quick test's band grows with them and the definition
decides more leaves): a problem moved away from the origin has the same
neighbours, so its density and forces are those of the unmoved one.

Moving by s rounds every coordinate to 2^-53 s, which the FP32 pair terms do
not see for the s here (s 2^-53 < 2^-24 x spacing); tolerances are those of
the parity tests (rho 1e-5 relative, a 1e-4 of rms |a|; FP64 path: positions
rounded to 2^-53 s against h ~ 0.1 move rho by up to 1e-11)."""
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


def _eval(S, a, p, prec, **kw):
    prob = S.Problem(a, S.make_params(prec, **p, **kw))
    prob.density_h()
    prob.forces()
    g = prob.numpy()
    d = prob.diagnostics()
    prob.close()
    return g, d


@pytest.mark.parametrize("shift", [7.0, -300.0])
@pytest.mark.parametrize("kind", ["periodic", "thin", "isolated", "m6"])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_moved_problem_has_the_same_neighbours(S, shift, kind, prec):
    if kind == "thin":
        a, p = ics.sod(left=(96, 12, 12), right=(48, 6, 6), length=0.75, width=0.09375, jitter=0.05)
    elif kind == "isolated":
        a, p = ics.cloud(3000, seed=9)
    else:
        a, p = ics.lattice(14, seed=9)
    rng = np.random.default_rng(3)
    for c in ("vx", "vy", "vz"):
        a[c] = rng.normal(0.0, 0.3, len(a["x"]))
    kw = {}
    if kind == "m6":
        kw = dict(kernel=1, eta=1.0)
        a["h"] = a["h"] / 1.2
    pr = S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED
    g0, d0 = _eval(S, a, p, pr, **kw)
    b = dict(a)
    for c in "xyz":
        b[c] = a[c] + shift
    q = dict(p)
    if p["periodic"]:
        q["box_lo"] = tuple(v + shift for v in p["box_lo"])
    g1, d1 = _eval(S, b, q, pr, **kw)
    tol, atol = (1e-5, 1e-4) if prec == "mixed" else (1e-10, 1e-9)
    assert np.max(np.abs(g1["rho"] / g0["rho"] - 1.0)) < tol
    assert np.max(np.abs(g1["h"] / g0["h"] - 1.0)) < tol
    a0 = np.stack([g0[k] for k in ("ax", "ay", "az")], 1)
    a1 = np.stack([g1[k] for k in ("ax", "ay", "az")], 1)
    assert np.max(np.linalg.norm(a1 - a0, axis=1)) < atol * np.sqrt(np.mean(np.sum(a0 ** 2, 1)))
    assert (d1.ngb_min, d1.ngb_max) == (d0.ngb_min, d0.ngb_max) or prec == "mixed"
