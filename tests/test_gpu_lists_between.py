"""sph_neighbours between other calls of a context: what follows it is what
follows without it."""
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


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("kind", ["lattice", "cloud"])
def test_slow_path_of_a_step_that_keeps_the_leaves(S, kind, prec):
    """Particles of the slow density path look up their leaf, which the
    lists' counts must not replace.  (Sums over other leaves differ by
    rounding: 1e-5 relative in mixed precision, 1e-10 in FP64.)"""
    import torch
    a, p = ics.lattice(12, seed=5) if kind == "lattice" else ics.cloud(1800, seed=6)
    pr = S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED
    got = []
    for lists in (False, True):
        prob = S.Problem(a, S.make_params(pr, **p, tree_rebuild_every=4))
        prob.density_h()
        prob.forces()
        prob.step(1e-4)
        if lists:
            prob.neighbours(1)
        prob.t["h"].mul_(1.6)  # first guesses that overflow the lists
        torch.cuda.synchronize()
        prob.step(1e-4)
        assert prob.diagnostics().fallback > 100
        got.append(prob.numpy("h", "rho"))
        prob.close()
    for f in ("h", "rho"):
        assert np.max(np.abs(got[1][f] / got[0][f] - 1.0)) < (1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("kind", ["lattice", "cloud"])
@pytest.mark.parametrize("h", [None, 0.3, 1.2])
@pytest.mark.parametrize("after", ["density", "short guess", "kept step"])
def test_forces_after_lists(S, kind, prec, h, after):
    """A force pass after the lists sees the boxes of the state's h, the order
    of what the density pass staged, and no recorded groups that do not cover
    its h: the same bits as without the lists."""
    a, p = ics.lattice(12, seed=5) if kind == "lattice" else ics.cloud(1800, seed=6)
    if after == "short guess":  # (h grows beyond the recorded groups)
        a["h"] = a["h"] * 0.7
    pr = S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED
    got = []
    for lists in (False, True):
        prob = S.Problem(a, S.make_params(pr, **p, tree_rebuild_every=4))
        prob.density_h()
        if after == "kept step":
            prob.forces()
            prob.step(2e-3)
            prob.step(2e-3)
        if lists:
            prob.neighbours(1, h=None if h is None else prob.numpy("h")["h"] * h)
        prob.forces()
        f0 = prob.numpy("ax", "ay", "az", "du", "vsig")
        prob.step(1e-3)
        got.append((f0, prob.numpy("x", "vx", "u", "h", "rho", "ax")))
        prob.close()
    for x, y in zip(*got):
        for f in x:
            assert np.array_equal(x[f], y[f]), f
