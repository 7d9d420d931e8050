"""A problem in another unit of length: every length times 2^k, masses,
velocities and internal energies as they are.  A power of two rounds nothing,
so each output of an FP64 problem is the unscaled one times its power of two,
bit for bit, and the neighbour lists are the same lists.  (Squares of the
lengths leave the range of FP32 at k = 70 and k = -80: 1.2e21 and 8e-25.)"""
import numpy as np
import pytest

from paper_1709_04488_gb300 import ics

pytestmark = pytest.mark.gpu

POWER = dict(x=1, y=1, z=1, vx=0, vy=0, vz=0, u=0, m=0, h=1, rho=-3, omega=0, P=-3, c=0, ax=-1, ay=-1, az=-1, du=-1, vsig=0)


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_04488_gb300 import build as b
    b.build()
    from paper_1709_04488_gb300 import sph
    return sph


def _problem(kind):
    kw = {}
    if kind == "thin":
        a, p = ics.sod(left=(96, 12, 12), right=(48, 6, 6), length=0.75, width=0.09375, jitter=0.05)
    elif kind == "isolated":
        a, p = ics.cloud(2000, seed=6)
        a["m"] = a["m"] * np.random.default_rng(1).uniform(0.9, 1.1, 2000)
    else:
        a, p = ics.lattice(12, seed=5)
    if kind == "m6":
        kw = dict(kernel=1, eta=1.0)
        a["h"] = a["h"] / 1.2
    if kind == "slow":  # first guesses that overflow the lists: the slow density path
        a["h"] = a["h"] * 1.6
    if kind == "block":
        kw = dict(block_levels=2)
    rng = np.random.default_rng(3)
    for c in ("vx", "vy", "vz"):
        a[c] = rng.normal(0.0, 0.3, len(a["x"]))
    return a, p, kw


def _scaled(a, p, s):
    a, q = dict(a), dict(p)
    for c in "xyzh":
        a[c] = a[c] * s
    if p["periodic"]:
        q["box_lo"] = tuple(v * s for v in p["box_lo"])
        q["box_len"] = tuple(v * s for v in p["box_len"])
    return a, q


@pytest.mark.parametrize("k", [70, -80])
@pytest.mark.parametrize("kind", ["lattice", "thin", "isolated", "m6", "slow", "block"])
def test_fp64_outputs_scale_exactly(S, kind, k):
    a, p, kw = _problem(kind)
    out = []
    for s in (1.0, 2.0 ** k):
        b, q = _scaled(a, p, s)
        prob = S.Problem(b, S.make_params(S.PREC_FP64, **q, tree_rebuild_every=2, **kw))
        prob.density_h()
        prob.forces()
        got = [prob.numpy(*POWER)]
        if kind == "block":
            prob.block_step()
        else:
            for _ in range(3):  # (leaves kept and built)
                prob.step()
        got.append(prob.numpy(*POWER))
        d = prob.diagnostics()
        out.append((got, d.ngb_min, d.ngb_max, d.force_pairs))
        prob.close()
    for g0, g1 in zip(out[0][0], out[1][0]):
        for f, w in POWER.items():
            assert np.array_equal(g1[f], np.ldexp(g0[f], w * k)), f
    assert out[0][1:] == out[1][1:]


@pytest.mark.parametrize("k", [70, -80])
@pytest.mark.parametrize("kind", ["lattice", "thin", "isolated", "m6"])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_lists_do_not_depend_on_the_unit(S, kind, k, prec):
    a, p, kw = _problem(kind)
    lists = []
    for s in (1.0, 2.0 ** k):
        b, q = _scaled(a, p, s)
        prob = S.Problem(b, S.make_params(S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED, **q, **kw))
        lists.append([t.cpu().numpy() for n in (0, 1) for t in prob.neighbours(n)])
        prob.close()
    assert len(lists[0][1]) > 20 * len(a["x"])
    for x, y in zip(*lists):
        assert np.array_equal(x, y)


def test_far_clumps(S):
    """Two copies of a clump 2^18 of its sizes apart: the lists of each are
    the clump's, although the walk's boxes are as coarse as the domain."""
    a, p = ics.cloud(1500, seed=6)
    two = {k: np.concatenate([v, v]) for k, v in a.items()}
    two["x"][1500:] += 2.0 ** 18
    for prec in (S.PREC_FP64, S.PREC_MIXED):
        for kind in (0, 1):
            lists = []
            for b in (a, two):
                prob = S.Problem(b, S.make_params(prec, **p))
                lists.append([t.cpu().numpy() for t in prob.neighbours(kind, h=b["h"])])
                prob.close()
            (o1, i1), (o2, i2) = lists
            # (the moved copy's coordinates are rounded to 2^-35: its own
            # lists may differ in pairs at the radius, the first copy's not)
            assert np.array_equal(o2[:1501], o1) and np.array_equal(i2[:o1[-1]], i1)
            assert abs(int(o2[-1]) - 2 * int(o1[-1])) <= 4


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("periodic", [False, True])
def test_reach_out_of_the_domain_s_scale(S, prec, periodic):
    """Smoothing lengths whose squares leave the range of FP32 beside a domain
    of order one: every particle alone, or (isolated) every pair."""
    a, p = ics.random_cloud(900, 8, periodic=periodic)
    n = 900
    prob = S.Problem(a, S.make_params(S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED, **p))
    for h in (1e-22, 1e-30, 1e25):
        if h > 1 and periodic:
            continue
        for kind in (0, 1):
            off, idx = (t.cpu().numpy() for t in prob.neighbours(kind, h=np.full(n, h)))
            want = np.ones((n, n), bool) if h > 1 else np.eye(n, dtype=bool)
            if kind:
                np.fill_diagonal(want, False)
            assert np.array_equal(off, np.concatenate([[0], np.cumsum(want.sum(1))]))
            assert np.array_equal(idx, np.nonzero(want)[1])
    prob.close()


def test_far_clumps_take_no_longer(S):
    """The band of pairs that FP64 decides is the rounding of separations, not
    of the domain: the FP64 force pass of two clumps 2^18 of their sizes apart
    takes the time of two clumps 2^8 apart (best of five; 1.07 times; with a
    band of 1e-6 of the domain, wider than h, 5.7 times)."""
    import torch
    a, p = ics.cloud(1500, seed=6)
    best = []
    for e in (8, 18):
        b = {k: np.concatenate([v, v]) for k, v in a.items()}
        b["x"][1500:] += 2.0 ** e
        prob = S.Problem(b, S.make_params(S.PREC_FP64, **p))
        prob.density_h()
        prob.forces()
        t = []
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            prob.forces()
            t1.record()
            t1.synchronize()
            t.append(t0.elapsed_time(t1))
        best.append(min(t))
        prob.close()
    assert best[1] < 2.0 * best[0]


@pytest.mark.parametrize("kernel,lanes,over", [(0, 2, 1.2), (0, 4, 1.3), (1, 2, 1.1), (1, 4, 1.22)])
@pytest.mark.parametrize("equal", [True, False])
def test_a_first_guess_too_large_stays_in_the_lists(S, kernel, lanes, over, equal):
    """FP64 neighbour lists hold 128 and 160 entries a particle (M6 192 and
    256) at two and four lanes: 1.26, 1.36 (1.16, 1.27) times the solved h of
    a uniform problem.  Beyond that each particle takes the slow path."""
    a, p = ics.lattice(16, seed=3)
    a["h"] = a["h"] * over / (1.2 if kernel else 1.0)
    if not equal:
        a["m"] = a["m"] * np.random.default_rng(1).uniform(0.999, 1.001, len(a["m"]))
    kw = dict(kernel=1, eta=1.0) if kernel else {}
    prob = S.Problem(a, S.make_params(S.PREC_FP64, **p, lanes_per_particle=lanes, **kw))
    prob.density_h()
    assert prob.diagnostics().fallback == 0
    prob.close()
