"""The neighbour lists against brute force over every pair (the same rounding:
differences, minimum image and r^2 in FP64 without fused multiply-add): whole
numbers, identical.  Lanes per particle, both staging precisions, thin and
wide-support boxes, far-off coordinates, unequal h, sizes around a leaf, and a
capacity that cuts a particle's list."""
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


def _brute(a, p, h, kind, kr):
    n = len(a["x"])
    r2 = np.zeros((n, n))
    for c, L in zip("xyz", p["box_len"]):
        d = a[c][:, None] - a[c][None]
        if p["periodic"]:
            d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
        r2 += d * d
    R = kr * (np.maximum(h[:, None], h[None]) if kind else h[:, None])
    near = r2 < R * R
    if kind:
        np.fill_diagonal(near, False)
    off = np.concatenate([[0], np.cumsum(near.sum(1))])
    return off, np.nonzero(near)[1]


def _case(kind):
    rng = np.random.default_rng(len(kind))
    kr = 2.0
    if kind == "thin":  # support near half the box, wide leaves
        a, p = ics.sod(left=(96, 12, 12), right=(48, 6, 6), length=0.75, width=0.09375, jitter=0.05)
        sel = np.sort(rng.choice(len(a["x"]), 2500, replace=False))
        a = {k: v[sel] for k, v in a.items()}
        h = a["h"] * 1.2
    elif kind == "m6":
        a, p = ics.lattice(12, seed=5)
        h, kr = a["h"] / 1.2, 3.0
    elif kind == "far":  # coordinates large against h
        a, p = ics.cloud(2000, seed=6)
        for c in "xyz":
            a[c] = a[c] + 500.0
        h = a["h"]
    elif kind == "spread":  # h over a factor of eight, random points
        a, p = ics.random_cloud(2111, 7)
        h = a["h"] * np.exp(rng.uniform(np.log(0.25), np.log(2.0), 2111))
        h = np.minimum(h, 0.24)
    else:
        a, p = ics.random_cloud(int(kind), 8, periodic=False)
        h = a["h"]
    return a, p, h, kr


@pytest.mark.parametrize("kind", ["thin", "m6", "far", "spread", "1", "31", "33", "65"])
@pytest.mark.parametrize("lanes", [1, 2, 8])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_lists_match_brute_force(S, kind, lanes, prec):
    a, p, h, kr = _case(kind)
    kw = dict(kernel=1) if kind == "m6" else {}
    prob = S.Problem(a, S.make_params(S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED, **p, lanes_per_particle=lanes, **kw))
    for k in (0, 1):
        off, idx = prob.neighbours(k, h=h)
        off_r, idx_r = _brute(a, p, h, k, kr)
        assert np.array_equal(off.cpu().numpy(), off_r)
        assert np.array_equal(idx.cpu().numpy(), idx_r)
    prob.close()


@pytest.mark.parametrize("cut", [0, 1, 7, 500, -1])
def test_capacity_cuts_a_list(S, cut):
    """A short index array receives the first cap entries, in order, and the
    call says how many there are."""
    import torch
    a, p, h, kr = _case("spread")
    prob = S.Problem(a, S.make_params(S.PREC_MIXED, **p))
    off_r, idx_r = _brute(a, p, h, 1, kr)
    cap = cut if cut >= 0 else len(idx_r) + cut
    ht = torch.as_tensor(h, device="cuda")
    off = torch.zeros(len(h) + 1, dtype=torch.int64, device="cuda")
    idx = torch.full((cap + 8,), -7, dtype=torch.int32, device="cuda")
    rc, tot = S.sph_neighbours(prob.ctx, 1, ht.data_ptr(), off.data_ptr(), idx.data_ptr(), cap)
    assert rc == S.ENOSPACE and tot == len(idx_r)
    got = idx.cpu().numpy()
    assert np.array_equal(got[:cap], idx_r[:cap])
    assert np.all(got[cap:] == -7)
    prob.close()
