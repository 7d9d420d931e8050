"""The direct gravity sum at the edges of its partner ranges (one range, the
first split, blocks and ranges with remainders, the most ranges), against the
same sum in FP64 over the same particles and smoothing lengths.

The density solve's h enters both sides.  A pair term has about ten FP32
roundings of 2^-24, so |delta a_i| <= 10 x 2^-24 sum_j |f_ij| <= 1e-6 sum_j
|f_ij|; positions are cast relative to the problem's corner (box side 2, ulp
2^-23 per coordinate), which moves r_ij by up to 2^-22 and a softened term,
which changes over h, by 2^-22 / h of itself: both are below 1e-5 of the sum of
magnitudes for the h > 0.05 of these clouds."""
import math

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


def _mass(q):
    inner = 4 * (q ** 3 / 3 - 0.3 * q ** 5 + 0.125 * q ** 6)
    outer = 4 * (2 * q ** 3 / 3 - 0.75 * q ** 4 + 0.3 * q ** 5 - q ** 6 / 24 - 1 / 60)
    return np.where(q < 1, inner, np.where(q < 2, outer, 1.0))


@pytest.mark.parametrize("n", [90, 255, 256, 257, 511, 513, 4097, 5000])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_direct_sum_ranges(S, n, prec):
    """The accelerations with gravity minus those without: the long range and
    the zeta term, both summed here from their definitions."""
    a, p = ics.cloud(n, seed=n)
    a["m"] = a["m"] * np.random.default_rng(n).uniform(0.5, 1.5, n)
    for c in ("vx", "vy", "vz"):
        a[c][:] = 0.0
    pr = S.PREC_MIXED if prec == "mixed" else S.PREC_FP64
    prob = S.Problem(a, S.make_params(pr, **p, gravity=1, G=1.0))
    prob.density_h()
    prob.forces()
    g = prob.numpy()
    base = S.Problem(a, S.make_params(pr, **p))
    base.density_h()
    base.forces()
    h0 = base.numpy()
    got = np.stack([g[k] - h0[k] for k in ("ax", "ay", "az")], 1)
    x = np.stack([g["x"], g["y"], g["z"]], 1)
    h, m, rho, om = g["h"], g["m"], g["rho"], g["omega"]
    d = x[:, None] - x[None]
    r = np.sqrt((d ** 2).sum(-1))
    np.fill_diagonal(r, 1.0)
    f = 0.5 * (_mass(r / h[:, None]) + _mass(r / h[None])) * m[None] / r ** 3
    np.fill_diagonal(f, 0.0)
    ref = -(f[..., None] * d).sum(1)
    mag = (f * r).sum(1)
    # the zeta term, from its definition
    q = np.sqrt((d ** 2).sum(-1)) / h[:, None]
    qs = np.maximum(q, 1e-12)
    psi = np.where(q < 1, 2 * q ** 2 / 3 - 0.3 * q ** 4 + 0.1 * q ** 5 - 1.4,
                   np.where(q < 2, 4 * q ** 2 / 3 - q ** 3 + 0.3 * q ** 4 - q ** 5 / 30 + 1 / (15 * qs) - 1.6, -1 / qs))
    zeta = ((psi + np.where(q > 0, _mass(q) / qs, 0.0)) * m[None]).sum(1) / (3 * rho * h)

    def grad(hh):
        t = r / hh
        return np.where(t < 1, -3 * t + 2.25 * t ** 2, -0.75 * np.clip(2 - t, 0, None) ** 2) / math.pi / hh ** 4

    zw = 0.5 * m[None] * ((zeta / om)[:, None] * grad(h[:, None]) + (zeta / om)[None] * grad(h[None])) / r
    np.fill_diagonal(zw, 0.0)
    ref -= (zw[..., None] * d).sum(1)
    mag += np.abs(zw * r).sum(1)
    # got is a difference of two force sums: their rounding too
    hyd = np.sqrt(sum(h0[k] ** 2 for k in ("ax", "ay", "az")))
    tol = (1e-5 if prec == "mixed" else 1e-12) * (mag + hyd.max())
    assert np.all(np.linalg.norm(got - ref, axis=1) < tol)
    prob.close()
    base.close()
