"""Direct gravity's partial sums: a batch holds those of its split problems
only, and the ranges on both sides of the size to which they are limited by
the allocation-free call's fixed scratch (32768) give the direct sum."""
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


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_batch_pays_for_its_split_problems_only(S, prec):
    """One problem of 5000 particles with gravity among 60000 without: no more
    workspace than the contexts' own together, and the states of the contexts
    stepped alone."""
    import torch
    pr = S.PREC_FP64 if prec == "fp64" else S.PREC_MIXED
    parts = [(ics.lattice(31, seed=2), {}), (ics.cloud(5000, seed=3), dict(gravity=1, G=1.0)),
             (ics.lattice(31, seed=4), {}), (ics.cloud(700, seed=5), dict(gravity=1, G=2.0))]

    def contexts():
        out = []
        for (a, p), kw in parts:
            prob = S.Problem(a, S.make_params(pr, **p, **kw))
            prob.density_h()
            prob.forces()
            out.append(prob)
        return out

    alone, batched = contexts(), contexts()
    need = S.sph_batch_workspace_bytes([p.ctx for p in batched])
    assert need <= sum(p.ws_bytes for p in batched)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert S.sph_batch_step([p.ctx for p in batched], 2, ws.data_ptr(), need) == S.OK
    for p, q in zip(alone, batched):
        p.step()
        p.step()
        x, y = p.numpy(), q.numpy()
        for f in x:
            assert np.array_equal(x[f], y[f]), f
        p.close()
        q.close()


@pytest.mark.parametrize("n", [20001, 32768, 32769])
def test_ranges_around_the_fixed_scratch_limit(S, n):
    """Sampled particles against the sum over all partners in FP64 (terms and
    tolerance as derived in test_gpu_gravity_split.py)."""
    import torch
    a, p = ics.cloud(n, seed=n)
    for c in ("vx", "vy", "vz"):
        a[c][:] = 0.0
    acc = []
    for kw in (dict(gravity=1, G=1.0), {}):
        prob = S.Problem(a, S.make_params(S.PREC_MIXED, **p, **kw))
        prob.density_h()
        prob.forces()
        acc.append(torch.stack([prob.t[k][:n].clone() for k in ("ax", "ay", "az")], 1))
        t = prob.t
    x = torch.stack([t[k][:n] for k in "xyz"], 1)
    h, m, rho, om = (t[k][:n] for k in ("h", "m", "rho", "omega"))

    def mass(q):
        inner = 4 * (q ** 3 / 3 - 0.3 * q ** 5 + 0.125 * q ** 6)
        outer = 4 * (2 * q ** 3 / 3 - 0.75 * q ** 4 + 0.3 * q ** 5 - q ** 6 / 24 - 1 / 60)
        return torch.where(q < 1, inner, torch.where(q < 2, outer, torch.ones_like(q)))

    def grad(r, hh):
        q = r / hh
        return torch.where(q < 1, -3 * q + 2.25 * q ** 2, -0.75 * (2 - q).clamp(min=0) ** 2) / math.pi / hh ** 4

    zeta = torch.empty(n, dtype=torch.float64, device="cuda")
    for lo in range(0, n, 512):
        q = torch.cdist(x[lo:lo + 512], x, compute_mode="donot_use_mm_for_euclid_dist") / h[lo:lo + 512, None]
        qs = q.clamp(min=1e-12)
        psi = torch.where(q < 1, 2 * q ** 2 / 3 - 0.3 * q ** 4 + 0.1 * q ** 5 - 1.4,
                          torch.where(q < 2, 4 * q ** 2 / 3 - q ** 3 + 0.3 * q ** 4 - q ** 5 / 30 + 1 / (15 * qs) - 1.6, -1 / qs))
        zeta[lo:lo + 512] = ((psi + torch.where(q > 0, mass(q) / qs, torch.zeros_like(q))) * m[None]).sum(1)
    zo = zeta / (3 * rho * h) / om
    s = torch.as_tensor(np.sort(np.random.default_rng(1).choice(n, 400, replace=False)), device="cuda")
    d = x[s][:, None] - x[None]
    r = d.norm(dim=2)
    r[torch.arange(400, device="cuda"), s] = 1.0
    f = 0.5 * (mass(r / h[s][:, None]) + mass(r / h[None])) * m[None] / r ** 3
    f = f + 0.5 * m[None] * (zo[s][:, None] * grad(r, h[s][:, None]) + zo[None] * grad(r, h[None])) / r
    f[torch.arange(400, device="cuda"), s] = 0.0
    ref, mag = -(f[..., None] * d).sum(1), (f.abs() * r).sum(1)
    got = (acc[0] - acc[1])[s]
    tol = 1e-5 * (mag + acc[1].norm(dim=1).max())
    assert bool(((got - ref).norm(dim=1) < tol).all())
