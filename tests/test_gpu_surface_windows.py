"""M' solves from a window of neighbouring elements (mass1d_window) against the oracle's banded solve.

Sizes where the windows can go wrong: rings shorter than the window (it wraps several times), tanks of
one to three elements between walls, one more or one less element than a block of the recovery kernel,
several segments per CTA (SEM_GRID_LIMIT=1), element widths that differ by a factor of 50, the
smallest and largest order.  Tolerance 1e-12 as for the other recovery tests: the window's truncation
is below 1e-18 relative by construction, rounding of a few hundred terms is what remains; times the
condition of the S_x rows (2/Δx), which the reference shares.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from oracle import sem as osem  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def tank(P, Nx, Nz, periodic, uneven):
    rng = np.random.default_rng(P * 100 + Nx)
    w = rng.uniform(1.0, 50.0 if uneven else 1.0, Nx) if uneven else np.ones(Nx)
    edges = np.concatenate([[0.0], np.cumsum(w)]) / w.sum() * 2 * np.pi
    edges[-1] = 2 * np.pi
    ncol = Nx * P if periodic else Nx * P + 1
    prm = osem.Params(Pf=(3 * P + 1) // 2, filter_alpha=36.0, filter_s=12.0, filter_ic=P - 1)
    om = osem.Mesh(P, Nx, Nz, edges, periodic, np.ones(ncol), prm)
    return om, edges, dict(Pf=prm.Pf, filter_alpha=36.0, filter_s=12.0, filter_ic=P - 1, periodic=periodic)


def T(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def rel(a, b):
    return np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)


@pytest.mark.parametrize("P,Nx,periodic,uneven", [
    (2, 3, True, False), (2, 90, True, True), (12, 3, True, True), (6, 16, True, False), (6, 17, True, True),
    (6, 1, False, False), (6, 3, False, True), (4, 15, False, True), (4, 33, False, False), (2, 200, False, True)])
def test_recovery_and_rhs(P, Nx, periodic, uneven, monkeypatch):
    om, edges, kw = tank(P, Nx, 1, periodic, uneven)
    x = om.xcol
    eta = 0.02 * np.cos(x) + 0.005 * np.cos(2 * x)
    phis = 0.05 * np.cos(x) + 0.02 * np.cos(3 * x)
    if periodic:
        phis = phis + 0.03 * np.sin(2 * x)
    ke, kp, parts = om.zakharov_rhs(eta, phis, return_parts=True)
    for limit in (None, "1"):
        if limit:
            monkeypatch.setenv("SEM_GRID_LIMIT", limit)
        m = sem.Mesh(P, Nx, 1, edges, om.h, **kw)
        outs = [torch.empty(om.ncol, dtype=torch.float64, device=DEV) for _ in range(3)]
        m.update_geometry(T(eta))
        m.recover_gradient(T(parts["Phi"]), T(eta), T(phis), *outs)
        for got, name in zip(outs, ("w", "etax", "phisx")):
            assert rel(got, parts[name]) < 1e-12, name
        de, dp = torch.empty_like(outs[0]), torch.empty_like(outs[0])
        m.zakharov_rhs(T(eta), T(phis), de, dp)
        assert rel(de, ke) < 1e-10 and rel(dp, kp) < 1e-10
        # the fused stage: one RK4 step (stable step on the narrowest element)
        dt = 0.02 * np.sqrt(np.diff(edges).min()) / P
        e2, p2 = T(eta), T(phis)
        m.rk4_step(e2, p2, dt, 1)
        er, pr = om.rk4_step(eta, phis, dt)
        assert rel(e2, er) < 1e-10 and rel(p2, pr) < 1e-10
