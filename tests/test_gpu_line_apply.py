"""The line form of the solver's apply (at least 112 σ-lines per chunk, orders up to 9) and its neighbour, the
node-by-node form, against the oracle's banded solve: chunks at, below and above the limit, several
passes with a short last one (SEM_GRID_LIMIT=1), one to four layers, both precisions, both ends.
Tolerances as for the other solves: 1e-10 (FP64, residual 1e-13), 1e-8 (mixed).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from oracle import sem as osem  # noqa: E402
from sem_workloads import small_case, initial_state  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def T(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("P,Nx,Nz,periodic", [
    (6, 4, 4, True), (6, 8, 2, False), (6, 7, 2, False), (3, 28, 1, True), (3, 27, 1, False), (4, 23, 1, True),
    (5, 37, 3, False), (9, 6, 2, True), (9, 5, 2, False), (10, 11, 1, True), (8, 13, 2, True), (7, 40, 4, False)])
def test_step_on_one_cta(P, Nx, Nz, periodic, precision, monkeypatch):
    monkeypatch.setenv("SEM_GRID_LIMIT", "1")
    wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic, H_over_L=0.02)
    om = osem.mesh_for(wl)
    m = sem.Mesh.from_workload(wl, h=om.h, precision=precision, tol=1e-13 if precision == "fp64" else 1e-12)
    if periodic:
        eta, phis = initial_state(wl, om.xcol, om.h)
    else:
        eta = 0.03 * np.cos(om.xcol / 2) + 0.01
        phis = 0.1 * np.cos(om.xcol / 2) + 0.02 * np.cos(om.xcol)
    ref = om.laplace_solve(eta, phis)
    Phi = torch.zeros(om.n, dtype=torch.float64, device=DEV)
    b = sem.Batch([m])
    b.laplace_solve([T(eta)], [T(phis)], [Phi])
    err = np.linalg.norm(Phi.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < (1e-10 if precision == "fp64" else 1e-8)
    # the mesh's own launch (all columns in one pass, cached factors)
    dt = 0.2 * wl.dt
    e2, p2 = T(eta), T(phis)
    m.rk4_step(e2, p2, dt, 1)
    er, pr = om.rk4_step(eta, phis, dt)
    tol = 1e-10 if precision == "fp64" else 1e-8
    assert np.linalg.norm(e2.cpu().numpy() - er) / np.linalg.norm(er) < tol
    assert np.linalg.norm(p2.cpu().numpy() - pr) / np.linalg.norm(pr) < tol
