"""zakharov_rhs with relaxation zones and a generated signal: the fused stage without its update, against the oracle.

The left zone's signal comes from the tabulated columns (angle addition), the damping from the mesh's own
relax_tau, at times other than zero.  1e-10 as for the other right-hand sides (solves to 1e-13).
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


@pytest.mark.parametrize("fused", ["1", "0"])
@pytest.mark.parametrize("left,right", [(2.5, 3.0), (2.5, 0.0), (0.0, 3.0)])
def test_rhs_in_zones(left, right, fused, monkeypatch):
    monkeypatch.setenv("SEM_FUSED_STAGE", fused)
    P, Nx, Nz, L = 5, 24, 2, 12.0
    amp, omega = np.array([0.02, 0.01, 0.004]), np.array([2.6, 3.4, 5.1])
    k, phase = omega ** 2 / 9.81, np.array([0.3, 1.7, -0.6])
    edges = np.linspace(0.0, L, Nx + 1)
    h = np.ones(Nx * P + 1)
    prm = osem.Params(Pf=8, filter_alpha=36.0, filter_s=12.0, filter_ic=P - 1, relax_left=left, relax_right=right,
                      relax_tau=0.7, wave=(amp, omega, k, phase))
    om = osem.Mesh(P, Nx, Nz, edges, False, h, prm)
    gm = sem.Mesh(P, Nx, Nz, edges, h, periodic=False, Pf=8, filter_alpha=36.0, filter_s=12.0, filter_ic=P - 1,
                  relax_left=left, relax_right=right, relax_tau=0.7, wave=(amp, omega, k, phase))
    x = om.xcol
    eta, phis = 0.03 * np.cos(0.9 * x), 0.05 * np.sin(0.8 * x)
    de, dp = (torch.empty(om.ncol, dtype=torch.float64, device=DEV) for _ in range(2))
    for t in (0.0, 0.37, 11.3):
        gm.zakharov_rhs(torch.tensor(eta, device=DEV), torch.tensor(phis, device=DEV), de, dp, t=t)
        for got, ref in zip((de, dp), om.zakharov_rhs(eta, phis, t=t)):
            assert np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10
