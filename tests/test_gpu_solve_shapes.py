"""The stand-alone FP64 solve with two CTAs per SM, where its rule takes it, against the batched solve.

Between one and two element columns per SM; long tanks that the fused launch's shape would work through in several
passes, the last of them ragged, order 12 with 16 layers among them.  The same tank solved as a batch of one (the
stage kernel's own build and teams) is the reference: both meet 1e-13, so 1e-10 apart as in the other solves.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from sem_workloads import small_case, initial_state  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("P,Nx,Nz,periodic", [(6, 160, 8, False), (8, 194, 16, True), (12, 303, 4, True), (8, 304, 8, False),
                                              (6, 5333, 4, True), (6, 5333, 4, False), (12, 460, 16, True)])
def test_two_ctas_per_sm(P, Nx, Nz, periodic):
    wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic)
    wl.length = 2 * np.pi * max(1, Nx // 64)
    x = np.linspace(0.0, wl.length, wl.ncol, endpoint=not periodic)
    m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol))
    assert m.info.grid_ctas > m.info.stage_ctas      # the rule took the wide launch
    eta, phis = (torch.tensor(v, device=DEV) for v in initial_state(wl, x, np.ones(wl.ncol)))
    a, b = (torch.zeros(m.n, dtype=torch.float64, device=DEV) for _ in range(2))
    m.update_geometry(eta)
    assert m.laplace_solve(phis, a).rel_residual <= 1e-13
    sem.Batch([m]).laplace_solve([eta], [phis], [b])
    assert float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) < 1e-10
