"""A trajectory whose state the caller changes a little between calls keeps the history of stages 2 to 4.

Steps of one tank, one call each, on four meshes: the state untouched, changed after every call by a given
share of its largest value (alternating in sign, the worst case for an extrapolation), and with a dt that alternates
by a rounding, which starts a new history at every call.  From the sixth step on, when the history is full:

* a change of 1e-9 costs at most the extrapolation of stage 1, four iterations a step, and saves at
  least one iteration in each of the three other stages and one more against starting anew (their guesses are
  nearer by two decades or more, an iteration's worth being about two);
* a change of 1e-3 (15e-3 of an increment after a cubic extrapolation) takes no more than starting anew;
* the results are the oracle's, changed likewise (1e-10: solves to 1e-13).
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
STEPS, FIRST = 9, 5


def T(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("limit", [None, "1"])
def test_small_changes_keep_the_stages_history(limit, monkeypatch):
    if limit:
        monkeypatch.setenv("SEM_GRID_LIMIT", limit)
    wl = small_case(P=5, Nx=11, Nz=2, H_over_L=0.02)
    om = osem.mesh_for(wl)
    e0, p0 = initial_state(wl, om.xcol, om.h)
    bump = np.sin(2 * np.pi * om.xcol / wl.length + 0.4)

    def run(share, anew=False):
        m = sem.Mesh.from_workload(wl, h=om.h)
        e, p, its = T(e0), T(p0), []
        for k in range(STEPS):
            m.reset_counters()
            m.rk4_step(e, p, wl.dt * (1 + 1e-14 * (k % 2)) if anew else wl.dt, 1)
            its.append(m.counters().iterations)
            e += T((-1) ** k * share * np.abs(e0).max() * bump)
            p += T((-1) ** k * share * np.abs(p0).max() * bump)
        return e, p, sum(its[FIRST:])

    n = STEPS - FIRST
    _, _, untouched = run(0.0)
    _, _, anew = run(0.0, anew=True)
    for share in (1e-9, 1e-3):
        e, p, its = run(share)
        if share == 1e-9:
            assert its <= untouched + 4 * n and its <= anew - 4 * n, (untouched, its, anew)
        else:
            assert its <= anew, (its, anew)
        er, pr = e0, p0
        for k in range(STEPS):
            er, pr = om.rk4_step(er, pr, wl.dt)
            er = er + (-1) ** k * share * np.abs(e0).max() * bump
            pr = pr + (-1) ** k * share * np.abs(p0).max() * bump
        for got, ref in ((e, er), (p, pr)):
            assert np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10
