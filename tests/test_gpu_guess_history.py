"""The trajectory of the initial guesses is recognised by the state's values, not by its buffers.

* the same trajectory moved to other buffers between calls takes the iterations of one that stayed;
* another state in the same buffers takes those of a fresh mesh (one more or less for rounding);
* a mesh stepped alone, then in a batch, then alone again keeps its history, on several CTAs and one;
* the results match the oracle throughout (1e-10: solves to 1e-13).
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


def setup(Nx=9, steep=0.02):
    wl = small_case(P=5, Nx=Nx, Nz=2, H_over_L=steep)
    om = osem.mesh_for(wl)
    e, p = initial_state(wl, om.xcol, om.h)
    return wl, om, sem.Mesh.from_workload(wl, h=om.h), e, p


def iterations(m, call):
    m.reset_counters()
    call()
    return m.counters().iterations


def test_moved_buffers_continue_and_new_states_start_anew():
    wl, om, m, e0, p0 = setup()
    e, p = T(e0), T(p0)
    first = iterations(m, lambda: m.rk4_step(e, p, wl.dt, 1))
    m.rk4_step(e, p, wl.dt, 5)
    e2, p2 = e.clone(), p.clone()
    moved = iterations(m, lambda: m.rk4_step(e2, p2, wl.dt, 1))
    stayed = setup()
    es, ps = T(e0), T(p0)
    stayed[2].rk4_step(es, ps, wl.dt, 6)
    assert moved == iterations(stayed[2], lambda: stayed[2].rk4_step(es, ps, wl.dt, 1))
    assert torch.equal(e2, es) and torch.equal(p2, ps)
    assert moved < first
    # other values in the same buffers: a first step again, from the last potential instead of zero
    e2.copy_(T(-e0))
    p2.copy_(T(0.5 * p0))
    again = iterations(m, lambda: m.rk4_step(e2, p2, wl.dt, 1))
    assert again > moved
    er, pr = om.rk4_step(-e0, 0.5 * p0, wl.dt)
    for got, ref in ((e2, er), (p2, pr)):
        assert np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10


@pytest.mark.parametrize("limit", [None, "1"])
def test_alone_and_batched_share_the_history(limit, monkeypatch):
    if limit:
        monkeypatch.setenv("SEM_GRID_LIMIT", limit)
    wl, om, m, e0, p0 = setup(Nx=11)
    other = setup(Nx=11)[2]                       # the same steps, always alone
    e, p, eo, po = T(e0), T(p0), T(e0), T(p0)
    b = sem.Batch([m])
    for k in range(8):
        want = iterations(other, lambda: other.rk4_step(eo, po, wl.dt, 1))
        step = (lambda: b.rk4_step([e], [p], [wl.dt], 1)) if k % 3 == 2 else (lambda: m.rk4_step(e, p, wl.dt, 1))
        assert abs(iterations(m, step) - want) <= 4   # one per solve for the teams' summation order
    er, pr = e0, p0
    for _ in range(8):
        er, pr = om.rk4_step(er, pr, wl.dt)
    for got, ref in ((e, er), (p, pr)):
        assert np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-10
