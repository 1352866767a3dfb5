"""A batch's Laplace solves on a plan of their own, beside its steps.

Solves take larger teams than steps (half the share of work per CTA).  Forced cluster plans with shares at which the
two differ, and the planner's own choice: solves and steps in turn on one batch, solves twice (the plan is made by
the first), against each tank's own solve and step, 1e-10 as for the other batch tests (solves to 1e-13).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from sem_workloads import c3_instances, initial_state  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


@pytest.mark.parametrize("count,tune", [(24, dict(plan=1, cluster_share=2.0)), (24, dict(plan=1, cluster_share=0.25)),
                                        (24, dict(plan=0)), (100, dict())])
def test_solves_beside_steps(count, tune):
    wls = c3_instances(count, seed=4)
    meshes, state = [], []
    for wl in wls:
        x, h = np.linspace(0.0, wl.length, wl.ncol, endpoint=False), np.full(wl.ncol, wl.depth)
        meshes.append(sem.Mesh.from_workload(wl, h=h))
        state.append([torch.tensor(v, device=DEV) for v in initial_state(wl, x, h)])
    etas, phis = [s[0].clone() for s in state], [s[1].clone() for s in state]
    Phis = [torch.zeros(m.n, dtype=torch.float64, device=DEV) for m in meshes]
    try:
        sem.set_batch_tuning(reset=True, **tune)
        b = sem.Batch(meshes, tuned=False)
        b.laplace_solve(etas, phis, Phis)
        b.rk4_step(etas, phis, [wl.dt for wl in wls], 1)
        first = [p.clone() for p in Phis]
        for p in Phis:
            p.zero_()
        b.laplace_solve([s[0] for s in state], [s[1] for s in state], Phis)
        assert all(torch.equal(p, q) for p, q in zip(Phis, first)) and not any(b.status())
        b.close()
    finally:
        sem.set_batch_tuning(reset=True)
    for i in range(0, count, max(1, count // 12)):
        m = sem.Mesh.from_workload(wls[i], h=np.full(wls[i].ncol, wls[i].depth))
        e, p = (v.clone() for v in state[i])
        want = torch.zeros_like(Phis[i])
        m.update_geometry(e)
        m.laplace_solve(p, want)
        assert rel(Phis[i], want) < 1e-10
        m.rk4_step(e, p, wls[i].dt, 1)
        assert rel(etas[i], e) < 1e-10 and rel(phis[i], p) < 1e-10
