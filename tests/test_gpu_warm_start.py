"""A solve that starts from its own solution takes no iteration and leaves it as it is.

The start's FP64 residual is tested against the tolerance itself (only the stages' extrapolated guesses ask
for more).  Tolerance 1e-9: far above the difference between a recurred and a computed FP64 residual (1e-15 of
‖A‖‖x‖, 1e-12 of ‖b‖ on these tanks), so every solution passes that test again, wherever below it the first
solve ended.
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


def tanks(precision):
    for P, Nx, Nz, periodic in ((2, 9, 1, True), (3, 40, 2, False), (4, 300, 1, True), (5, 17, 3, True), (6, 64, 4, False),
                                (7, 150, 1, True), (8, 33, 2, False), (12, 5, 1, True)):
        wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic)
        x = np.linspace(0.0, wl.length, wl.ncol, endpoint=not periodic)
        m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol), precision=precision, tol=1e-9)
        eta, phis = (torch.tensor(v, device=DEV) for v in initial_state(wl, x, np.ones(wl.ncol)))
        yield m, eta, phis, torch.zeros(m.n, dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solution_as_start(precision):
    ms, es, ps, Ps = zip(*tanks(precision))
    for m, eta, phis, Phi in zip(ms, es, ps, Ps):
        m.update_geometry(eta)
        assert m.laplace_solve(phis, Phi).iterations > 0
        first = Phi.clone()
        assert m.laplace_solve(phis, Phi).iterations == 0
        assert torch.equal(first, Phi)
        m.reset_counters()
    first = [Phi.clone() for Phi in Ps]
    sem.Batch(ms).laplace_solve(list(es), list(ps), list(Ps))
    for m, a, b in zip(ms, first, Ps):
        assert m.counters().iterations == 0 and torch.equal(a, b)
