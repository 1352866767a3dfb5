"""Gradient recovery with outputs over its inputs, whole, crosswise and in part.

The recovery's blocks read the state around their own elements while others store, so the call has to
finish its results before they go over an input.  Several blocks (17, 40 and 100 elements of 16 a block); the result is
bit for bit that of separate arrays.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from sem_workloads import small_case, initial_state, random_field  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("Nx,periodic", [(17, True), (40, False), (100, True)])
def test_outputs_over_inputs(Nx, periodic):
    wl = small_case(P=5, Nx=Nx, Nz=2, periodic=periodic)
    x = np.linspace(0.0, wl.length, wl.ncol, endpoint=not periodic)
    m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol))
    e0, p0 = (torch.tensor(v, device=DEV) for v in initial_state(wl, x, np.ones(wl.ncol)))
    Phi0 = torch.tensor(random_field(m.n, 3), device=DEV)
    m.update_geometry(e0)
    n = m.ncol
    want = [torch.empty_like(e0) for _ in range(3)]
    m.recover_gradient(Phi0, e0, p0, *want)

    def check(place):
        """place(Phi, eta, phis, free) -> the three outputs."""
        Phi, buf, free = Phi0.clone(), torch.cat([e0, p0, p0]), torch.empty_like(e0)
        eta, phis = buf[:n], buf[n:2 * n]
        outs = place(Phi, eta, phis, free, buf)
        m.recover_gradient(Phi, eta, phis, *outs)
        for got, ref in zip(outs, want):
            assert torch.equal(got, ref)

    check(lambda Phi, eta, phis, free, buf: (free, eta, phis))
    check(lambda Phi, eta, phis, free, buf: (free, phis, eta))
    check(lambda Phi, eta, phis, free, buf: (eta, free, phis))
    check(lambda Phi, eta, phis, free, buf: (Phi[:n], Phi[n:2 * n], free))
    check(lambda Phi, eta, phis, free, buf: (free, torch.empty_like(e0), buf[n + n // 2:2 * n + n // 2]))
    # outputs over one another: the last argument stays
    a, b = torch.empty_like(e0), torch.empty_like(e0)
    m.recover_gradient(Phi0, e0, p0, b, a, a)
    assert torch.equal(b, want[0]) and torch.equal(a, want[2])
