"""Device bytes of a mesh: a mesh carries what its own precision and preconditioner use.

Bytes per node of three long tanks (order 6 with four layers, 4 with one, 8 with two).  The limits are what such a mesh
took before the stages' guess history (72 bytes a node) came to it, the same for both precisions and
preconditioners: a tank that fitted a device then still does.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("precond", ["separable", "jacobi"])
@pytest.mark.parametrize("P,Nx,Nz,limit", [(6, 2048, 4, 236.8), (4, 5000, 1, 269.0), (8, 999, 2, 242.3)])
def test_bytes_per_node(P, Nx, Nz, limit, precision, precond):
    prm = sem.mesh_params(P, Nx, Nz, Pf=(3 * P + 1) // 2, precision=precision, precond=precond)
    nbytes = sem.mesh_footprint(prm, np.linspace(0.0, 1.0, Nx + 1), np.ones(Nx * P))
    assert nbytes <= limit * Nx * P * (Nz * P + 1)
