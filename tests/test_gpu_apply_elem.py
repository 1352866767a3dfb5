"""FP32 apply with one element per thread (orders up to 8, up to four layers) against the oracle's assembled
operator, where its tiling can go wrong: fewer elements than a tile, one less, as many and one more,
several tiles per CTA being one launch's normal case on long tanks; every layer count; both ends; an
output that is not 16-byte aligned.  Tolerance 2e-6 on random input, the FP32 applies' own: a few
hundred FP32 roundings of 6e-8 on sums with cancellation.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from oracle import sem as osem  # noqa: E402
from sem_workloads import small_case  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
TILE = {1: 127, 2: 63, 3: 63, 4: 31}   # own elements of a tile per layer count


def run(P, Nx, Nz, periodic, offset=0):
    wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic)
    om = osem.mesh_for(wl)
    gm = sem.Mesh.from_workload(wl, h=om.h)
    eta = 0.05 * np.cos(om.xcol) + 0.01
    x = np.random.default_rng(P + Nx).standard_normal(om.n).astype(np.float32)
    gm.update_geometry(torch.tensor(eta, device=DEV))
    buf = torch.full((om.n + 8,), float("nan"), dtype=torch.float32, device=DEV)
    xin = torch.zeros(om.n + 4, dtype=torch.float32, device=DEV)[offset:offset + om.n]
    xin.copy_(torch.tensor(x))
    y = buf[offset:offset + om.n]
    gm.laplace_apply_f32(xin, y)
    assert torch.isnan(buf[:offset]).all() and torch.isnan(buf[offset + om.n:]).all()
    ref = om.stiffness(eta) @ x.astype(np.float64)
    return np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("P", range(2, 9))
@pytest.mark.parametrize("Nz", [1, 2, 3, 4])
def test_orders_and_layers(P, Nz):
    assert run(P, 5, Nz, True) < 2e-6
    assert run(P, TILE[Nz] + 1, Nz, False) < 2e-6


@pytest.mark.parametrize("Nz", [1, 2, 3, 4])
@pytest.mark.parametrize("delta", [-1, 0, 1])
@pytest.mark.parametrize("periodic", [True, False])
def test_tile_edges(Nz, delta, periodic):
    assert run(3, TILE[Nz] + delta, Nz, periodic) < 2e-6
    assert run(4, 2 * TILE[Nz] + delta, Nz, periodic, offset=1 + delta % 3) < 2e-6


def test_single_element_between_walls():
    for Nz in TILE:
        assert run(6, 1, Nz, False, offset=3) < 2e-6


def test_many_tiles_per_cta_match_the_fp64_apply():
    # more tiles than co-resident CTAs, so that both staging buffers are reused
    wl = small_case(P=2, Nx=31 * 152 * 16 * 3 + 5, Nz=4, periodic=True)
    m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol))
    x = torch.randn(m.n, dtype=torch.float32, device=DEV)
    m.update_geometry(0.01 * torch.sin(torch.arange(m.ncol, dtype=torch.float64, device=DEV) * 0.01))
    y, y64 = torch.empty_like(x), torch.empty(m.n, dtype=torch.float64, device=DEV)
    m.laplace_apply_f32(x, y)
    m.laplace_apply(x.double(), y64)
    assert float(torch.linalg.norm(y.double() - y64) / torch.linalg.norm(y64)) < 2e-6


@pytest.mark.parametrize("P,Nz", [(6, 1), (7, 1), (7, 2), (7, 3), (7, 4), (8, 1), (8, 2), (8, 3), (8, 4)])
@pytest.mark.parametrize("periodic", [True, False])
def test_orders_that_take_it_from_a_size_on(P, Nz, periodic):
    # the first size of the rule and one element more (a ragged last tile), against the FP64 apply
    for Nx in (152 * TILE[Nz], 152 * TILE[Nz] + 1):
        wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic)
        wl.length = 2 * np.pi * Nx / 64
        m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol))
        x = torch.randn(m.n, dtype=torch.float32, device=DEV)
        m.update_geometry(0.01 * torch.sin(torch.arange(m.ncol, dtype=torch.float64, device=DEV) * 0.01))
        y, y64 = torch.empty_like(x), torch.empty(m.n, dtype=torch.float64, device=DEV)
        m.laplace_apply_f32(x, y)
        m.laplace_apply(x.double(), y64)
        assert float(torch.linalg.norm(y.double() - y64) / torch.linalg.norm(y64)) < 2e-6
        m.close()
