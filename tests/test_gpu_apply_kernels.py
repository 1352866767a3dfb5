"""The two FP32 apply kernels, each at sizes where the dispatch would take the other one too.

SEM_APPLY_F32=line and =elem choose a kernel at every size that it serves.  Line passes: several tiles, a ragged
last one, an input that is not 16-byte aligned, every tile width, bitwise repeatable.  One element per
thread: the padded layout (P·Nrow a multiple of 8: (5, 3), (7, 1), order 8) with input and output off 16-byte alignment and
both ends, and orders 7 and 8 below the size from which the dispatch takes it.  The dispatch itself: one element below
its line and at it, the result bit for bit that of the kernel meant.  Against the FP64 apply, 2e-6 on random input, the
FP32 applies' own tolerance.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402
from sem_workloads import small_case  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
TOL = 2e-6


class Tank:
    def __init__(self, P, Nx, Nz, periodic=True, seed=0):
        wl = small_case(P=P, Nx=Nx, Nz=Nz, periodic=periodic)
        wl.length = 2 * np.pi * max(1.0, Nx / 64)
        self.m = sem.Mesh.from_workload(wl, h=np.ones(wl.ncol))
        i = torch.arange(self.m.ncol, dtype=torch.float64, device=DEV)
        self.m.update_geometry(0.05 * torch.cos(0.03 * i) + 0.01)
        self.x = torch.randn(self.m.n, generator=torch.Generator().manual_seed(seed), dtype=torch.float32).to(DEV)
        self.ref = torch.empty(self.m.n, dtype=torch.float64, device=DEV)
        self.m.laplace_apply(self.x.double(), self.ref)

    def apply(self, offset=0):
        """y, with x and y `offset` floats off their buffers' alignment; nothing else is written."""
        n = self.m.n
        xb, yb = torch.zeros(n + 4, device=DEV), torch.full((n + 8,), float("nan"), device=DEV)
        xb[offset:offset + n] = self.x
        y = yb[offset:offset + n]
        self.m.laplace_apply_f32(xb[offset:offset + n], y)
        assert torch.isnan(yb[:offset]).all() and torch.isnan(yb[offset + n:]).all()
        return y

    def error(self, y):
        return float(torch.linalg.norm(y.double() - self.ref) / torch.linalg.norm(self.ref))


@pytest.mark.parametrize("P,Nz", [(2, 1), (3, 4), (5, 2), (6, 1), (6, 4), (7, 3), (8, 2), (9, 2), (6, 6)])
@pytest.mark.parametrize("periodic", [True, False])
def test_line_passes(P, Nz, periodic, monkeypatch):
    monkeypatch.setenv("SEM_APPLY_F32", "line")
    t = Tank(P, 53, Nz, periodic)
    y = t.apply()
    assert t.error(y) < TOL and torch.equal(t.apply(), y)
    for offset in (1, 2, 3):
        assert torch.equal(t.apply(offset), y)
    try:
        for E in (1, 3, 7, 16):
            sem.set_apply_tile_width(P, Nz, E)
            assert t.error(t.apply()) < TOL, E
    finally:
        sem.set_apply_tile_width(P, Nz, 0)


@pytest.mark.parametrize("P,Nz", [(5, 3), (7, 1), (8, 1), (8, 2), (8, 3), (8, 4), (6, 4)])
@pytest.mark.parametrize("periodic", [True, False])
def test_element_kernel_off_alignment(P, Nz, periodic, monkeypatch):
    monkeypatch.setenv("SEM_APPLY_F32", "elem")
    for Nx in (5, 300):                     # less than a tile; several tiles, the last one ragged
        t = Tank(P, Nx, Nz, periodic)
        y = t.apply()
        assert t.error(y) < TOL
        for offset in (1, 2, 3):
            assert torch.equal(t.apply(offset), y)


@pytest.mark.parametrize("P,Nz,share,E", [(3, 1, 0.5, 127), (5, 1, 0.5, 127), (5, 2, 0.75, 63), (6, 1, 0.75, 127),
                                          (6, 4, 0.75, 31), (7, 4, 1.4, 31), (8, 2, 1.54, 63)])
def test_dispatch_line(P, Nz, share, E, monkeypatch):
    """share: tiles of E own elements per SM from which one element per thread serves (orders 7 and 8: of whole tiles,
    0.7 and 0.77 of a wave of two an SM)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = int(np.ceil(share * sms - 1e-9)) * E - E + 1 if P > 6 else int(np.ceil(share * sms * E - 1e-9))
    for Nx, kernel in ((line - 1, "line"), (line, "elem")):
        t = Tank(P, Nx, Nz)
        y = t.apply()
        assert t.error(y) < TOL
        monkeypatch.setenv("SEM_APPLY_F32", kernel)
        assert torch.equal(t.apply(), y)
        monkeypatch.delenv("SEM_APPLY_F32")
        t.m.close()
