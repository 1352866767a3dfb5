"""The applies are at least as accurate as plain lines on smooth fields.

A flat tank at rest (d = 1, no slopes), a field that varies by a fiftieth per element: its derivatives are small
beside its values, so what a line's sums round, and what the derivative's rounded rows leave of a constant,
shows in full.  Reference: the same contractions in extended precision, with nodes and weights computed there.
Plain: D u, weights, Dᵀ f, one product after the other in the kernel's own precision.  The kernels may
not be further from the reference than that, in either precision, whichever kernel serves.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1512_02548_gb300 as sem  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
X = np.longdouble


def gll(P):
    """Nodes, weights and derivative matrix in extended precision (Newton on P'_P)."""
    def leg(x):
        p0, p1 = np.ones_like(x), x.copy()
        for k in range(1, P):
            p0, p1 = p1, ((2 * k + 1) * x * p1 - k * p0) / X(k + 1)
        return p0, p1
    r = -np.cos(np.pi * np.arange(P + 1) / X(P))
    r[0], r[-1] = -1, 1
    for _ in range(60):
        x = r[1:-1]
        p0, p1 = leg(x)
        dp = P * (p0 - x * p1) / (1 - x * x)
        r[1:-1] = x - dp / ((2 * x * dp - P * (P + 1) * p1) / (1 - x * x))
    L = leg(r)[1]
    D = np.zeros((P + 1, P + 1), dtype=X)
    for i in range(P + 1):
        for j in range(P + 1):
            if i != j:
                D[i, j] = L[i] / (L[j] * (r[i] - r[j]))
        D[i, i] = -D[i].sum()
    return r, X(2) / (P * (P + 1) * L ** 2), D


def lines(M, u, axis, transpose=False):
    """Σ_c M[a, c] u[c] along `axis`, term after term in u's precision."""
    u = np.moveaxis(u, axis, 0)
    M = (M.T if transpose else M).astype(u.dtype)
    out = []
    for row in M:
        s = row[0] * u[0]
        for c in range(1, len(row)):
            s = s + row[c] * u[c]
        out.append(s)
    return np.moveaxis(np.stack(out), 0, axis)


def apply(w, D, u, dx, dsl, dtype):
    """-(contributions) of every node from its elements; u: (Nx·P+1, Nz·P+1)."""
    P = len(w) - 1
    Nx, Nz = (u.shape[0] - 1) // P, (u.shape[1] - 1) // P
    y = np.zeros(u.shape, dtype=dtype)
    ww = w.astype(dtype)[:, None] * w.astype(dtype)[None, :]
    for e in range(Nx):
        for l in range(Nz):
            v = u[e * P:(e + 1) * P + 1, l * P:(l + 1) * P + 1].astype(dtype)
            g1, g2 = ww * (dsl / dx[e]).astype(dtype), ww * (dx[e] / dsl).astype(dtype)
            y[e * P:(e + 1) * P + 1, l * P:(l + 1) * P + 1] -= (
                lines(D, g1 * lines(D, v, 0), 0, True) + lines(D, g2 * lines(D, v, 1), 1, True))
    return y


@pytest.mark.parametrize("P", range(2, 13))
@pytest.mark.parametrize("kind", ["float64", "line", "elem"])
def test_smooth_fields(P, kind, monkeypatch):
    if kind == "elem" and P > 8:
        pytest.skip("served by the line passes")
    dtype = np.float64 if kind == "float64" else np.float32
    if dtype == np.float32:
        monkeypatch.setenv("SEM_APPLY_F32", kind)
    Nx, Nz = 5, 2
    r, w, D = gll(P)
    edges = np.linspace(0.0, 2.0, Nx + 1)
    dx = np.diff(edges.astype(X))
    s = np.concatenate([e + (r[:-1] + 1) / 2 for e in range(Nx)] + [[X(Nx)]])
    z = np.concatenate([(l + (r[:-1] + 1) / 2) / Nz for l in range(Nz)] + [[X(1)]])
    u = (np.sin(0.3 + 0.02 * s)[:, None] * (1 + 0.01 * z ** 2)[None, :]).astype(dtype)
    ref = apply(w, D, u, dx, X(1) / Nz, X)
    plain = apply(w, D, u, dx, X(1) / Nz, dtype)

    m = sem.Mesh(P, Nx, Nz, edges, np.ones(Nx * P + 1), periodic=False)
    m.update_geometry(torch.zeros(m.ncol, dtype=torch.float64, device=DEV))
    x = torch.tensor(u.ravel(), device=DEV)
    y = torch.empty_like(x)
    (m.laplace_apply if dtype == np.float64 else m.laplace_apply_f32)(x, y)
    err = [float(np.linalg.norm((v - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64)))
           for v in (y.cpu().numpy().reshape(u.shape), plain)]
    assert err[0] <= err[1], err
