"""The fixed-point FP64 operator on elements whose values differ by many orders of magnitude: every point is as accurate as
its own terms, as in FP64, although the values of an element share one exponent."""

import numpy as np
import pytest

import long_double
from oracle import gll, mesh as omesh, operator, solver
from test_gpu_fixed_accuracy import curved

pytestmark = pytest.mark.gpu

# Emulated: an error of 2^-51 of a point's terms where its best line lies 2^-6 below the element's largest value, and
# twice that for each further bit, of which the integer path takes 12
BOUND = 2.0 ** -45


def _fields(E, n, rng):
    """E elements of values of size 1e-9 with large ones among them."""
    def some():
        return rng.standard_normal((E, n, n, n))
    small, mid = 1e-9 * some(), n // 2
    out = {}
    u = small.copy()
    u[:, 0, 0, 0] = 1.0
    out["one value"] = u
    u = small.copy()
    u[:, :, mid, mid] = 1.0 + 0.1 * some()[:, :, mid, mid]
    out["a t-line"] = u
    u = small.copy()
    u[:, mid, :, 0] = 1.0 + 0.1 * some()[:, mid, :, 0]
    out["an s-line"] = u
    u = small.copy()
    u[:, -1, 0] = 1.0 + 0.1 * some()[:, -1, 0]
    out["an r-line"] = u
    u = small.copy()
    u[:, 0] = some()[:, 0]
    u[..., 0] = 0.0
    out["a plane, beside zeros on a face"] = u
    u = some()
    u[:, :, :, : n - 1] *= 1e-9
    out["a plane"] = u
    d = ((np.stack(np.meshgrid(*[np.linspace(0, 1, n)] * 3)) - 0.2) ** 2).sum(0)
    out["a narrow Gaussian"] = np.exp(-40 * d) * (1 + 0.01 * some())
    u = some()
    u[1::2] = small[1::2]
    u[1::2, 0, 0, 0] = 1.0
    out["every other element"] = u
    u = 2.0 ** -14 * some()
    u[:, 0, 0, 0] = 1.0
    out["just beyond the line"] = u
    return out


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N,h1,h2", [(1, 1.0, 0.0), (2, 1.0, 0.5), (3, 0.3, 0.0), (4, 1.0, 0.0), (7, 1.0, 0.0), (7, 2.0, 3.0), (8, 1.0, 7.0), (11, 1.0, 0.0)])
def test_every_point_to_its_own_terms(N, h1, h2, variant, monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    E, n = 7, N + 1
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    xyz, vert = curved(N, E, 3)
    m = sem.Mesh(dict(kind="explicit", N=N, xyz=xyz, vert=vert, dirichlet_face=np.zeros((E, 6), np.uint8)))
    assert m.ax_variant(sem.FP64) == variant
    G, B = (a.cpu().numpy().astype(long_double.LD) for a in m.geometry())  # (its own rounding is not the question)
    Gabs = np.broadcast_to(np.abs(G).max(1, keepdims=True), G.shape)  # small factors are rounded like the point's largest
    D = long_double.basis(N)[2]
    for name, u in _fields(E, n, np.random.default_rng(N)).items():
        w = m.ax(torch.from_numpy(u).cuda(), torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, h2).cpu().numpy()
        ref = operator.ax_local(u.astype(D.dtype), G, B, D, h1, h2)
        terms = operator.ax_local(np.abs(u).astype(D.dtype), Gabs, B, np.abs(D), h1, h2)
        assert float((np.abs(w - ref) / terms).max()) < BOUND, name


@pytest.mark.parametrize("N", [3, 4, 7, 11])
def test_rounding_of_zeros(N, monkeypatch):
    """Lines that hold the rounding of zeros (2^-44 of the element's largest and below) are carried to that precision."""
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", "4")
    m = sem.Mesh(dict(kind="box", nx=2, ny=2, nz=2, N=N))
    om = omesh.box(2, 2, 2, N)
    P = solver.Problem(om)
    x, y, z = (om.xyz[:, c] for c in range(3))
    u = np.sin(2 * np.pi * x) * np.sin(2 * np.pi * y) * np.sin(2 * np.pi * z)
    w = m.ax(torch.from_numpy(u).cuda(), torch.empty(m.shape, dtype=torch.float64, device="cuda")).cpu().numpy()
    terms = operator.ax_local(np.abs(u), np.abs(P.G), P.B, np.abs(P.D)).reshape(8, -1).max(1)
    err = np.abs(w - operator.ax_local(u, P.G, P.B, P.D)).reshape(8, -1).max(1)
    assert (err < 16 * 2.0 ** -53 * terms).all()


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [1, 4, 7, 9])
@pytest.mark.parametrize("h1,h2", [(0.0, 3.0), (1e-12, 5.0), (1.0, 1e12)])
def test_mass_alone(N, h1, h2, variant, monkeypatch):
    """Where the mass term is most of the result it is rounded point by point."""
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    E = 5
    m = sem.Mesh(dict(kind="box", nx=E, ny=1, nz=1, N=N, lx=1.0 * E, ly=0.7, lz=1.3))
    G, B = (a.cpu().numpy() for a in m.geometry())
    D = gll.derivative_matrix(N)
    u = np.random.default_rng(5).standard_normal(m.shape) * 10.0 ** np.random.default_rng(6).uniform(-3, 0, m.shape)
    w = m.ax(torch.from_numpy(u).cuda(), torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, h2).cpu().numpy()
    ref = operator.ax_local(u, G, B, D, h1, h2)
    terms = operator.ax_local(np.abs(u), np.abs(G), B, np.abs(D), h1, h2)
    assert (np.abs(w - ref) < 8 * 2.0 ** -53 * terms).all()


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [3, 5, 7, 8, 11])
def test_solve_with_a_narrow_source(N, variant, monkeypatch):
    """The fused form: a source much narrower than an element leaves directions of very uneven size."""
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    m = sem.Mesh(dict(kind="box", nx=3, ny=2, nz=2, N=N))
    om = omesh.box(3, 2, 2, N)
    P = solver.Problem(om, 1.0, 2.0)
    b = P.rhs(np.exp(-150 * ((om.xyz - 0.45) ** 2).sum(1)))
    x = torch.zeros(m.shape, dtype=torch.float64, device="cuda")
    res = m.solve(torch.from_numpy(b).cuda(), x, tol=1e-10, h2=2.0)
    ref = solver.pcg(P, b, tol=1e-10)
    assert res["status"] == 0 and abs(res["iters"] - ref.iters) <= 2
    assert np.linalg.norm(x.cpu().numpy() - ref.x.reshape(m.shape)) <= 1e-8 * np.linalg.norm(ref.x)
