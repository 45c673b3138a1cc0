"""The fixed-point FP64 local operator (variants 4 and 5 of the native FP64
operator) at the edges of its ranges: every order, ragged last tiles, elements
of very different sizes of values, exponents on both sides of the integer
path's limits, non-finite values, and scalar coefficients of any size."""

import numpy as np
import pytest

from oracle import mesh as omesh, operator, solver
from sem_inputs import forcing, vectors

pytestmark = pytest.mark.gpu

AX_TOL = 1e-12  # FP64 Ax: relative L2 error bound, here of every element by itself


def _mesh(monkeypatch, N, variant, E=5):
    """A mesh of E affine elements (a ragged last tile) whose FP64 operator is `variant`, and the oracle's problem."""
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    desc = dict(kind="box", nx=E, ny=1, nz=1, N=N, lx=1.0 * E, ly=0.7, lz=1.3)
    m = sem.Mesh(desc)
    assert m.ax_variant(sem.FP64) == variant and not m.fp64_double_float()
    return m, solver.Problem(omesh.box(E, 1, 1, N, 1.0 * E, 0.7, 1.3))


def _ax(m, u, h1=1.0, h2=0.0):
    import torch
    w = torch.empty(m.shape, dtype=torch.float64, device="cuda")
    return m.ax(torch.from_numpy(np.ascontiguousarray(u)).cuda(), w, h1, h2).cpu().numpy()


def _worst(w, ref):
    d = np.sqrt(((w - ref) ** 2).reshape(len(w), -1).sum(1)) / np.sqrt((ref ** 2).reshape(len(w), -1).sum(1))
    return d.max()


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", range(1, 12))
def test_orders(N, variant, monkeypatch):
    m, P = _mesh(monkeypatch, N, variant)
    # each element's values of another size, one element all zeros
    u = vectors.local_field(3, m.E, m.n) * np.array([1.0, 1e-90, 0.0, 1e60, 1e-3]).reshape(-1, 1, 1, 1)
    on = [0, 1, 3, 4]
    for h1, h2 in [(1.0, 0.0), (0.3, 7.0), (-2.0, 1e-9), (1e-20, 1e20), (0.0, 3.0), (1e3, 1e-25)]:
        w = _ax(m, u, h1, h2)
        ref = operator.ax_local(u, P.G, P.B, P.D, h1, h2)
        assert not w[2].any()
        assert _worst(w[on], ref[on]) < AX_TOL, (h1, h2)


@pytest.mark.parametrize("N", [2, 3, 5, 7, 8, 9, 11])
def test_power_of_two_scaling(N, monkeypatch):
    """Inside the integer path's exponent range a power of two passes through exactly; outside it the element is
    evaluated in FP64, to the same bound."""
    m, P = _mesh(monkeypatch, N, 4)
    u = vectors.local_field(4, m.E, m.n)
    w = _ax(m, u)
    for k in (-450, -40, 1, 450):
        assert np.array_equal(_ax(m, np.ldexp(u, k)), np.ldexp(w, k))
    for k in (-700, 600, 900):
        assert _worst(np.ldexp(_ax(m, np.ldexp(u, k)), -k), w) < AX_TOL


@pytest.mark.parametrize("N", [4, 7])
@pytest.mark.parametrize("h1,h2", [(1e-50, 0.0), (1.0, 1e50), (1e70, 1e-70)])
def test_scalar_coefficients_out_of_range(N, h1, h2, monkeypatch):
    m, P = _mesh(monkeypatch, N, 5)
    u = vectors.local_field(5, m.E, m.n)
    assert _worst(_ax(m, u, h1, h2), operator.ax_local(u, P.G, P.B, P.D, h1, h2)) < AX_TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("N", [4, 7])
def test_non_finite_stays_where_fp64_puts_it(N, bad, monkeypatch):
    m, P = _mesh(monkeypatch, N, 4)
    u = vectors.local_field(6, m.E, m.n)
    clean = _ax(m, u)
    u[1, 1, 2, 3] = bad
    with np.errstate(invalid="ignore"):
        ref = operator.ax_local(u, P.G, P.B, P.D)
    w = _ax(m, u)
    keep = [0, 2, 3, 4]
    assert np.array_equal(w[keep], clean[keep])
    assert np.array_equal(np.isfinite(w[1]), np.isfinite(ref[1]))


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [1, 2, 3, 6, 7, 9, 10, 11])
def test_fused_in_the_fp64_solve(N, variant, monkeypatch):
    import torch
    m, P = _mesh(monkeypatch, N, variant, E=7)
    P = solver.Problem(P.mesh, 1.0, 2.0)
    b = P.rhs(forcing.evaluate(P.mesh.xyz, forcing.random_modes(4, L=3.0)))
    x = torch.zeros(m.shape, dtype=torch.float64, device="cuda")
    res = m.solve(torch.from_numpy(b).cuda(), x, tol=1e-10, h2=2.0)
    ref = solver.pcg(P, b, tol=1e-10)
    assert res["status"] == 0 and abs(res["iters"] - ref.iters) <= 2
    if np.linalg.norm(b):
        assert np.linalg.norm(x.cpu().numpy() - ref.x.reshape(m.shape)) <= 1e-8 * np.linalg.norm(ref.x)


def test_coefficients_out_of_range_use_the_fp64_pipe(monkeypatch):
    """Per-point coefficients too large for the integer path, then ordinary ones, then none."""
    import torch
    m, P = _mesh(monkeypatch, 7, 4)
    u = vectors.local_field(8, m.E, m.n)
    plain = _ax(m, u, 1.0, 2.0)
    one = torch.ones(m.shape, dtype=torch.float64, device="cuda")
    for h1, h2, s1, s2 in [(one * 1e80, None, 1e80, 1.0), (None, one * 1e80, 1.0, 1e80), (one * 3, one * 5, 3.0, 5.0)]:
        m.set_coefficients(h1, h2)
        assert _worst(_ax(m, u, 1.0, 2.0), operator.ax_local(u, P.G, P.B, P.D, s1, 2.0 * s2)) < AX_TOL
    m.set_coefficients(None, None)
    assert np.array_equal(_ax(m, u, 1.0, 2.0), plain)
    G, B = m.geometry()
    assert np.linalg.norm(G.cpu().numpy() - P.G) < 1e-13 * np.linalg.norm(P.G)
