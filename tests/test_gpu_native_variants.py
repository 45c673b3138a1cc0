"""Every kernel of the native FP64 operator (0 and 1: FP64 pipe, 4 and 5: fixed point), forced, on a curved pipe: plain, with
per-point coefficients, fused inside the CG; and the elements that the fixed-point operators evaluate in FP64 where no
factor vanishes."""

import numpy as np
import pytest

from oracle import mesh as omesh, operator, pressure, solver
from sem_inputs import forcing, vectors

pytestmark = pytest.mark.gpu

TOL = 1e-12  # relative L2
PIPE = dict(kind="pipe", nc=2, nr=1, nzp=3, L=2.0)


def _pipe(N):
    return solver.Problem(omesh.pipe(2, 1, 3, N, L=2.0), 1.0, 2.0)


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _mesh(N, variant, monkeypatch):
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    m = sem.Mesh(dict(N=N, **PIPE))
    assert m.ax_variant(sem.FP64) == variant and not m.fp64_double_float()
    return m


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("variant", [0, 1, 4, 5])
@pytest.mark.parametrize("N", [3, 4, 7, 8])
def test_plain_coefficients_and_fused(N, variant, monkeypatch):
    import torch
    m, P = _mesh(N, variant, monkeypatch), _pipe(N)
    u = vectors.local_field(3, m.E, m.n)
    ax = lambda h1, h2: m.ax(_dev(u), torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, h2).cpu().numpy()
    for h1, h2 in [(1.0, 0.0), (0.3, 7.0), (0.0, 3.0)]:
        assert _rel(ax(h1, h2), operator.ax_local(u, P.G, P.B, P.D, h1, h2)) < TOL
    c = 1.0 + 0.3 * np.sin(2 * P.mesh.xyz[:, 0]) * np.cos(P.mesh.xyz[:, 2])
    m.set_coefficients(_dev(c), _dev(2 * c))
    assert _rel(ax(1.0, 0.5), operator.ax_local(u, P.G, P.B, P.D, c, c)) < TOL
    m.set_coefficients(None, None)
    b = P.rhs(forcing.evaluate(P.mesh.xyz, forcing.random_modes(4, L=2.0)))
    x = torch.zeros(m.shape, dtype=torch.float64, device="cuda")
    res = m.solve(_dev(b), x, tol=1e-10, h2=2.0)
    ref = solver.pcg(P, b, tol=1e-10)
    assert res["status"] == 0 and abs(res["iters"] - ref.iters) <= 2
    assert _rel(x.cpu().numpy(), ref.x.reshape(m.shape)) <= 1e-8


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [3, 4, 7, 8])
@pytest.mark.parametrize("value", [1e200, 1e-200, np.nan, np.inf])
def test_elements_taken_in_fp64(N, variant, value, monkeypatch):
    import torch
    m, P = _mesh(N, variant, monkeypatch), _pipe(N)
    u = vectors.local_field(6, m.E, m.n)
    ax = lambda v: m.ax(_dev(v), torch.empty(m.shape, dtype=torch.float64, device="cuda"), 0.7, 2.0).cpu().numpy()
    clean, taken = ax(u), [1, 8, 20, m.E - 1]
    kept = [e for e in range(m.E) if e not in taken]
    v = u.copy()
    if np.isfinite(value):
        v[taken] *= value
    else:
        v[taken, 1, 2, 0] = value
    with np.errstate(invalid="ignore"):
        ref = operator.ax_local(v, P.G, P.B, P.D, 0.7, 2.0)
    w = ax(v)
    assert np.array_equal(w[kept], clean[kept])
    for e in taken:
        if np.isfinite(value):
            assert _rel(w[e] / value, ref[e] / value) < TOL
        else:
            assert np.array_equal(np.isfinite(w[e]), np.isfinite(ref[e]))


@pytest.mark.parametrize("N", [3, 4, 7, 8])
@pytest.mark.parametrize("value", [1e200, 1e-200, np.nan])
def test_pressure_elements_taken_in_fp64(N, value):
    import torch
    import paper_2109_03592_gb300 as sem
    m, P = sem.Mesh(dict(N=N, **PIPE)), _pipe(N)
    Q = pressure.Pressure(P)
    rng = np.random.default_rng(7)
    p, v = rng.standard_normal(Q.shape), rng.standard_normal((3,) + m.shape)
    u = torch.empty(3 * m.n_local, dtype=torch.float64, device="cuda")
    q = torch.empty(Q.shape, dtype=torch.float64, device="cuda")

    def grad(a):
        m.pressure_grad(_dev(a), u)
        return u.cpu().numpy().reshape(v.shape).copy()

    def div(a):
        m.pressure_div(_dev(a).reshape(-1), q)
        return q.cpu().numpy().copy()
    g0, d0, taken = grad(p), div(v), [1, 8, 20, m.E - 1]
    kept = [e for e in range(m.E) if e not in taken]
    r, w = p.copy(), v.copy()
    if np.isfinite(value):
        r[taken] *= value
        w[:, taken] *= value
    else:
        r[taken, 0, 0, 0] = value
        w[1, taken, 0, 0, 0] = value
    g, d = grad(r), div(w)
    assert np.array_equal(g[:, kept], g0[:, kept]) and np.array_equal(d[kept], d0[kept])
    gr, dr = pressure.grad_local(N, Q.F, r), pressure.div_local(N, Q.F, w)
    for e in taken:
        if np.isfinite(value):
            assert _rel(g[:, e] / value, gr[:, e] / value) < TOL and _rel(d[e] / value, dr[e] / value) < TOL
        else:
            assert not np.isfinite(g[:, e]).all() and not np.isfinite(d[e]).all()
