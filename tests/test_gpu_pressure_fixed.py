"""GPU parity of the fixed-point pressure operators (FP64 weak gradient, weak divergence and E) where they can go
wrong: every order with a partial last CTA, inputs at the bound of the integer sums, elements with values that are not
finite or far from one another, and elements and components of zeros."""

import numpy as np
import pytest

from oracle import mesh as omesh, pressure, solver

pytestmark = pytest.mark.gpu

TOL = 1e-12  # relative L2, as for the other FP64 operators
TOL32 = 2e-5

_cache = {}


def setup(N, shape=(3, 2, 1)):
    import paper_2109_03592_gb300 as sem
    key = (N, shape)
    if key not in _cache:
        nx, ny, nz = shape
        d = dict(kind="box", nx=nx, ny=ny, nz=nz, N=N, lx=1.5, ly=1.0, lz=0.5)
        _cache[key] = (sem.Mesh(d), pressure.Pressure(solver.Problem(omesh.box(nx, ny, nz, N, 1.5, 1.0, 0.5))))
    return _cache[key]


def gpu(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def grad(m, p):
    import torch
    u = torch.empty(3 * m.n_local, dtype=torch.float64, device="cuda")
    m.pressure_grad(gpu(p), u)
    return u.cpu().numpy()


def div(m, u, shape):
    import torch
    q = torch.empty(shape, dtype=torch.float64, device="cuda")
    m.pressure_div(gpu(u), q)
    return q.cpu().numpy()


@pytest.mark.parametrize("N", range(2, 12))
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 3, 1)])
def test_every_order_and_ragged_counts(N, shape):
    import torch
    m, P = setup(N, shape)
    rng = np.random.default_rng(N)
    p = rng.standard_normal(P.shape)
    u = P.grad(p)
    assert rel(grad(m, p).reshape(u.shape), u) < TOL
    v = rng.standard_normal(u.shape)
    assert rel(div(m, v, P.shape), P.div(v)) < TOL
    if N > 2 or shape != (1, 1, 1):  # (a single element of order 2 has one free node)
        q = torch.empty(P.shape, dtype=torch.float64, device="cuda")
        m.pressure_apply(gpu(p), q)
        ref = P.E(p)
        assert rel(q.cpu().numpy(), ref) < TOL
        q32 = torch.empty(P.shape, dtype=torch.float32, device="cuda")
        m.pressure_apply_f32(gpu(p.astype(np.float32)), q32)
        assert rel(q32.cpu().numpy(), ref) < TOL32


@pytest.mark.parametrize("N", [2, 3, 5, 7, 8, 9, 11])
def test_inputs_at_the_bound_of_the_sums(N):
    """Fields whose signs follow the rows of the 1D matrices: every sum of a contraction takes its largest value."""
    m, P = setup(N)
    I, Dg, _ = pressure.interpolation_matrices(N)
    top = 2.0 - 2.0 ** -52  # all mantissa bits set: the largest value below the next exponent
    for X, Y, Z in ((I, I, I), (Dg, I, I), (I, Dg, I), (I, I, Dg), (Dg, Dg, Dg)):
        for r in (0, (N - 1) // 2, N - 2):
            s = [np.where(M[r] < 0, -1.0, 1.0) for M in (X, Y, Z)]
            v = np.broadcast_to(top * np.einsum("k,j,i->kji", *s), P.grad(np.zeros(P.shape)).shape).copy()
            if np.ptp(v) == 0.0:  # a constant: its divergence is zero, so the error is bounded by the terms that cancel
                terms = sum(np.abs(P.F[:, b, a]) for a in range(3) for b in range(3)) * top * np.abs(Dg).sum(1).max()
                assert np.linalg.norm(div(m, v, P.shape) - P.div(v)) < TOL * np.linalg.norm(terms)
            else:
                assert rel(div(m, v, P.shape), P.div(v)) < TOL
        for l in (0, N // 2, N):
            s = [np.where(M[:, l] < 0, -1.0, 1.0) for M in (X, Y, Z)]
            p = np.broadcast_to(top * np.einsum("k,j,i->kji", *s), P.shape).copy()
            u = P.grad(p)
            assert rel(grad(m, p).reshape(u.shape), u) < TOL


@pytest.mark.parametrize("N", [4, 7, 11])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e200, 1e-200, 3e-310])
def test_elements_out_of_range(N, value):
    """One element (in the middle, and the last) not finite or far out of scale: the others stay as they are, bit for
    bit, and a finite one keeps its relative accuracy."""
    m, P = setup(N)
    rng = np.random.default_rng(7)
    p, v = rng.standard_normal(P.shape), rng.standard_normal((3,) + P.shape[:1] + (N + 1,) * 3)
    g0, d0 = grad(m, p).reshape(v.shape), div(m, v, P.shape)
    for e in (2, P.shape[0] - 1):
        q, w = p.copy(), v.copy()
        if np.isfinite(value):
            q[e] *= value
            w[:, e] *= value
        else:
            q[e, 0, 0, 0] = value
            w[1, e, 0, 0, 0] = value
        g, d = grad(m, q).reshape(v.shape), div(m, w, P.shape)
        rest = np.arange(P.shape[0]) != e
        assert np.array_equal(g[:, rest], g0[:, rest]) and np.array_equal(d[rest], d0[rest])
        if np.isfinite(value):
            tol = TOL if value > 1e-300 else 1e-3  # values below 2^-1022 keep few bits
            assert rel(g[:, e] / value, g0[:, e]) < tol and rel(d[e] / value, d0[e]) < tol
        else:
            ref_g, ref_d = P.grad(q), P.div(w)
            assert np.array_equal(np.isfinite(g[:, e]), np.isfinite(ref_g[:, e]))
            assert np.array_equal(np.isfinite(d[e]), np.isfinite(ref_d[e]))


@pytest.mark.parametrize("N", [3, 7])
def test_zeros_and_components_of_different_size(N):
    m, P = setup(N)
    rng = np.random.default_rng(3)
    v = rng.standard_normal((3,) + P.shape[:1] + (N + 1,) * 3)
    for scale in ((1.0, 0.0, 0.0), (0.0, 1e-30, 0.0), (1e-30, 1.0, 1e30), (0.0, 0.0, 0.0), (1e-160, 1e160, 0.0)):
        w = v * np.array(scale).reshape(3, 1, 1, 1, 1)
        d, ref = div(m, w, P.shape), P.div(w)
        assert np.array_equal(d, ref) if not ref.any() else rel(d / abs(ref).max(), ref / abs(ref).max()) < TOL
    p = rng.standard_normal(P.shape)
    p[1] = 0.0
    g = grad(m, p).reshape(v.shape)
    assert not g[:, 1].any() and rel(g, P.grad(p)) < TOL
