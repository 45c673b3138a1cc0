"""Scalar coefficients far from 1 on the fixed-point FP64 operator: a power of two passes through it exactly, so they cost
no more than others (they used to be evaluated in FP64, element by element)."""

import numpy as np
import pytest

from oracle import mesh as omesh, operator, solver

pytestmark = pytest.mark.gpu

AX_TOL = 1e-12


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [1, 4, 7, 8, 11])
def test_powers_of_two_pass_through(N, variant, monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    E = 5
    m = sem.Mesh(dict(kind="box", nx=E, ny=1, nz=1, N=N, lx=1.0 * E, ly=0.7, lz=1.3))
    assert m.ax_variant(sem.FP64) == variant
    P = solver.Problem(omesh.box(E, 1, 1, N, 1.0 * E, 0.7, 1.3))
    u = np.random.default_rng(N).standard_normal(m.shape)
    ud = torch.from_numpy(u).cuda()
    ax = lambda h1, h2: m.ax(ud, torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, h2).cpu().numpy()
    w, wh = ax(0.75, 0.0), ax(0.75, 0.375)
    for k in (-900, -150, -101, 101, 150, 900):
        assert np.array_equal(ax(np.ldexp(0.75, k), 0.0), np.ldexp(w, k))
        assert np.array_equal(ax(np.ldexp(0.75, k), np.ldexp(0.375, k)), np.ldexp(wh, k))
    for h1, h2 in [(1e-300, 1e300), (1e300, 1e-300), (-1e200, 1e199), (1.0, 1e-200), (0.0, 1e250), (1e-250, 0.0)]:
        ref = operator.ax_local(u, P.G, P.B, P.D, h1, h2)
        d, s = ax(h1, h2) - ref, np.abs(ref).max()
        assert np.linalg.norm(d / s) < AX_TOL * np.linalg.norm(ref / s)
    with np.errstate(invalid="ignore", over="ignore"):
        assert not np.isfinite(ax(np.inf, 0.0)).any() and np.isnan(ax(np.nan, 1.0)).all()
        assert np.array_equal(np.isinf(ax(1e308, 0.0)), np.isinf(1e308 * w / 0.75))
    b = P.rhs(np.ones(m.shape))
    if np.linalg.norm(b):  # the fused form
        x, y = (torch.zeros(m.shape, dtype=torch.float64, device="cuda") for _ in range(2))
        r = m.solve(torch.from_numpy(b).cuda(), x, tol=1e-10, h1=0.75, h2=0.5)
        q = m.solve(torch.from_numpy(np.ldexp(b, -150)).cuda(), y, tol=1e-10, h1=0.75 * 2.0 ** -150, h2=2.0 ** -151)
        assert r["status"] == q["status"] == 0 and r["iters"] == q["iters"]
        assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
