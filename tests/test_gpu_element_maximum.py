"""The element maximum behind the fixed-point operators' exponents where only some lanes of a warp take the branch
ahead of it: last CTAs of one element, and values of very different size in the lanes outside the branch."""

import numpy as np
import pytest

from oracle import mesh as omesh, operator, pressure, solver

pytestmark = pytest.mark.gpu

TOL = 1e-12  # relative L2 per element


def _worst(a, b, terms):
    """Per element, against the terms of the sums: the large values cancel in some of the results."""
    return max(np.linalg.norm(x - y) / np.linalg.norm(z) for x, y, z in zip(a, b, terms))


def _div_terms(Q, u):
    I, Dg, _ = pressure.interpolation_matrices(Q.N)
    C = [[np.abs(Dg if d == b else I) for d in (2, 1, 0)] for b in range(3)]  # (Mk, Mj, Mi)
    return sum(np.abs(Q.F[:, b, a]) * pressure._contract(*C[b], np.abs(u[a])) for a in range(3) for b in range(3))


@pytest.mark.parametrize("N", [1, 2, 3, 4, 6, 7, 8, 11])
@pytest.mark.parametrize("E", [1, 3])
def test_largest_value_in_any_lane(N, E):
    import torch
    import paper_2109_03592_gb300 as sem
    n = N + 1
    m = sem.Mesh(dict(kind="box", nx=E, ny=1, nz=1, N=N, lx=1.0 * E, ly=0.7, lz=1.3))
    P = solver.Problem(omesh.box(E, 1, 1, N, 1.0 * E, 0.7, 1.3))
    Q = pressure.Pressure(P) if N >= 2 else None
    rng = np.random.default_rng(N)
    for line in {0, n * n // 2, max(0, n * (N - 1) - 1), n * (N - 1), n * n - 1}:
        u = rng.standard_normal((3, E, n, n, n))
        u[1, :, :, line // n, line % n] = 1e3  # the second component's largest values sit in one thread's line
        for v in u:
            w = m.ax(torch.from_numpy(v).cuda(), torch.empty(m.shape, dtype=torch.float64, device="cuda"))
            assert _worst(w.cpu().numpy(), operator.ax_local(v, P.G, P.B, P.D),
                          operator.ax_local(np.abs(v), np.abs(P.G), P.B, np.abs(P.D))) < TOL
        if Q is not None:
            q = torch.empty(Q.shape, dtype=torch.float64, device="cuda")
            m.pressure_div(torch.from_numpy(u).cuda(), q)
            assert _worst(q.cpu().numpy(), Q.div(u), _div_terms(Q, u)) < TOL
