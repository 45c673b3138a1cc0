"""<p, A p> of the FP64 CG's fused fixed-point operator, seen through the step length of one iteration, on smooth p with a
mean: the element's contributions cancel, so an error of one sign would add up."""

import numpy as np
import pytest

from oracle import gll, mesh as omesh, operator, solver

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _derivative(N):
    """D in long double."""
    n = N + 1
    x = gll.nodes_weights(N)[0].astype(LD)
    for i in range(1, N):
        for _ in range(5):
            q, p = LD(1), x[i]
            for j in range(1, N):
                q, p = p, ((2 * j + 1) * x[i] * p - j * q) / LD(j + 1)
            x[i] += (q - x[i] * p) / ((N + 1) * p)
    x = (x - x[::-1]) / 2
    D = np.zeros((n, n), LD)
    for i in range(n):
        for l in range(n):
            if l != i:
                k = [k for k in range(n) if k not in (i, l)]
                D[i, l] = np.prod((x[i] - x[k]) / (x[l] - x[k])) / (x[l] - x[i])
        D[i, i] = -D[i].sum()
    return D


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N,h1,h2", [(3, 1.0, 0.0), (5, 0.7, 0.0), (7, 1.0, 0.0), (7, 1.0, 2.5), (8, 1.0, 0.0), (11, 1.0, 1e-4)])
@pytest.mark.parametrize("amp", [1.0, 1e-2, 1e-3])
def test_step_length_of_one_iteration(N, h1, h2, amp, variant, monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    om = omesh.box(3, 3, 2, N, 1.0, 1.0, 0.7)
    free = np.zeros((om.xyz.shape[0], 6), np.uint8)  # no Dirichlet faces: p keeps its mean
    m = sem.Mesh(dict(kind="explicit", N=N, xyz=om.xyz, vert=sem.mesh_vertices(dict(kind="box", nx=3, ny=3, nz=2, N=N)), dirichlet_face=free))
    assert m.ax_variant(sem.FP64) == variant
    x, y, z = om.xyz[:, 0], om.xyz[:, 1], om.xyz[:, 2]
    p = 1.0 + amp * np.cos(2 * x + 0.3) * np.cos(3 * y + 0.1) * np.sin(2 * z + 0.5)
    inv = m.jacobi(torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, h2).cpu().numpy()
    b = p / inv
    p = inv * b  # the first direction, as the solver rounds it
    out = torch.zeros(m.shape, dtype=torch.float64, device="cuda")
    m.solve(torch.from_numpy(b).cuda(), out, tol=1e-10, maxit=1, h1=h1, h2=h2)
    alpha = (out.cpu().numpy().astype(LD) * p).sum() / (p.astype(LD) ** 2).sum()

    mult = solver.Problem(om).mult
    G, B = (a.cpu().numpy().astype(LD) for a in m.geometry())
    w = operator.ax_local(p.astype(LD), G, B, _derivative(N), LD(h1), LD(h2))
    pap = (p * w).sum()
    rz = (b.astype(LD) * p / mult).sum()
    # one rounding of every product is eps |p w|; the vectors' own roundings and the sums' take no more than three others
    bound = 4 * 2.0 ** -53 * float(np.abs(p * w).sum() / pap) + 4 * 2.0 ** -53
    assert abs(float(alpha * pap / rz) - 1.0) < bound
