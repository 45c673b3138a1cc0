"""The FP64 pressure operators in fixed point against FP64 evaluation (the oracle), both against long double: over all
points, and for the gradient at interior, face, edge and corner points, which differ in the size of their values."""

import numpy as np
import pytest

import long_double
from oracle import pressure
from test_gpu_fixed_accuracy import rms

pytestmark = pytest.mark.gpu

MOST = 1.5  # emulated: 0.25 to 0.45 times FP64's for E, 0.1 to 1.3 for the gradient, beside equal errors of the geometry


@pytest.mark.parametrize("field", ["random", "smooth"])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 9, 10, 11])
def test_no_further_off_than_fp64(N, field):
    import torch
    import paper_2109_03592_gb300 as sem
    E, n, rng = 24, N + 1, np.random.default_rng(N)
    x = ((long_double.basis(N)[0] + 1) / 2).astype(float)
    X = np.stack(np.meshgrid(x, x, x, indexing="ij")[::-1])
    xyz = np.stack([np.einsum("ab,bkji->akji", np.eye(3) + 0.12 * rng.standard_normal((3, 3)), X) for _ in range(E)])
    m = sem.Mesh(dict(kind="explicit", N=N, xyz=xyz, vert=np.arange(8 * E).reshape(E, 8), dirichlet_face=np.zeros((E, 6), np.uint8)))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    z = np.polynomial.legendre.leggauss(N - 1)[0]
    Z = np.meshgrid(z, z, z, indexing="ij")
    p = rng.standard_normal((E,) + (N - 1,) * 3)
    if field == "smooth":
        p = np.stack([np.cos(2 * Z[2] + e) * np.sin(1.5 * Z[1] + 0.2) * np.cos(Z[0] + 0.1 * e) for e in range(E)])

    class Elements:
        pass
    mesh = Elements()
    mesh.N, mesh.E, mesh.xyz = N, E, xyz
    F64, F = pressure.div_factors(mesh)[0], long_double.div_factors(N, xyz)
    B64, B = m.geometry()[1].cpu().numpy(), long_double.factors(N, xyz)[1]  # unconnected: also the assembled mass

    u = torch.empty(3 * m.n_local, dtype=torch.float64, device="cuda")
    q = torch.empty(p.shape, dtype=torch.float64, device="cuda")
    ref = long_double.grad(N, F, p.astype(long_double.LD))
    m.pressure_grad(dev(p), u)
    e = (u.cpu().numpy().reshape(ref.shape) - ref).astype(float)
    e64 = (pressure.grad_local(N, F64, p) - ref).astype(float)
    end = np.zeros(n, int)
    end[[0, -1]] = 1
    kind = end[:, None, None] + end[:, None] + end
    for k in range(4):
        if (kind == k).any():
            assert rms(e[..., kind == k]) <= MOST * rms(e64[..., kind == k]), k

    v = (ref / B).astype(float)
    exact = long_double.div(N, F, v.astype(long_double.LD))
    m.pressure_div(dev(v).reshape(-1), q)
    assert rms(q.cpu().numpy() - exact) <= MOST * rms(pressure.div_local(N, F64, v) - exact)

    exact = long_double.div(N, F, ref / B)
    m.pressure_apply(dev(p), q)
    assert rms(q.cpu().numpy() - exact) <= MOST * rms(pressure.div_local(N, F64, pressure.grad_local(N, F64, p) / B64) - exact)
