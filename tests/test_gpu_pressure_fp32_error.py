"""The FP32 pressure operator's error against the plain contractions' (one multiply-add per entry and value), which the
even-odd form must not exceed: low orders have few terms for its extra roundings to be lost in."""

import numpy as np
import pytest

from oracle import pressure
from test_gpu_fixed_accuracy import curved

pytestmark = pytest.mark.gpu

F = np.float32


def fma(a, b, c):
    return (np.multiply(a, b, dtype=np.float64) + c).astype(F)  # the product of two FP32 numbers is exact in FP64


def line(M, v, axis, out=None):
    """M along `axis` of v, term by term, onto `out`."""
    v = np.moveaxis(v, axis, -1)
    out = np.zeros(v.shape[:-1] + (len(M),), F) if out is None else np.moveaxis(out, axis, -1).copy()
    for l in range(M.shape[1]):
        out = fma(M[:, l].astype(F), v[..., l : l + 1], out)
    return np.moveaxis(out, -1, axis)


def plain(N, F64, p, inv_mass):
    I, D, _ = pressure.interpolation_matrices(N)
    Ff, q = F64.astype(F), np.zeros(p.shape, F)
    for a in range(3):
        t = [(Ff[:, b, a] * p).astype(F) for b in range(3)]
        S = [line(D.T, t[0], 3), line(I.T, t[1], 3), line(I.T, t[2], 3)]
        u = line(I.T, line(I.T, S[0], 2, line(D.T, S[1], 2)), 1, line(D.T, line(I.T, S[2], 2), 1))
        u = (u * inv_mass).astype(F)
        XD, XI = line(D, u, 1), line(I, u, 1)
        g = [line(D, line(I, XI, 2), 3), line(I, line(D, XI, 2), 3), line(I, line(I, XD, 2), 3)]
        for b in (2, 1, 0):
            q = fma(Ff[:, b, a], g[b], q)
    return q


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7])
def test_no_further_off_than_plain_contractions(N):
    import torch
    import paper_2109_03592_gb300 as sem
    E = 500
    xyz, vert = curved(N, E, N)
    m = sem.Mesh(dict(kind="explicit", N=N, xyz=xyz, vert=vert, dirichlet_face=np.zeros((E, 6), np.uint8)))

    class Elements:
        pass
    mesh = Elements()
    mesh.N, mesh.E, mesh.xyz = N, E, xyz
    F64 = pressure.div_factors(mesh)[0]
    p = np.random.default_rng(N).standard_normal((E,) + (N - 1,) * 3).astype(F)
    B = m.geometry()[1].cpu().numpy()  # unconnected elements: the assembled mass is the local one
    u = pressure.grad_local(N, F64, p.astype(float)) / B
    ref = pressure.div_local(N, F64, u)
    q = m.pressure_apply_f32(torch.from_numpy(p).cuda(), torch.empty(p.shape, dtype=torch.float32, device="cuda")).cpu().numpy()
    err = lambda a: np.linalg.norm(a - ref) / np.linalg.norm(ref)
    assert err(q) <= 1.02 * err(plain(N, F64, p, (1.0 / B).astype(F)))
