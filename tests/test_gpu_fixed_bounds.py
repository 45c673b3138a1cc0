"""The FP64 local operator in fixed point on lines that bring the 64-bit sums
of its contractions to their bound, with a scalar h1 that the tables carry."""

import math

import numpy as np
import pytest

from oracle import gll, mesh as omesh, operator, solver

pytestmark = pytest.mark.gpu

AX_TOL = 1e-12  # FP64 Ax: relative L2 error bound (a wrapped sum is 2^32 of 2^60: 4e-9 of a gradient)
LD = np.longdouble


def _even_odd_tables(N):
    """E and O of D as 64-bit integers: rows of the first half, scaled so that D's largest row sum of magnitudes is
    0.8 (n even) or 0.5 (n odd) times 2^64."""
    n = N + 1
    x = gll.nodes_weights(N)[0].astype(LD)
    for i in range(1, N):
        for _ in range(5):  # Newton on P_{N-1} - x P_N, whose derivative is -(N + 1) P_N
            q, p = LD(1), x[i]
            for j in range(1, N):
                q, p = p, ((2 * j + 1) * x[i] * p - j * q) / LD(j + 1)
            x[i] += (q - x[i] * p) / ((N + 1) * p)
    x = (x - x[::-1]) / 2
    D = np.zeros((n, n), LD)
    for i in range(n):
        for l in range(n):
            if l != i:
                others = [k for k in range(n) if k not in (i, l)]
                D[i, l] = np.prod((x[i] - x[others]) / (x[l] - x[others])) / (x[l] - x[i])
        D[i, i] = -D[i].sum()
    s = np.ldexp(LD(0.5 if n % 2 else 0.8), 64) / np.abs(D).sum(1).max()
    num = lambda v: int(np.rint(v * s))
    rows = range((n + 1) // 2)
    E = [[num((D[r, l] + D[r, N - l]) / 2) for l in range(n // 2)] + ([num(D[r, n // 2])] if n % 2 else []) for r in rows]
    O = [[num((D[r, l] - D[r, N - l]) / 2) for l in range(n // 2)] for r in rows]
    return E, O


def _split(v):
    lo = ((v + 2 ** 31) & (2 ** 32 - 1)) - 2 ** 31
    return lo, (v - lo) >> 32


def _worst_line(N, h1):
    """The line whose folded values bring one middle sum of the contraction with h1 D nearest to (or beyond) 2^63, and
    that sum / 2^63."""
    n, half = N + 1, (N + 1) // 2
    mant = int(math.ldexp(math.frexp(h1)[0], 53))
    best = (0, None)
    for even, table in enumerate(reversed(_even_odd_tables(N))):  # O (antisymmetric lines), then E (symmetric)
        for row in table:
            total, v = 2 ** 31, [0] * n
            for l, c in enumerate(row):
                lo, hi = _split((c * mant + 2 ** 52) >> 53)
                mid = l == half  # the middle point of an odd n stands for itself
                top = 2 ** (60 if mid else 61)
                # of 53-bit values near +-top, the one whose halves meet the entry's signs
                f = max((s * (top - 2 ** 31 + d * 2 ** 9) for s in (1, -1) for d in (1, -1)),
                        key=lambda f: lo * _split(f)[1] + hi * _split(f)[0])
                total += lo * _split(f)[1] + hi * _split(f)[0]
                v[l] = f if mid else f // 2
                if not mid:
                    v[N - l] = v[l] if even else -v[l]
            if total / 2 ** 63 > best[0]:
                best = (total / 2 ** 63, np.ldexp(np.array(v, dtype=float), -59))
    return best


@pytest.mark.parametrize("variant", [4, 5])
@pytest.mark.parametrize("N", [3, 6, 7, 8, 9, 10, 11])
def test_sums_at_their_bound(N, variant, monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    E = 3
    m = sem.Mesh(dict(kind="box", nx=E, ny=1, nz=1, N=N, lx=1.0 * E, ly=0.7, lz=1.3))
    assert m.ax_variant(sem.FP64) == variant
    P = solver.Problem(omesh.box(E, 1, 1, N, 1.0 * E, 0.7, 1.3))
    rng = np.random.default_rng(12)
    sums = []
    for h1 in [1.0, 3.901, 0.9706] + list(np.ldexp(1.0 + rng.random(20), -1)):
        s, line = _worst_line(N, h1)
        sums.append(s)
        u = np.empty((E,) + (N + 1,) * 3)
        u[0], u[1], u[2] = line[None, None, :], line[None, :, None], line[:, None, None]
        w = m.ax(torch.from_numpy(u).cuda(), torch.empty(m.shape, dtype=torch.float64, device="cuda"), h1, 0.0).cpu().numpy()
        ref = operator.ax_local(u, P.G, P.B, P.D, h1, 0.0)
        # against the terms of the sums: some of these lines are nearly constant, and their derivatives cancel
        terms = operator.ax_local(np.abs(u), np.abs(P.G), P.B, np.abs(P.D), abs(h1), 0.0)
        d = np.sqrt(((w - ref) ** 2).reshape(E, -1).sum(1) / (terms ** 2).reshape(E, -1).sum(1))
        assert d.max() < AX_TOL, (h1, s, d)
    # the lines do what they are for: at N = 11 some sums of the tables times h1 pass 2^63
    assert max(sums) > (1.0 if N == 11 else 0.3)
