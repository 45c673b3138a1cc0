"""GLL bases, geometric factors and the local operator in long double, for tests that compare two FP64 results."""

import numpy as np

from oracle import gll, operator
from oracle.geometry import reference_gradient

LD = np.longdouble


def basis(N):
    """Points, weights and derivative matrix."""
    n = N + 1
    x = gll.nodes_weights(N)[0].astype(LD)

    def legendre(x):
        q, p = x * 0 + 1, x
        for j in range(1, N):
            q, p = p, ((2 * j + 1) * x * p - j * q) / LD(j + 1)
        return p, q

    for _ in range(5):  # Newton on P_{N-1} - x P_N, whose derivative is -(N + 1) P_N
        p, q = legendre(x[1:-1])
        x[1:-1] += (q - x[1:-1] * p) / ((N + 1) * p)
    x = (x - x[::-1]) / 2
    w = 2 / (N * (N + 1) * legendre(x)[0] ** 2)
    D = np.zeros((n, n), LD)
    for i in range(n):
        for l in range(n):
            if l != i:
                k = [k for k in range(n) if k not in (i, l)]
                D[i, l] = np.prod((x[i] - x[k]) / (x[l] - x[k])) / (x[l] - x[i])
        D[i, i] = -D[i].sum()
    return x, w, D


def factors(N, xyz):
    """G [E, 6, n, n, n] (as oracle.geometry) and B of the coordinates xyz [E, 3, n, n, n]."""
    _, w, D = basis(N)
    X = xyz.astype(LD) - xyz[:, :, :1, :1, :1].astype(LD)
    J = [reference_gradient(D, X[:, c]) for c in range(3)]
    C = [[J[(a + 1) % 3][(b + 1) % 3] * J[(a + 2) % 3][(b + 2) % 3] - J[(a + 1) % 3][(b + 2) % 3] * J[(a + 2) % 3][(b + 1) % 3]
          for b in range(3)] for a in range(3)]
    det = sum(J[0][b] * C[0][b] for b in range(3))
    w3 = w[:, None, None] * w[:, None] * w
    G = [w3 / det * sum(C[a][p] * C[a][q] for a in range(3)) for p, q in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    return np.stack(G, 1), w3 * det


def ax(N, xyz, u, h1=1.0, h2=0.0):
    G, B = factors(N, xyz)
    return operator.ax_local(u.astype(LD), G, B, basis(N)[2], LD(h1), LD(h2))
