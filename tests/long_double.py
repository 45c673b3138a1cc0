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


def gl_basis(N):
    """Values and derivatives [m, n] of the GLL basis at the GL points, m = N - 1, and the GL weights."""
    from oracle import pressure
    x, m = basis(N)[0], N - 1
    z = pressure.gl_nodes_weights(m)[0].astype(LD)

    def legendre(z):
        q, p = z * 0 + 1, z
        for j in range(1, m):
            q, p = p, ((2 * j + 1) * z * p - j * q) / LD(j + 1)
        return p, m * (q - z * p) / (1 - z * z)

    for _ in range(5):
        p, dp = legendre(z)
        z = z - p / dp
    z = (z - z[::-1]) / 2
    rho = 2 / ((1 - z * z) * legendre(z)[1] ** 2)
    V, D = np.zeros((m, N + 1), LD), np.zeros((m, N + 1), LD)
    for l in range(N + 1):
        k = [k for k in range(N + 1) if k != l]
        for i in range(m):
            V[i, l] = np.prod((z[i] - x[k]) / (x[l] - x[k]))
            D[i, l] = sum(np.prod([(z[i] - x[q]) / (x[l] - x[q]) for q in k if q != r]) / (x[l] - x[r]) for r in k)
    return V, D, rho


def along(M, v, axis):
    return np.moveaxis(np.tensordot(M, v, axes=(1, axis)), 0, axis)


def div_factors(N, xyz):
    """F [E, 3 (b), 3 (a), m, m, m] (as oracle.pressure)."""
    V, D, rho = gl_basis(N)
    X = xyz.astype(LD) - xyz[:, :, :1, :1, :1].astype(LD)
    J = [[along(V if b != 2 else D, along(V if b != 1 else D, along(V if b != 0 else D, X[:, a], 3), 2), 1) for b in range(3)]
         for a in range(3)]
    adj = [[J[(a + 1) % 3][(b + 1) % 3] * J[(a + 2) % 3][(b + 2) % 3] - J[(a + 1) % 3][(b + 2) % 3] * J[(a + 2) % 3][(b + 1) % 3]
            for a in range(3)] for b in range(3)]
    return np.stack([np.stack(r, 1) for r in adj], 1) * (rho[:, None, None] * rho[:, None] * rho)


def div(N, F, u):
    V, D, _ = gl_basis(N)
    return sum(F[:, b, a] * along(D if b == 2 else V, along(D if b == 1 else V, along(D if b == 0 else V, u[a], 3), 2), 1)
               for a in range(3) for b in range(3))


def grad(N, F, p):
    V, D, _ = gl_basis(N)
    return np.stack([sum(along((D if b == 2 else V).T, along((D if b == 1 else V).T, along((D if b == 0 else V).T, F[:, b, a] * p, 3), 2), 1)
                         for b in range(3)) for a in range(3)])
