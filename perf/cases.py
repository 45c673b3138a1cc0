"""What a program that uses this library spends its GPU time on, as measurable cases.

Each case is one call (or the two calls that belong together) of the Python binding on a mesh, a
preconditioner and fields that such a program keeps: a time step of the flow solver applies operators and
solves Helmholtz and pressure problems thousands of times on one mesh, so meshes and preconditioners are
made once per descriptor and kept, and every pass works on its own fields.

``exact`` evaluates the same operators, right-hand sides and solutions in FP64 with plain torch, from the
mesh's definition (box and O-grid pipe coordinates, GLL / GL bases) alone.
"""

import math
from collections import OrderedDict

import numpy as np
import torch

import paper_2109_03592_gb300 as sem

DEV = "cuda"
PIPES = [(2, 1), (4, 1), (4, 2), (8, 2), (8, 4), (16, 4)]  # (nc, nr) cross-sections


def _box(n, N, **kw):
    return dict(kind="box", nx=n[0], ny=n[1], nz=n[2], N=N, L=1.0, **kw)


def _pipe(nc, nr, nzp, N, L=8.0, **kw):
    return dict(kind="pipe", nc=nc, nr=nr, nzp=nzp, N=N, L=L, **kw)


def listed():
    return [
        # the smallest solve: the unit-cube Poisson problem, FP64 Jacobi-PCG to 1e-10 (latency of the iteration)
        dict(name="solve_fp64_box4_n7", op="solve", prec="fp64", h2=0.0, tol=1e-10, **_box((4, 4, 4), 7)),
        # the FP64 assembled operator at the strong-scaling limit of elements per GPU
        dict(name="apply_fp64_pipe4096_n7", op="apply", prec="fp64", h2=0.0, coef=False, **_pipe(8, 2, 32, 7)),
        # the same on a whole-GPU load: the headline FP64 operator
        dict(name="apply_fp64_pipe262144_n7", op="apply", prec="fp64", h2=0.0, coef=False, **_pipe(16, 4, 512, 7)),
        # variable-viscosity Helmholtz operator of even order on an odd box
        dict(name="apply_fp64_coef_box_n8", op="apply", prec="fp64", h2=10.0, coef=True, **_box((13, 17, 19), 8)),
        # the highest order, Helmholtz, FP64
        dict(name="apply_fp64_pipe16384_n11", op="apply", prec="fp64", h2=1.0, coef=False, **_pipe(16, 4, 32, 11, 1.0)),
        # the FP32 operator and gather-scatter of the mixed solver's inner iteration, whole-GPU load
        dict(name="apply_fp32_pipe262144_n7", op="apply", prec="fp32", h2=0.0, coef=False, **_pipe(16, 4, 512, 7)),
        # the same for one served Helmholtz request of ordinary size
        dict(name="apply_fp32_box1056_n9", op="apply", prec="fp32", h2=5.0, coef=False, **_box((8, 11, 12), 9)),
        # the consistent pressure operator in FP64 (the FP64 pressure solve, and every true residual of the mixed one)
        dict(name="pressure_fp64_pipe32768_n7", op="pressure", prec="fp64", **_pipe(16, 4, 64, 7, 1.0)),
        # the same in FP32: the mixed pressure solve's inner operator
        dict(name="pressure_fp32_pipe32768_n7", op="pressure", prec="fp32", **_pipe(16, 4, 64, 7, 1.0)),
        # one application of the overlapping Schwarz preconditioner inside the mixed solver
        dict(name="schwarz_fp32_pipe32768_n7", op="schwarz", prec="fp32", h2=0.0, **_pipe(16, 4, 64, 7, 1.0)),
        # a velocity step: the three components' Helmholtz solves as one mixed-precision batch
        dict(name="velocity_mixed_pipe4096_n7", op="velocity", prec="mixed", h2=1000.0, tol=1e-10, **_pipe(8, 2, 32, 7)),
        # one mixed-precision Helmholtz solve of a large served request
        dict(name="solve_mixed_pipe32768_n7", op="solve", prec="mixed", h2=1000.0, tol=1e-10, **_pipe(16, 4, 64, 7, 1.0)),
    ]


# most local points of a drawn case, by operation (fewest: the unit cube's 32,768)
_MOST = dict(apply=1 << 27, pressure=1 << 24, schwarz=1 << 24, velocity=1 << 21, solve=1 << 21)


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "pressure", "schwarz", "velocity", "solve"])
    # batches take the odd orders; the operators every order from 3 on
    N = rng.choice([5, 7, 9]) if op in ("velocity", "schwarz") else rng.choice([3, 5, 6, 7, 7, 8, 9, 10, 11])
    E = math.exp(rng.uniform(math.log(1 << 15), math.log(_MOST[op]))) / (N + 1) ** 3
    if rng.random() < 0.5:
        nx = max(2, int(E ** (1 / 3) * rng.uniform(0.75, 1.0)))
        ny = max(2, int(math.sqrt(E / nx) * rng.uniform(0.8, 1.0)))
        case = _box((nx, ny, max(2, int(E / (nx * ny)))), N)
    else:
        nc, nr = rng.choice([p for p in PIPES if p[0] * (p[0] + 4 * p[1]) * 3 <= E] or PIPES[:1])
        nzp = max(3, int(E / (nc * (nc + 4 * nr))))
        case = _pipe(nc, nr, nzp, N, round(nzp * 1.5 / nc, 4))  # elements about as long as they are wide
    case["op"] = op
    if op in ("apply", "pressure"):
        case["prec"] = rng.choice(["fp64", "fp64", "fp32"])
    elif op == "solve":
        case["prec"] = rng.choice(["fp64", "mixed"])
    else:
        case["prec"] = "fp32" if op == "schwarz" else "mixed"
    if op == "apply":
        case["h2"] = rng.choice([0.0, round(10.0 ** rng.uniform(-2, 2), 3)])
        case["coef"] = rng.random() < 0.25
    elif op == "schwarz":
        case["h2"] = rng.choice([0.0, round(10.0 ** rng.uniform(-2, 2), 3)])
    elif op in ("velocity", "solve"):
        case["h2"] = round(10.0 ** rng.uniform(2.5, 3.5), 2)  # h2 = b0 / dt of a time step
        case["tol"] = 1e-10
    return case


def _sizes(case):
    n = case["N"] + 1
    E = case["nx"] * case["ny"] * case["nz"] if case["kind"] == "box" else case["nc"] * (case["nc"] + 4 * case["nr"]) * case["nzp"]
    return E, n, E * n ** 3


def work(case):
    E, n, P = _sizes(case)
    op, size = case["op"], 8 if case["prec"] == "fp64" else 4
    h = bool(case.get("h2"))
    ax = 12 * n + 18 + 4 * h + 0.0  # contractions with D and D^T, the six factors, the mass term
    if op == "apply":  # u in, six factors (and B), w out
        return {"bytes": P * size * (8 + h), "flops": P * ax}
    if op == "pressure":  # p in, nine factors, the assembled mass, q out; D and D^T by shared 1D contractions
        m = n - 2
        line = 2 * m * n ** 3 + 3 * m * m * n * n + 3 * m ** 3 * n
        return {"bytes": E * size * (11 * m ** 3 + n ** 3), "flops": E * (2 * 6 * line + 36 * m ** 3)}
    if op == "schwarz":  # r in, z out, point flags; six 1D contractions
        return {"bytes": P * (2 * size + 1), "flops": P * (12 * n + 4)}
    # a solve cannot do without one operator application and its fields; iterations are not counted
    k = 3 if op == "velocity" else 1
    return {"bytes": P * (k * 16 + 8 * (6 + h) + 1), "flops": P * k * ax}


# ---- fields ------------------------------------------------------------------------------------------------


def _gll(N):
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # Newton on (1 - x^2) P_N'
        i = slice(1, -1)
        x[i] += (1 - x[i] ** 2) * P.deriv()(x[i]) / (N * (N + 1) * P(x[i]))
    x = (x - x[::-1]) / 2
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    return x, w


def _basis(x, at):
    """Values and derivatives of the Lagrange basis on nodes x at the points `at`: [len(at), len(x)] each."""
    d = x[:, None] - x[None, :]
    np.fill_diagonal(d, 1.0)
    c = d.prod(axis=1)
    D = c[:, None] / c[None, :] / d
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(axis=1))
    V = np.empty((len(at), len(x)))
    for q, z in enumerate(at):
        hit = np.isclose(z, x, rtol=0, atol=1e-14)
        t = 1.0 / (c * np.where(hit, 1.0, z - x))
        V[q] = hit.astype(float) if hit.any() else t / t.sum()
    return V, V @ D


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _section(case):
    """Pipe cross-section [e2d, 2, n, n] (j, i): x and y of every element's points."""
    N, nc, nr, a = case["N"], case["nc"], case["nr"], 0.5
    g = (_gll(N)[0] + 1) / 2
    out = []
    for ey in range(nc):
        for ex in range(nc):
            X, Y = a * (2 * (ex + g) / nc - 1), a * (2 * (ey + g) / nc - 1)
            out.append(np.stack(np.broadcast_arrays(X[None, :], Y[:, None])))
    lev = 1 - np.tanh(2.0 * (1 - np.arange(nr + 1) / nr)) / np.tanh(2.0)
    for q in range(4):
        co, si = [(1, 0), (0, 1), (-1, 0), (0, -1)][q]
        for r in range(nr):
            t = (lev[r] + (lev[r + 1] - lev[r]) * g)[None, :]
            for m in range(nc):
                s = (2 * (m + g) / nc - 1)[:, None]
                X = (1 - t) * a + t * np.cos(np.pi * s / 4)
                Y = (1 - t) * a * s + t * np.sin(np.pi * s / 4)
                out.append(np.stack([co * X - si * Y, si * X + co * Y]))
    return np.stack(out)


def _coords(case, e0, e1, sec=None):
    """Coordinates [e, 3, n, n, n] (k, j, i) of elements e0 .. e1."""
    n = case["N"] + 1
    g = (_t(_gll(case["N"])[0]) + 1) / 2
    e = torch.arange(e0, e1, device=DEV)
    out = torch.empty((e1 - e0, 3, n, n, n), dtype=torch.float64, device=DEV)
    if case["kind"] == "box":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        out[:, 0] = (((e % nx)[:, None] + g) / nx)[:, None, None, :]
        out[:, 1] = (((e // nx % ny)[:, None] + g) / ny)[:, None, :, None]
        out[:, 2] = (((e // (nx * ny))[:, None] + g) / nz)[:, :, None, None]
    else:
        sec = _t(_section(case)) if sec is None else sec
        out[:, :2] = sec[e % sec.shape[0]][:, :, None]
        out[:, 2] = (((e // sec.shape[0])[:, None] + g) * (case["L"] / case["nzp"]))[:, :, None, None]
    return out


def _chunks(case, most=1 << 23):
    E, n, _ = _sizes(case)
    sec = _t(_section(case)) if case["kind"] == "pipe" else None
    step = max(1, most // n ** 3)
    for e0 in range(0, E, step):
        e1 = min(E, e0 + step)
        yield e0, e1, _coords(case, e0, e1, sec)


def _wave(case, seed, waves=6, mean=0.0):
    """A seeded field of some long and some short waves, the same at all copies of a node: [E, n, n, n]."""
    E, n, _ = _sizes(case)
    rng = np.random.default_rng(seed)
    Lz = case["L"] if case["kind"] == "pipe" else 1.0
    top = [3 if q % 2 else 12 for q in range(waves)]
    k = np.array([[rng.integers(-t, t + 1) * math.pi, rng.integers(-t, t + 1) * math.pi, 2 * math.pi / Lz * rng.integers(-t, t + 1)] for t in top])
    amp, ph = rng.standard_normal(waves), rng.uniform(0, 2 * math.pi, waves)
    out = torch.empty((E, n, n, n), dtype=torch.float64, device=DEV)
    for e0, e1, X in _chunks(case):
        f = torch.full_like(X[:, 0], mean)
        for q in range(waves):
            f += amp[q] * torch.cos(k[q, 0] * X[:, 0] + k[q, 1] * X[:, 1] + k[q, 2] * X[:, 2] + ph[q])
        out[e0:e1] = f
    return out


def _coefficients(case):
    """h1 (viscosity) and h2 (density) of a variable-property step, or (None, None)."""
    if not case.get("coef"):
        return None, None
    return 1.0 + 0.04 * _wave(case, 901), 1.0 + 0.03 * _wave(case, 902)


def _pressure_field(case, seed):
    E, n, _ = _sizes(case)
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    p = torch.randn((E,) + (n - 2,) * 3, generator=g, dtype=torch.float64, device=DEV)
    return p if case["prec"] == "fp64" else p.float()


# ---- what a program keeps ----------------------------------------------------------------------------------

_kept = OrderedDict()  # descriptor -> (mesh, {h2: preconditioner}, points)
_KEPT_POINTS = 230_000_000


def _keep(case):
    key = tuple(case.get(k) for k in ("kind", "N", "nx", "ny", "nz", "nc", "nr", "nzp", "L", "coef"))
    if key not in _kept:
        P = _sizes(case)[2]
        while _kept and sum(v[2] for v in _kept.values()) + P > _KEPT_POINTS:
            _kept.popitem(last=False)
        d = {k: case[k] for k in ("kind", "N", "nx", "ny", "nz", "nc", "nr", "nzp", "L") if k in case}
        mesh = sem.Mesh(d)
        h1, h2 = _coefficients(case)
        if h1 is not None:
            mesh.set_coefficients(h1, h2)
        _kept[key] = (mesh, {}, P)
    _kept.move_to_end(key)
    return _kept[key]


def prepare(case, seed):
    mesh, precs, _ = _keep(case)
    op, st = case["op"], dict(case=case, mesh=mesh)
    if op == "apply":
        u = _wave(case, seed)
        st["u"] = u if case["prec"] == "fp64" else u.float()
        st["w"] = torch.empty_like(st["u"])
    elif op == "pressure":
        st["p"] = _pressure_field(case, seed)
        st["q"] = torch.empty_like(st["p"])
        st["work"] = torch.empty(3 * mesh.n_local, dtype=st["p"].dtype, device=DEV)
    elif op == "schwarz":
        h2 = case["h2"]
        if h2 not in precs:
            precs[h2] = sem.Schwarz(mesh, h2=h2)
        st["sw"] = precs[h2]
        b = mesh.rhs(_wave(case, seed), torch.empty(mesh.shape, dtype=torch.float64, device=DEV))
        st["r"] = (b / b.norm()).float()
        st["z"] = torch.empty_like(st["r"])
    else:
        st["b"] = [mesh.rhs(_wave(case, 3 * seed + c), torch.empty(mesh.shape, dtype=torch.float64, device=DEV))
                   for c in range(3 if op == "velocity" else 1)]
        st["x"] = [torch.zeros_like(b) for b in st["b"]]
    return st


def run(st):
    case, mesh = st["case"], st["mesh"]
    op, fp64 = case["op"], case["prec"] == "fp64"
    if op == "apply":
        if fp64:
            return mesh.apply(st["u"], st["w"], h1=1.0, h2=case["h2"])
        return mesh.gs(mesh.ax(st["u"], st["w"], h1=1.0, h2=case["h2"], prec=sem.FP32), prec=sem.FP32)
    if op == "pressure":
        return (mesh.pressure_apply if fp64 else mesh.pressure_apply_f32)(st["p"], st["q"], st["work"])
    if op == "schwarz":
        st["sw"].apply(st["r"], st["z"], prec=sem.FP32)
        return st["z"]
    for x in st["x"]:
        x.zero_()
    opts = dict(tol=case["tol"], h1=1.0, h2=case["h2"], prec=sem.FP64 if fp64 else sem.MIXED)
    if op == "velocity":
        sem.solve_batch([mesh] * 3, st["b"], st["x"], **opts)
    else:
        mesh.solve(st["b"][0], st["x"][0], **opts)
    return st["x"]


# ---- the same in 64 bits, with plain torch -----------------------------------------------------------------


class _Plain:
    """Numbering, mask and, element chunk by chunk, the operators of a case's mesh."""

    def __init__(self, case):
        self.case, N = case, case["N"]
        self.E, self.n, self.P = _sizes(case)
        x, w = _gll(N)
        self.D, self.w = _t(_basis(x, x)[1]), _t(w)
        n, l = self.n, torch.arange(self.n, device=DEV)
        e = torch.arange(self.E, device=DEV)
        if case["kind"] == "box":
            nx, ny, nz = case["nx"], case["ny"], case["nz"]
            a = ((e % nx)[:, None] * N + l)[:, None, None, :]
            b = ((e // nx % ny)[:, None] * N + l)[:, None, :, None]
            c = ((e // (nx * ny))[:, None] * N + l)[:, :, None, None]
            self.ids = (a + (nx * N + 1) * (b + (ny * N + 1) * c)).reshape(-1)
            self.nodes = (nx * N + 1) * (ny * N + 1) * (nz * N + 1)
            wall = (a == 0) | (a == nx * N) | (b == 0) | (b == ny * N) | (c == 0) | (c == nz * N)
        else:
            sec = _section(case)
            key = np.floor(sec * 1e5 + 0.37).astype(np.int64)  # coincident points share it; distinct ones are > 1e-4 apart
            _, ids = np.unique(key[:, 0] * 10 ** 7 + key[:, 1], return_inverse=True)
            ids = torch.as_tensor(ids.reshape(sec.shape[0], 1, n, n), device=DEV)
            m, per = sec.shape[0], int(ids.max()) + 1
            z = ((e // m)[:, None] * N + l) % (case["nzp"] * N)
            self.ids = (ids[e % m] + per * z[:, :, None, None]).reshape(-1)
            self.nodes = per * case["nzp"] * N
            wall = torch.as_tensor(np.hypot(sec[:, 0], sec[:, 1]) > 1 - 1e-9, device=DEV)[e % m][:, None].expand(-1, n, -1, -1)
        self.free = torch.ones(self.nodes, dtype=torch.float64, device=DEV)
        self.free[self.ids[wall.expand(self.E, n, n, n).reshape(-1)]] = 0.0

    def add(self, v):
        """Sum over the copies of every node."""
        return torch.zeros(self.nodes, dtype=torch.float64, device=DEV).index_add_(0, self.ids, v.reshape(-1))

    def grad(self, A, B, C, v):
        """A along i, B along j, C along k."""
        v = torch.einsum("il,ekjl->ekji", A, v)
        v = torch.einsum("jl,ekli->ekji", B, v)
        return torch.einsum("kl,elji->ekji", C, v)

    def metric(self, X, I=None, D=None):
        """J = dx/dr [e, 3 (x), 3 (r), ...] at the nodes, or at the points of (I, D); its determinant and adjugate."""
        eye = torch.eye(self.n, dtype=torch.float64, device=DEV) if I is None else I
        D = self.D if D is None else D
        X = X - X[:, :, :1, :1, :1]
        J = torch.stack([torch.stack([self.grad(*(D if a == b else eye for a in range(3)), X[:, c]) for b in range(3)], 1) for c in range(3)], 1)
        adj = torch.stack([torch.stack([J[:, (a + 1) % 3, (b + 1) % 3] * J[:, (a + 2) % 3, (b + 2) % 3]
                                        - J[:, (a + 1) % 3, (b + 2) % 3] * J[:, (a + 2) % 3, (b + 1) % 3] for a in range(3)], 1) for b in range(3)], 1)
        det = (J[:, :, 0] * adj[:, 0]).sum(1)
        return det, adj

    def factors(self, X):
        det, adj = self.metric(X)
        W = self.w[:, None, None] * self.w[:, None] * self.w
        G = torch.einsum("eb...,ec...->ebc...", adj[:, :, 0], adj[:, :, 0])
        for a in (1, 2):
            G += torch.einsum("eb...,ec...->ebc...", adj[:, :, a], adj[:, :, a])
        return G * (W / det)[:, None, None], W * det

    def local(self, u, G, B, h1, h2):
        i = torch.eye(self.n, dtype=torch.float64, device=DEV)
        M = [[self.D if a == b else i for a in range(3)] for b in range(3)]
        g = [self.grad(*M[b], u) for b in range(3)]
        w = h2 * B * u if h2 is not None else torch.zeros_like(u)
        for b in range(3):
            q = h1 * sum(G[:, b, c] * g[c] for c in range(3))
            w = w + self.grad(*(m.T.contiguous() for m in M[b]), q)
        return w

    def over(self, f):
        """[E, n, n, n] of f(e0, e1, coordinates) over the element chunks."""
        out = torch.empty((self.E, self.n, self.n, self.n), dtype=torch.float64, device=DEV)
        for e0, e1, X in _chunks(self.case, 1 << 22):
            out[e0:e1] = f(e0, e1, X)
        return out

    def spread(self, v):
        return (v * self.free)[self.ids].reshape(self.E, self.n, self.n, self.n)


def _exact_apply(p, case, u):
    h1, h2 = _coefficients(case)

    def f(e0, e1, X):
        G, B = p.factors(X)
        s = case["h2"] * (1.0 if h2 is None else h2[e0:e1])
        return p.local(u[e0:e1], G, B, 1.0 if h1 is None else h1[e0:e1], s if case["h2"] else None)

    return p.spread(p.add(p.over(f)))


def _exact_solve(p, case, fields):
    """Jacobi CG on the global nodes, well below the case's tolerance."""
    G, B = zip(*(p.factors(X) for _, _, X in _chunks(case, 1 << 22)))
    G, B, h2 = torch.cat(G), torch.cat(B), case["h2"]
    D2 = p.D ** 2
    d = torch.einsum("li,ekjl->ekji", D2, G[:, 0, 0]) + torch.einsum("lj,ekli->ekji", D2, G[:, 1, 1]) + torch.einsum("lk,elji->ekji", D2, G[:, 2, 2])
    inv = p.free / p.add(d + h2 * B)
    out = []
    for f in fields:
        b = p.add(B * f) * p.free
        x, r = torch.zeros_like(b), b.clone()
        z = inv * r
        q, rho, rr0 = z.clone(), r @ z, float(r @ r)
        for it in range(600):
            w = p.add(p.local(p.spread(q), G, B, 1.0, h2)) * p.free
            a = rho / (q @ w)
            x += a * q
            r -= a * w
            if it % 8 == 0 and float(r @ r) <= 1e-27 * rr0:
                break
            z = inv * r
            new = r @ z
            q, rho = z + (new / rho) * q, new
        out.append(p.spread(x))
    return out


def _exact_pressure(p, case, v):
    x, _ = _gll(case["N"])
    z, rho = np.polynomial.legendre.leggauss(case["N"] - 1)
    I, D = (_t(a) for a in _basis(x, z))
    rho = _t(rho)
    R = rho[:, None, None] * rho[:, None] * rho
    mass = p.add(p.over(lambda e0, e1, X: p.factors(X)[1]))
    C = [[D if a == b else I for a in range(3)] for b in range(3)]
    CT = [[m.T.contiguous() for m in c] for c in C]
    q = torch.zeros_like(v)
    for a in range(3):
        u = p.over(lambda e0, e1, X: _grad_t(p, CT, R * p.metric(X, I, D)[1][:, :, a], v[e0:e1]))
        u = p.spread(p.add(u) / mass)
        for e0, e1, X in _chunks(case, 1 << 22):
            F = R * p.metric(X, I, D)[1][:, :, a]
            q[e0:e1] += sum(F[:, b] * p.grad(*C[b], u[e0:e1]) for b in range(3))
    return q


def _grad_t(p, CT, F, v):
    return sum(p.grad(*CT[b], F[:, b] * v) for b in range(3))


def exact(case, seed):
    op = case["op"]
    if op == "schwarz":  # the local solves' eigenvectors are the library's own choice
        return None
    p = _Plain(case)
    if op == "apply":
        u = _wave(case, seed)
        return _exact_apply(p, case, u if case["prec"] == "fp64" else u.float().double())
    if op == "pressure":
        return _exact_pressure(p, case, _pressure_field(case, seed).double())
    return _exact_solve(p, case, [_wave(case, 3 * seed + c) for c in range(3 if op == "velocity" else 1)])
