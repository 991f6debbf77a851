"""The workloads whose speed is watched: what a user of the library has it do, through the binding.

Uniform cubes of n^3 cells (n = c 2^k with c = 1, 3 or 5) and adaptive octrees with the sinker
viscosity of the benchmark (Section 3.2): the level operator, the outer Stokes operator, the V-cycle
and the preconditioner on their own, whole solves, and a batch of solves. `exact` restates each
operator and the V-cycle in 64 bits with plain torch and numpy.
"""
from __future__ import annotations

import itertools

import numpy as np
import torch

from paper_1907_06696_gb300 import capi

DEV = "cuda"
DELTA, OMEGA, BETA = 200.0, 0.1, 10.0      # Section 3.2
CHEB_DEGREE, SCHUR_DEGREE, LANCZOS = 4, 5, 12

# Multiply-adds that one cell's velocity operator cannot do without: the element matrix is a sum of
# tensor products, so 1D transforms of 81 lines each way (4 and 5 operations a line) and about 230
# products in the basis where most of it is diagonal.
FLOPS_A = 2 * (81 * 9 + 230)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest level operator: a coarse multigrid level; launches and latency
        {"name": "vmult_f32_n16", "kind": "vmult", "n": 16, "prec": "f32", "sinkers": 4, "ratio": 1e4},
        # the level operator on the finest mesh of the largest benchmark configuration
        {"name": "vmult_f32_n128", "kind": "vmult", "n": 128, "prec": "f32", "sinkers": 16, "ratio": 1e6},
        # the outer Krylov operator [A B^T; B 0], FP64 vectors: a small odd size, and the benchmark's
        {"name": "stokes_n20", "kind": "stokes", "n": 20, "sinkers": 3, "ratio": 1e3},
        {"name": "stokes_n64", "kind": "stokes", "n": 64, "sinkers": 8, "ratio": 1e4},
        # one FP32 V-cycle, what the solver's preconditioner spends most of its time in: small and large
        {"name": "vcycle_f32_n24", "kind": "vcycle", "n": 24, "prec": "f32", "sinkers": 4, "ratio": 1e4},
        {"name": "vcycle_f32_n96", "kind": "vcycle", "n": 96, "prec": "f32", "sinkers": 8, "ratio": 1e4},
        # the FP64 V-cycle, the accurate option
        {"name": "vcycle_f64_n40", "kind": "vcycle", "n": 40, "prec": "f64", "sinkers": 5, "ratio": 1e4},
        # the whole block-triangular preconditioner (S_hat^-1, B^T, V-cycle) with the FP64 V-cycle
        {"name": "precondition_n48", "kind": "precondition", "n": 48, "sinkers": 8, "ratio": 1e4},
        # the outer operator on an adaptive mesh with hanging nodes
        {"name": "octree_stokes", "kind": "oct_stokes", "base": 3, "top": 8, "sinkers": 4, "ratio": 1e6},
        # a whole solve on an adaptive mesh (FP32 local-smoothing V-cycle, FGMRES)
        {"name": "octree_solve", "kind": "oct_solve", "base": 3, "top": 6, "sinkers": 3, "ratio": 1e4, "rtol": 1e-10},
        # the benchmark's solve: 64^3 cells, 8 sinkers, viscosity ratio 1e4, to more digits
        {"name": "solve_n64", "kind": "solve", "n": 64, "sinkers": 8, "ratio": 1e4, "rtol": 1e-10},
        # many small problems at once
        {"name": "batch_solve", "kind": "batch", "problems": 8, "ratio": 1e3, "rtol": 1e-10},
    ]


def _sizes(lo, hi):
    return [n for n in sorted({c << k for c in (1, 3, 5) for k in range(9)}) if lo <= n <= hi]


def draw(rng):
    """One more case of the same ranges; the sizes c 2^k (c = 1, 3, 5) are spread over their logarithm."""
    kind = rng.choice(["vmult", "vmult", "stokes", "stokes", "vcycle", "vcycle", "precondition", "oct_stokes",
                       "oct_solve", "solve", "batch"])
    case = {"kind": kind, "sinkers": rng.randint(1, 12), "ratio": round(10.0 ** rng.uniform(2.0, 4.5), 3)}
    if kind == "vmult":
        case["prec"] = rng.choice(["f32", "f32", "f64"])
        case["n"] = rng.choice(_sizes(8, 128 if case["prec"] == "f32" else 64))
    elif kind == "stokes":
        case["n"] = rng.choice(_sizes(8, 96))
    elif kind == "vcycle":
        case["prec"] = rng.choice(["f32", "f32", "f64"])
        case["n"] = rng.choice(_sizes(8, 96 if case["prec"] == "f32" else 48))
    elif kind == "precondition":
        case["n"] = rng.choice(_sizes(8, 48))
    elif kind == "oct_stokes":
        case.update(base=rng.randint(2, 3), top=rng.randint(5, 8), sinkers=rng.randint(1, 4))
    elif kind == "oct_solve":
        case.update(base=rng.randint(2, 3), top=rng.randint(4, 6), sinkers=rng.randint(1, 3), rtol=1e-10)
        case["ratio"] = min(case["ratio"], 1e4)
    elif kind == "solve":
        case.update(n=rng.choice(_sizes(8, 48)), rtol=1e-10)
        case["ratio"] = min(case["ratio"], 1e4)
    else:
        case.update(problems=rng.randint(2, 8), ratio=min(case["ratio"], 1e3), rtol=1e-10)
    return case


def _levels(n):
    k = 1
    while n % 2 == 0:
        n, k = n // 2, k + 1
    return k


# ------------------------------------------------------------------ inputs
def _centres(seed, count):
    return np.random.default_rng(1907 + 7919 * seed).uniform(0.2, 0.8, (count, 3))


def _mu(case):
    return case["ratio"] ** -0.5, case["ratio"] ** 0.5


def _vector(seed, size, dtype):
    """Noise whose size varies over the vector by two decades, as residuals beside viscosity jumps do."""
    g = torch.Generator(device=DEV).manual_seed(1000003 * seed + 17)
    v = torch.randn(size, generator=g, device=DEV, dtype=torch.float64)
    m = torch.arange(size, device=DEV, dtype=torch.float64) * (6.0 / size)
    return (v * 10.0 ** (2.0 * torch.sin(m) ** 2 - 1.0)).to(dtype)


def _octree_mesh(case):
    """Sinker centres and their maximum levels that an adaptive mesh was refined for: the mesh of a case
    stays while the sinkers (_oct_centres) move a little, as between the steps of a moving flow."""
    g = np.random.default_rng(1907 + 31 * case["top"] + case["sinkers"])
    lv = g.integers(case["top"] - 1, case["top"] + 1, case["sinkers"])
    lv[0] = case["top"]
    return g.uniform(0.2, 0.8, (case["sinkers"], 3)), lv.astype(np.int32)


def _oct_centres(case, seed):
    return _octree_mesh(case)[0] + np.random.default_rng(31 + 104729 * seed).uniform(-0.01, 0.01, (case["sinkers"], 3))


BATCH = (16, 20, 24)


def _batch(case, seed):
    """(n, centres) of the batch's problems."""
    g = np.random.default_rng(91 + 15485863 * seed)
    return [(BATCH[i % 3], g.uniform(0.2, 0.8, (int(g.integers(1, 9)), 3))) for i in range(case["problems"])]


def _dtype(case):
    return torch.float32 if case.get("prec") == "f32" else torch.float64


def prepare(case, seed):
    kind = case["kind"]
    lo, hi = _mu(case)
    st = {"case": case}
    if kind == "batch":
        st["ctx"] = [capi.stokes_setup(n, _levels(n), cen, lo, hi) for n, cen in _batch(case, seed)]
        st["up"] = [torch.zeros(c.n_u + c.n_p, dtype=torch.float64, device=DEV) for c in st["ctx"]]
        return st
    if kind.startswith("oct"):
        keys = capi.stokes_octree_sinker_mesh(case["base"], *_octree_mesh(case))
        ctx = capi.stokes_setup_octree(keys, 2, _oct_centres(case, seed), lo, hi)
    else:
        ctx = capi.stokes_setup(case["n"], _levels(case["n"]), _centres(seed, case["sinkers"]), lo, hi)
    st["ctx"] = ctx
    if kind in ("solve", "oct_solve"):
        st["up"] = torch.zeros(ctx.n_u + ctx.n_p, dtype=torch.float64, device=DEV)
        return st
    size = ctx.n_u + (0 if kind in ("vmult", "vcycle") else ctx.n_p)
    st["src"] = _vector(seed, size, _dtype(case))
    st["dst"] = torch.empty_like(st["src"])
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    prec = capi.STOKES_FP32 if case.get("prec") == "f32" else capi.STOKES_FP64
    if kind == "vmult":
        capi.stokes_vmult(ctx, -1, capi.BLOCK_A, prec, st["src"], st["dst"])
    elif kind in ("stokes", "oct_stokes"):
        capi.stokes_vmult(ctx, -1, capi.BLOCK_STOKES, capi.STOKES_FP64, st["src"], st["dst"])
    elif kind == "vcycle":
        capi.gmg_vcycle(ctx, prec, st["src"], st["dst"])
    elif kind == "precondition":
        capi.stokes_precondition(ctx, capi.STOKES_FP64, st["src"], st["dst"])
    elif kind in ("solve", "oct_solve"):
        st["up"].zero_()
        capi.stokes_solve(ctx, capi.STOKES_FP32, None, st["up"], rtol=case["rtol"])
        return st["up"]
    else:
        for up in st["up"]:
            up.zero_()
        capi.stokes_batch_solve(ctx, capi.STOKES_FP32, st["up"], rtol=case["rtol"])
        return st["up"]
    return st["dst"]


# ------------------------------------------------------------------ what a pass cannot do without
# Krylov iterations of a solve to 1e-10 that the counts below assume (8 sinkers, ratio 1e4), and the
# basis vectors that one of them reads and writes on average with a restart of 50, in two passes.
ITERATIONS, BASIS = 170, 2 * 25


def _n_u(n):
    return 3 * (2 * n + 1) ** 3


def _n_p(n):
    return (n + 1) ** 3


def _outer_work(n):
    return 8 * (2 * (_n_u(n) + _n_p(n)) + n ** 3), (FLOPS_A + 2 * 300) * n ** 3


def _vcycle_work(n, size):
    """Right-hand side and result on the finest level, inverse diagonal and viscosity of every level; per
    level 2 degree - 1 products of the smoothers, one of the residual, and the vector updates."""
    b, f = 2 * _n_u(n) * size, 0
    for _ in range(_levels(n) - 1):
        b += (_n_u(n) + n ** 3) * size
        f += 2 * CHEB_DEGREE * FLOPS_A * n ** 3 + 8 * CHEB_DEGREE * _n_u(n)
        n //= 2
    return b, f


def _iteration_work(n):
    vb, vf = _vcycle_work(n, 4)
    ob, of = _outer_work(n)
    size = _n_u(n) + _n_p(n)
    return vb + ob + 8 * (BASIS + 4) * size, vf + of + 2 * BASIS * size


def _oct_cells(case):
    """Leaves of such a mesh, roughly: each sinker's shell fills about this many cells per level."""
    shell = 8.0 * np.pi * 0.05 ** 2 * 0.07
    return int(8 ** case["base"] + case["sinkers"] * sum(shell * 8.0 ** (l - 0.5) for l in range(case["base"], case["top"] + 1)))


def work(case):
    kind = case["kind"]
    if kind == "vmult":
        s, n = (4 if case["prec"] == "f32" else 8), case["n"]
        return {"bytes": (2 * _n_u(n) + n ** 3) * s, "flops": FLOPS_A * n ** 3}
    if kind == "stokes":
        b, f = _outer_work(case["n"])
    elif kind == "vcycle":
        b, f = _vcycle_work(case["n"], 4 if case["prec"] == "f32" else 8)
    elif kind == "precondition":
        n = case["n"]
        b, f = _vcycle_work(n, 8)
        b, f = b + 8 * (3 * _n_p(n) + n ** 3), f + (SCHUR_DEGREE * 128 + 600) * n ** 3
    elif kind == "oct_stokes":
        cells = _oct_cells(case)
        b, f = 8 * 2 * 25 * cells + 4 * 35 * cells, (FLOPS_A + 600) * cells
    elif kind == "oct_solve":
        cells = _oct_cells(case)
        b = ITERATIONS * (8 * (BASIS + 8) * 25 + 4 * 35) * cells
        f = ITERATIONS * (2 * CHEB_DEGREE + 1) * FLOPS_A * cells
    elif kind == "solve":
        b, f = (ITERATIONS * v for v in _iteration_work(case["n"]))
    else:
        each = [_iteration_work(BATCH[i % 3]) for i in range(case["problems"])]
        b, f = (ITERATIONS * sum(e[k] for e in each) for k in (0, 1))
    return {"bytes": int(b), "flops": int(f)}


# ------------------------------------------------------------------ the same in 64 bits
_GP = np.array([0.5 - np.sqrt(15.0) / 10.0, 0.5, 0.5 + np.sqrt(15.0) / 10.0])
_GW = np.array([5.0, 8.0, 5.0]) / 18.0
_TRI = [(i, j, k) for k in range(3) for j in range(3) for i in range(3)]      # x fastest
_VERT = [(i, j, k) for k in range(2) for j in range(2) for i in range(2)]


def _q2(x):
    return np.stack([(2 * x - 1) * (x - 1), 4 * x * (1 - x), x * (2 * x - 1)], -1)


def _dq2(x):
    return np.stack([4 * x - 3, 4 - 8 * x, 4 * x - 1], -1)


def _element():
    """Reference-cell matrices: A (81 x 81), B moments (8 x 81: int d_c phi psi), pressure mass (8 x 8)."""
    V, D, P = _q2(_GP), _dq2(_GP), np.stack([1 - _GP, _GP], -1)
    A, R, Mp = np.zeros((3, 27, 3, 27)), np.zeros((8, 3, 27)), np.zeros((8, 8))
    for q in itertools.product(range(3), repeat=3):
        w = _GW[q[0]] * _GW[q[1]] * _GW[q[2]]
        grad = np.array([[np.prod([(D if d == a else V)[q[d], t[d]] for d in range(3)]) for t in _TRI] for a in range(3)])
        psi = np.array([np.prod([P[q[d], v[d]] for d in range(3)]) for v in _VERT])
        for c in range(3):
            A[c, :, c, :] += w * grad.T @ grad
            for d in range(3):   # row component c, column component d: d_d phi_row d_c phi_col
                A[c, :, d, :] += w * np.outer(grad[d], grad[c])
            R[:, c, :] += w * np.outer(psi, grad[c])
        Mp += w * np.outer(psi, psi)
    return [torch.tensor(m, dtype=torch.float64, device=DEV) for m in (A.reshape(81, 81), R.reshape(8, 81), Mp)]


def _cell_mu(lower, h, cen, lo, hi):
    """Harmonic mean of the sinker viscosity over the Gauss points of cells at `lower` (m, 3) of side h."""
    gp = torch.tensor(_GP, dtype=torch.float64, device=DEV)
    cen = torch.tensor(cen, dtype=torch.float64, device=DEV)
    inv = torch.zeros(lower.shape[0], dtype=torch.float64, device=DEV)
    for i, j, k in _TRI:
        x = lower + h * torch.stack([gp[i], gp[j], gp[k]])
        chi = torch.ones_like(inv)
        for c in cen:
            r = ((x - c) ** 2).sum(1).sqrt() - 0.5 * OMEGA
            chi *= 1.0 - torch.exp(-DELTA * r.clamp_min(0.0) ** 2)
        inv += _GW[i] * _GW[j] * _GW[k] / (chi * lo + (1.0 - chi) * hi)
    return 1.0 / inv


def _axis(n):
    return torch.arange(n, device=DEV)


class _Cube:
    """One uniform level: operators on component-blocked vectors, boundary rows the identity."""

    def __init__(self, n, mu, el):
        self.n, self.M, self.mu, (self.A, self.R, self.Mp) = n, 2 * n + 1, mu, el
        self.h, M = 1.0 / n, self.M
        c = _axis(n)
        cell = [x.reshape(-1) for x in torch.meshgrid(c, c, c, indexing="ij")][::-1]    # x fastest
        self.nodes = torch.stack([(2 * cell[0] + i) + M * ((2 * cell[1] + j) + M * (2 * cell[2] + k)) for i, j, k in _TRI], 1)
        self.verts = torch.stack([(cell[0] + i) + (n + 1) * ((cell[1] + j) + (n + 1) * (cell[2] + k)) for i, j, k in _VERT], 1)
        inner = ((_axis(M) > 0) & (_axis(M) < M - 1)).double()
        self.free = (inner[:, None, None] * inner[None, :, None] * inner[None, None, :]).reshape(-1)
        self.n_u, self.n_p = 3 * M ** 3, (n + 1) ** 3

    def _cells(self, u):
        u = u.reshape(3, -1) * self.free
        return torch.cat([u[c][self.nodes] for c in range(3)], 1)

    def _sum(self, y):
        out = torch.stack([torch.zeros(self.M ** 3, dtype=torch.float64, device=DEV).index_add_(
            0, self.nodes.reshape(-1), y[:, 27 * c:27 * c + 27].reshape(-1)) for c in range(3)])
        return out * self.free

    def apply(self, u):
        y = self._sum((self._cells(u) @ self.A.T) * (self.mu * self.h)[:, None])
        return (y + u.reshape(3, -1) * (1.0 - self.free)).reshape(-1)

    def bt(self, p):
        return self._sum(-self.h ** 2 * (p[self.verts] @ self.R)).reshape(-1)

    def b(self, u):
        y = -self.h ** 2 * (self._cells(u) @ self.R.T)
        return torch.zeros(self.n_p, dtype=torch.float64, device=DEV).index_add_(0, self.verts.reshape(-1), y.reshape(-1))

    def mass(self, p):
        y = (p[self.verts] @ self.Mp.T) * (self.h ** 3 / self.mu)[:, None]
        return torch.zeros(self.n_p, dtype=torch.float64, device=DEV).index_add_(0, self.verts.reshape(-1), y.reshape(-1))

    def inverse_diagonal(self):
        y = (self.mu * self.h)[:, None] * torch.diagonal(self.A)[None, :]
        d = self._sum(y)
        return torch.where(self.free.bool()[None, :], 1.0 / torch.where(d == 0, torch.ones_like(d), d), torch.zeros_like(d)).reshape(-1)


def _interpolation(nc):
    """1D Q2 embedding of nc cells into 2 nc: (4 nc + 1) x (2 nc + 1)."""
    P = np.zeros((4 * nc + 1, 2 * nc + 1))
    for f in range(4 * nc + 1):
        c = min(f // 4, nc - 1)
        P[f, 2 * c:2 * c + 3] = _q2(np.array((f - 4 * c) / 4.0))
    return torch.tensor(P, dtype=torch.float64, device=DEV)


def _along_axes(P, v, m):
    v = v.reshape(3, m, m, m)
    for ax in (1, 2, 3):
        v = torch.movedim(torch.tensordot(P, v, dims=([1], [ax])), 0, ax)
    return v.reshape(3, -1)


def _uniform01(seed, count):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) / 2.0 ** 53


class _Multigrid:
    def __init__(self, n, cen, lo, hi):
        el = _element()
        g = [x.reshape(-1) for x in torch.meshgrid(_axis(n), _axis(n), _axis(n), indexing="ij")][::-1]
        mu = _cell_mu(torch.stack(g, 1).double() / n, 1.0 / n, cen, lo, hi)
        self.lev = []
        for _ in range(_levels(n)):
            self.lev.insert(0, _Cube(n, mu, el))
            if n % 2 == 0:
                mu = mu.reshape(n // 2, 2, n // 2, 2, n // 2, 2).mean(dim=(1, 3, 5)).reshape(-1)
                n //= 2
        self.dinv = [L.inverse_diagonal() for L in self.lev]
        self.top = [0.0] + [1.2 * self._lanczos(l) for l in range(1, len(self.lev))]
        self.P = [None] + [_interpolation(L.n) for L in self.lev[:-1]]
        L0 = self.lev[0]
        free = torch.nonzero(L0.free.repeat(3)).reshape(-1)
        y = torch.eye(81, dtype=torch.float64, device=DEV)
        K = torch.zeros(L0.n_u, L0.n_u, dtype=torch.float64, device=DEV)
        dof = torch.cat([L0.nodes + c * L0.M ** 3 for c in range(3)], 1)
        for e in range(dof.shape[0]):
            K[dof[e][:, None], dof[e][None, :]] += L0.mu[e] * L0.h * (L0.A @ y)
        self.free0, self.K0 = free, K[free][:, free].cpu().numpy()

    def _lanczos(self, l):
        L, sq = self.lev[l], self.dinv[l].sqrt()
        v = torch.tensor(_uniform01(1907000 + l, L.n_u) - 0.5, device=DEV) * L.free.repeat(3)
        v, vp, beta, al, be = v / v.norm(), torch.zeros_like(v), 0.0, [], []
        for _ in range(LANCZOS):
            w = sq * L.apply(sq * v)
            al.append(float(w @ v))
            w = w - al[-1] * v - beta * vp
            beta = float(w.norm())
            if beta <= 1e-12 * abs(al[-1]):
                break
            be.append(beta)
            vp, v = v, w / beta
        T = np.diag(al) + np.diag(be[:len(al) - 1], 1) + np.diag(be[:len(al) - 1], -1)
        return float(np.linalg.eigvalsh(T)[-1])

    def _smooth(self, l, b, x):
        L, D, hi = self.lev[l], self.dinv[l], self.top[l]
        lo = hi / 15.0
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma = theta / delta
        rho = 1.0 / sigma
        d = D * (b if x is None else b - L.apply(x)) / theta
        x = d.clone() if x is None else x + d
        for _ in range(1, CHEB_DEGREE):
            new = 1.0 / (2.0 * sigma - rho)
            d = new * rho * d + 2.0 * new / delta * D * (b - L.apply(x))
            x, rho = x + d, new
        return x

    def _cycle(self, l, b):
        L = self.lev[l]
        if l == 0:
            x = torch.zeros_like(b)
            x[self.free0] = torch.tensor(np.linalg.solve(self.K0, b[self.free0].cpu().numpy()), device=DEV)
            return x
        C = self.lev[l - 1]
        x = self._smooth(l, b, None)
        r = _along_axes(self.P[l].T, (b - L.apply(x)) * L.free.repeat(3), L.M) * C.free
        e = self._cycle(l - 1, r.reshape(-1))
        return self._smooth(l, b, x + (_along_axes(self.P[l], e, C.M) * L.free).reshape(-1))

    def vcycle(self, rhs):
        f = self.lev[-1].free.repeat(3)
        return self._cycle(len(self.lev) - 1, rhs * f) + rhs * (1.0 - f)

    def schur(self, r):
        L = self.lev[-1]
        diag = torch.zeros(L.n_p, dtype=torch.float64, device=DEV).index_add_(
            0, L.verts.reshape(-1), ((L.h ** 3 / L.mu)[:, None] * torch.diagonal(L.Mp)[None, :]).reshape(-1))
        lo, hi = 1.0 / 8.0, 27.0 / 8.0
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma = theta / delta
        rho = 1.0 / sigma
        d = r / diag / theta
        z = d.clone()
        for _ in range(1, SCHUR_DEGREE):
            new = 1.0 / (2.0 * sigma - rho)
            d = new * rho * d + 2.0 * new / delta * (r - L.mass(z)) / diag
            z, rho = z + d, new
        return z

    def precondition(self, r):
        L = self.lev[-1]
        zp = -self.schur(r[L.n_u:])
        return torch.cat([self.vcycle(r[:L.n_u] - L.bt(zp)), zp])


# ---- adaptive meshes: leaves as rows (level, i, j, k); points on the lattice of half the finest cell
def _split(leaves, mark):
    kids = [np.concatenate([leaves[mark, :1] + 1, 2 * leaves[mark, 1:] + np.array(v)], 1) for v in _VERT]
    return np.concatenate([leaves[~mark]] + kids)


def _leaves(case):
    cen, top = _octree_mesh(case)
    n = 1 << case["base"]
    g = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)
    leaves = np.concatenate([np.full((len(g), 1), case["base"]), g], 1).astype(np.int64)
    while True:
        h = 2.0 ** -leaves[:, 0].astype(np.float64)
        a = leaves[:, 1:] * h[:, None]
        b = a + h[:, None]
        mark = np.zeros(len(leaves), bool)
        for c, t in zip(cen, top):
            near = np.maximum(np.maximum(a - c, c - b), 0.0)
            far = np.maximum(np.abs(c - a), np.abs(c - b))
            mark |= (leaves[:, 0] < t) & ((near ** 2).sum(1) < 0.07 ** 2) & ((far ** 2).sum(1) > 0.03 ** 2)
        if not mark.any():
            break
        leaves = _split(leaves, mark)
    while True:   # full 2:1 balance
        fine = leaves[:, 0].max()
        mark = np.zeros(len(leaves), bool)
        find = _finder(leaves, fine)
        size = 1 << (fine - leaves[:, 0])
        for d in itertools.product((-1, 0, 1), repeat=3):
            p = leaves[:, 1:] * size[:, None] + np.where(np.array(d) < 0, -1, np.where(np.array(d) > 0, size[:, None], 0))
            ok = ((p >= 0) & (p < (1 << fine))).all(1)
            at = find(p[ok])
            mark[at[leaves[at, 0] < leaves[ok, 0] - 1]] = True
        if not mark.any():
            break
        leaves = _split(leaves, mark)
    key = (leaves[:, 0] << 48) | (leaves[:, 3] << 32) | (leaves[:, 2] << 16) | leaves[:, 1]
    return leaves[np.argsort(key)]


def _morton(p):
    out = np.zeros(len(p), np.int64)
    for bit in range(16):
        for d in range(3):
            out |= ((p[:, d] >> bit) & 1) << (3 * bit + d)
    return out


def _finder(leaves, fine):
    """Cells of the finest level -> the leaf that holds them."""
    first = _morton(leaves[:, 1:] << (fine - leaves[:, 0])[:, None])
    order = np.argsort(first)
    first = first[order]
    return lambda p: order[np.searchsorted(first, _morton(p), side="right") - 1]


def _space(leaves, deg):
    """Points of the Q1 (deg 1) or Q2 (deg 2) space: (matrix leaves x locals -> active points, boundary)."""
    import scipy.sparse as sp
    fine = leaves[:, 0].max()
    top = np.int64(1) << (fine + 1)
    loc = _VERT if deg == 1 else _TRI
    S = np.int64(1) << (fine + 1 - leaves[:, 0])
    pts = np.stack([leaves[:, 1:] * S[:, None] + np.array(t) * (S // deg)[:, None] for t in loc], 1)
    keys, inv = np.unique(pts[..., 0] + (top + 1) * (pts[..., 1] + (top + 1) * pts[..., 2]), return_inverse=True)
    inv = inv.reshape(pts.shape[:2])
    p = np.stack([keys % (top + 1), keys // (top + 1) % (top + 1), keys // (top + 1) ** 2], 1)
    bnd = ((p == 0) | (p == top)).any(1)
    find, host = _finder(leaves, fine), np.full(len(p), -1)
    for d in itertools.product((-1, 0), repeat=3):      # the coarsest leaf that touches the point
        q = (p + np.array(d)) >> 1
        ok = ((q >= 0) & (q < (1 << fine))).all(1)
        at = find(q[ok])
        cur = host[ok]
        host[ok] = np.where((cur < 0) | (leaves[at, 0] < leaves[cur, 0]), at, cur)
    step = (S // deg)[host]
    hang = (p % step[:, None] != 0).any(1) & ~(bnd & (deg == 2))
    index = np.cumsum(~hang) - 1
    rows, cols, vals = [np.nonzero(~hang)[0]], [index[~hang]], [np.ones((~hang).sum())]
    at = host[hang]
    x = (p[hang] - leaves[at, 1:] * S[at][:, None]) / S[at][:, None]
    w1 = _q2(x) if deg == 2 else np.stack([1 - x, x], -1)
    for a, t in enumerate(loc):
        w = w1[:, 0, t[0]] * w1[:, 1, t[1]] * w1[:, 2, t[2]]
        rows.append(np.nonzero(hang)[0])
        cols.append(index[inv[at, a]])
        vals.append(w)
    rows, cols, vals = (np.concatenate(v) for v in (rows, cols, vals))
    keep = vals != 0.0
    C = sp.csr_matrix((vals[keep], (rows[keep], cols[keep])), shape=(len(p), int((~hang).sum())))
    return C[inv.reshape(-1)], bnd[~hang]


def _oct_stokes(case, seed):
    leaves = _leaves(case)
    h = 2.0 ** -leaves[:, 0].astype(np.float64)
    lo, hi = _mu(case)
    hd = torch.tensor(h, device=DEV)
    mu = _cell_mu(torch.tensor(leaves[:, 1:], device=DEV) * hd[:, None], hd[:, None], _oct_centres(case, seed), lo, hi).cpu().numpy()
    A, R, _ = (m.cpu().numpy() for m in _element())
    Cu, bnd = _space(leaves, 2)
    Cp, _ = _space(leaves, 1)
    nu, free = Cu.shape[1], (~bnd).astype(np.float64)
    x = _vector(seed, 3 * nu + Cp.shape[1], torch.float64).cpu().numpy()
    u, p = x[:3 * nu].reshape(3, nu), (Cp @ x[3 * nu:]).reshape(-1, 8)
    e = np.concatenate([(Cu @ (u[c] * free)).reshape(-1, 27) for c in range(3)], 1)
    y = (e @ A.T) * (mu * h)[:, None] - (h ** 2)[:, None] * (p @ R)
    out = [(Cu.T @ y[:, 27 * c:27 * c + 27].reshape(-1)) * free + u[c] * (1.0 - free) for c in range(3)]
    out.append(Cp.T @ (-(h ** 2)[:, None] * (e @ R.T)).reshape(-1))
    return np.concatenate(out)


def exact(case, seed):
    """None for the solves: reaching their tolerance again takes far longer than the solves themselves."""
    kind = case["kind"]
    if kind == "oct_stokes":
        return _oct_stokes(case, seed)
    if kind in ("oct_solve", "solve", "batch"):
        return None
    n = case["n"]
    size = _n_u(n) + (0 if kind in ("vmult", "vcycle") else _n_p(n))
    x = _vector(seed, size, _dtype(case)).double()
    lo, hi = _mu(case)
    cen = _centres(seed, case["sinkers"])
    if kind in ("vcycle", "precondition"):
        mg = _Multigrid(n, cen, lo, hi)
        return mg.vcycle(x) if kind == "vcycle" else mg.precondition(x)
    g = [v.reshape(-1) for v in torch.meshgrid(_axis(n), _axis(n), _axis(n), indexing="ij")][::-1]
    L = _Cube(n, _cell_mu(torch.stack(g, 1).double() / n, 1.0 / n, cen, lo, hi), _element())
    if kind == "vmult":
        return L.apply(x)
    u, p = x[:L.n_u], x[L.n_u:]
    free = L.free.repeat(3)
    return torch.cat([L.apply(u) + L.bt(p) * free, L.b(u)])
