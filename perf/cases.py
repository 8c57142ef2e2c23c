"""Measured cases: the work that a program which uses this library has it do.

Each case is one call (or the pair of transfers) of the public Python binding on inputs of the
shapes of the library's workloads: the 2-D finite-difference problem at 63^2 to 511^2, the
spectral-element Poisson problem on perturbed boxes of 8 to 32^3 elements at orders 2 to 9,
single vectors and batches of right-hand sides, FP64 and the mixed form.  ``exact`` evaluates
the same mathematics in plain torch FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2210_03179_gb300 as cm

# Upper bounds of the spectrum of S A per level: of this mesh family by order, and of the FD
# operators (five-point on the finest grid, Galerkin nine-point below).  A program that solves a
# sequence of problems on such grids passes its bounds instead of having them estimated anew.
LMAX_SEM = {1: 2.05, 2: 2.25, 3: 2.35, 4: 2.45, 5: 2.55, 6: 2.65, 7: 2.75, 8: 2.85, 9: 2.95}
LMAX_FD_FINE, LMAX_FD_COARSE = 2.0, 1.5

# Optimized 4th-kind weights (arXiv 2210.03179, Table 5) of the orders used here.
BETAS = {
    1: (1.12500000000000,),
    2: (1.02387287570313, 1.26408905371085),
    3: (1.00842544782028, 1.08867839208730, 1.33753125909618),
    4: (1.00391310427285, 1.04035811188593, 1.14863498546254, 1.38268869241000),
    6: (1.00128517255940, 1.01304293035233, 1.04678215124113, 1.11616489419675, 1.23829020218444,
        1.43524297106744),
}


def listed():
    return [
        # the model problem's preconditioner: 63 x 63, symmetric order-2 cycle, plain 4th kind
        {"name": "fd_vcycle_63", "op": "fd_vcycle", "m": 63, "kind": "4th", "k": 2, "sided": "symmetric"},
        # smoothing on a large grid by the 1st kind, starting from the current iterate
        {"name": "fd_smooth_511", "op": "fd_smooth", "m": 511, "kind": "1st", "order": 4, "zero": False},
        # weight tuning: objective and gradient of three cycles for 16 errors on 255 x 255
        {"name": "fd_grad_255", "op": "fd_grad", "m": 255, "k": 4, "nrhs": 16, "steps": 3},
        # an uneven mesh's operator in the mixed form's precision
        {"name": "sem_ax_f32_n9_e12", "op": "sem_ax", "nex": 12, "ney": 12, "nez": 12, "N": 9, "f32": True},
        # the outer Krylov product at the benchmark size
        {"name": "sem_ax_f64_n7_e32", "op": "sem_ax", "nex": 32, "ney": 32, "nez": 32, "N": 7, "f32": False},
        # the mixed form's pre-smoother at the benchmark size: order 6 from a zero guess
        {"name": "sem_smooth_f32_e32", "op": "sem_smooth", "nex": 32, "ney": 32, "nez": 32, "N": 7, "f32": True,
         "kind": "opt4th", "order": 6, "zero": True},
        # post-smoothing in FP64 on a ragged medium box
        {"name": "sem_smooth_f64_ragged", "op": "sem_smooth", "nex": 15, "ney": 18, "nez": 13, "N": 7, "f32": False,
         "kind": "opt4th", "order": 2, "zero": False},
        # p-multigrid restriction and interpolation of the mixed form
        {"name": "sem_transfer_f32", "op": "sem_transfer", "nex": 32, "ney": 28, "nez": 30, "N": 7, "Nc": 3,
         "f32": True},
        # the coarse problem of the benchmark size, FP32 preconditioner inside the FP64 CG
        {"name": "sem_coarse_e32", "op": "sem_coarse", "nex": 32, "ney": 32, "nez": 32, "mixed": True},
        # one FP64 cycle of the medium workload
        {"name": "sem_vcycle_f64_e16", "op": "sem_vcycle", "nex": 16, "ney": 16, "nez": 16, "N": 7, "kind": "opt4th",
         "k": 2, "sided": "one-sided"},
        # a whole mixed-precision solve at the benchmark size
        {"name": "sem_solve_mixed_e32", "op": "sem_solve", "nex": 32, "ney": 32, "nez": 32, "N": 7, "kind": "opt4th",
         "k": 3, "sided": "one-sided", "mixed": True, "nrhs": 1},
        # a batch of solves that share one operator
        {"name": "sem_solve_batch64_e8", "op": "sem_solve", "nex": 8, "ney": 8, "nez": 8, "N": 7, "kind": "opt4th",
         "k": 3, "sided": "one-sided", "mixed": True, "nrhs": 64},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, elements_max):
    """Element counts of a box of about a logarithmically spread number of elements, any parity."""
    e = _log(rng, 40, elements_max)
    side = e ** (1.0 / 3.0)
    nex, ney = (max(2, round(side * rng.uniform(0.75, 1.25))) for _ in range(2))
    nez = max(2, min(round(e / (nex * ney)), int(elements_max / (nex * ney))))
    return {"nex": nex, "ney": ney, "nez": nez}


def _grid(rng, lo, hi):
    """An FD grid that coarsens by two down to 8 .. 15 intervals."""
    q = rng.choice([8, 9, 10, 11, 12, 13, 14, 15])
    p = [p for p in range(1, 8) if lo <= q * 2 ** p - 1 <= hi]
    return q * 2 ** rng.choice(p) - 1


def draw(rng):
    op = rng.choice(["fd_vcycle", "fd_smooth", "fd_grad", "sem_ax", "sem_ax", "sem_smooth", "sem_smooth",
                     "sem_transfer", "sem_coarse", "sem_vcycle", "sem_solve", "sem_solve"])
    cycle = {"kind": rng.choice(["opt4th", "opt4th", "4th", "1st"]), "k": rng.choice([1, 2, 3]),
             "sided": rng.choice(["one-sided", "symmetric"])}
    if op == "fd_vcycle":
        return {"op": op, "m": _grid(rng, 31, 511), **cycle}
    if op == "fd_smooth":
        return {"op": op, "m": _grid(rng, 31, 511), "kind": cycle["kind"], "order": rng.choice([1, 2, 3, 4, 6]),
                "zero": rng.random() < 0.5}
    if op == "fd_grad":
        return {"op": op, "m": _grid(rng, 31, 255), "k": rng.choice([2, 3, 4]), "nrhs": rng.randint(1, 16),
                "steps": rng.choice([1, 2, 3])}
    f32 = rng.random() < 0.6
    if op == "sem_ax":
        N = rng.choice([3, 4, 5, 6, 7, 7, 8, 9])
        return {"op": op, **_box(rng, 1.6e7 / (N + 1) ** 3), "N": N, "f32": f32}
    if op == "sem_smooth":
        N = rng.choice([3, 5, 7, 7, 9])
        return {"op": op, **_box(rng, 1.6e7 / (N + 1) ** 3 * (1.0 if f32 else 0.25)), "N": N, "f32": f32,
                "kind": cycle["kind"], "order": rng.choice([1, 2, 3, 4, 6]), "zero": rng.random() < 0.5}
    if op == "sem_transfer":
        N, Nc = rng.choice([(7, 3), (7, 3), (3, 1), (7, 5), (5, 3), (9, 3)])
        return {"op": op, **_box(rng, 1.6e7 / (N + 1) ** 3), "N": N, "Nc": Nc, "f32": f32}
    if op == "sem_coarse":
        return {"op": op, **_box(rng, 32 ** 3), "mixed": rng.random() < 0.6}
    if op == "sem_vcycle":
        N = rng.choice([5, 7, 7, 9])
        return {"op": op, **_box(rng, 4e6 / (N + 1) ** 3), "N": N, **cycle}
    nrhs = rng.choice([1, 1, 1, 2, 5, 16])
    return {"op": op, **_box(rng, 2e6 / 512 / nrhs if nrhs > 1 else 8e6 / 512), "N": rng.choice([5, 7, 7]), **cycle,
            "mixed": rng.random() < 0.7, "nrhs": nrhs}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _vector(seed, *shape):
    g = torch.Generator(device=_device()).manual_seed(1000003 * seed + 17)
    return torch.rand(*shape, generator=g, dtype=torch.float64, device=_device()) * 2.0 - 1.0


def _vertices(nex, ney, nez, seed):
    """Vertices of the unit box, interior ones moved by up to a tenth of an element and bent."""
    rng = np.random.default_rng(seed + 7)
    Z, Y, X = np.meshgrid(*(np.linspace(0.0, 1.0, k + 1) for k in (nez, ney, nex)), indexing="ij")
    v = np.stack([X, Y, Z], axis=-1)
    inner = np.zeros(v.shape[:3] + (1,))
    inner[1:-1, 1:-1, 1:-1] = 1.0
    v = v + inner * rng.uniform(-0.1, 0.1, v.shape) / np.array([nex, ney, nez])
    bump = 0.05 * np.prod(np.sin(np.pi * v), axis=-1, keepdims=True)
    return np.ascontiguousarray(v + inner * bump)


def _orders(case):
    if case["op"] == "sem_coarse":
        return (3, 1)
    if case["op"] == "sem_transfer":
        return (case["N"], case["Nc"]) if case["Nc"] == 1 else (case["N"], case["Nc"], 1)
    if case["op"] in ("sem_vcycle", "sem_solve"):
        return (case["N"], 3, 1)
    return (case["N"], 1)


def _fd_sizes(m):
    sizes = [m]
    while sizes[-1] > 15:
        sizes.append((sizes[-1] + 1) // 2 - 1)
    return sizes


def _solver(case, seed):
    kw = {"kind": case.get("kind", "opt4th"), "order": case.get("k", 2), "sided": case.get("sided", "symmetric")}
    if case["op"].startswith("fd"):
        if case["op"] == "fd_grad":
            kw["kind"] = "4th"
        levels = len(_fd_sizes(case["m"])) - 1
        return cm.Solver("fd2d", m=case["m"], coarsening=2, coarsest=15,
                         lmax=[LMAX_FD_FINE] + [LMAX_FD_COARSE] * (levels - 1), **kw)
    mixed = case.get("mixed", case.get("f32", False))
    orders = _orders(case)
    return cm.Solver("sem", verts=_vertices(case["nex"], case["ney"], case["nez"], seed), orders=orders,
                     prec="mixed" if mixed else "fp64", lmax=[LMAX_SEM[N] for N in orders[:-1]], **kw)


def _nodes(case, N):
    return (case["nex"] * N + 1) * (case["ney"] * N + 1) * (case["nez"] * N + 1)


def _inputs(case, seed):
    op = case["op"]
    if op in ("fd_vcycle", "fd_smooth"):
        n = case["m"] ** 2
        return {"b": _vector(seed, n), "x0": _vector(seed + 500, n)}
    if op == "fd_grad":
        return {"b": _vector(seed, case["nrhs"], case["m"] ** 2)}
    if op == "sem_coarse":
        return {"b": _vector(seed, _nodes(case, 1))}
    n = _nodes(case, case["N"])
    if op == "sem_solve" and case["nrhs"] > 1:
        return {"b": _vector(seed, case["nrhs"], n)}
    out = {"b": _vector(seed, n)}
    if op == "sem_smooth":
        # an iterate: zero on the boundary
        inner = torch.zeros(*(case[k] * case["N"] + 1 for k in ("nez", "ney", "nex")), dtype=torch.float64,
                            device=_device())
        inner[1:-1, 1:-1, 1:-1] = 1.0
        out["x0"] = _vector(seed + 500, n) * inner.reshape(-1)
    if op == "sem_transfer":
        out["zc"] = _vector(seed + 500, _nodes(case, case["Nc"]))
    if case.get("f32"):
        out = {k: v.float() for k, v in out.items()}
    return out


def prepare(case, seed):
    s = _solver(case, seed)
    st = {"case": case, "solver": s, "dt": cm.CHEBMG_F32 if case.get("f32") else cm.CHEBMG_F64, **_inputs(case, seed)}
    st["out"] = torch.zeros_like(st["b"])
    if case["op"] == "sem_transfer":
        st["rc"] = torch.zeros_like(st["zc"])
    return st


def run(st):
    case, ctx, b, out, dt = st["case"], st["solver"].ctx, st["b"], st["out"], st["dt"]
    op = case["op"]
    if op in ("fd_vcycle", "sem_vcycle"):
        cm.chebmg_vcycle(ctx, b, out)
        return out
    if op in ("fd_smooth", "sem_smooth"):
        if not case["zero"]:
            out.copy_(st["x0"])
        cm.chebmg_smooth(ctx, 0, dt, b, out, case["order"], case["zero"])
        return out
    if op == "fd_grad":
        f, gb, gs, fe = cm.chebmg_cycle_error_grad(ctx, b, [1.0] * case["k"], 1.0, case["steps"])
        return {"f": np.float64(f), "betas": np.array(gb), "scale": np.float64(gs), "each": np.array(fe)}
    if op == "sem_ax":
        cm.chebmg_apply_A(ctx, 0, dt, b, out)
        return out
    if op == "sem_transfer":
        cm.chebmg_restrict(ctx, 0, dt, b, st["rc"])
        cm.chebmg_prolong(ctx, 0, dt, st["zc"], out)
        return {"coarse": st["rc"], "fine": out}
    if op == "sem_coarse":
        cm.chebmg_coarse_solve(ctx, b, out)
        return out
    if case["nrhs"] == 1:
        cm.chebmg_pcg_solve(ctx, b, out, 1e-8, 500)
    else:
        cm.chebmg_pcg_solve_batched(ctx, b, out, 1e-8, 500)
    return out


# ---------------------------------------------------------------------------
# bytes and operations
# ---------------------------------------------------------------------------
def _ax_work(case, N, nrhs=1):
    """Operations of one operator application and the bytes of its geometric factors, in values."""
    Q, E = N + 1, case["nex"] * case["ney"] * case["nez"]
    return nrhs * E * Q ** 3 * (12 * Q + 15), 6 * E * Q ** 3


def work(case):
    op = case["op"]
    w = 4 if case.get("f32") else 8
    if op == "fd_vcycle":
        steps = case["k"] * 2
        return {"bytes": 2 * 8 * case["m"] ** 2, "flops": (steps + 1) * 16 * case["m"] ** 2 * 4 / 3}
    if op == "fd_smooth":
        return {"bytes": (2 if case["zero"] else 3) * 8 * case["m"] ** 2, "flops": case["order"] * 16 * case["m"] ** 2}
    if op == "fd_grad":
        n = case["nrhs"] * case["m"] ** 2
        return {"bytes": 8 * n, "flops": case["steps"] * (2 * case["k"] + 2) * 16 * 4 / 3 * n * 4}
    E = case["nex"] * case["ney"] * case["nez"]
    if op == "sem_coarse":
        n = _nodes(case, 1)
        return {"bytes": 8 * n * (27 + 3), "flops": 100 * 54 * n}
    n = _nodes(case, case["N"])
    if op == "sem_transfer":
        Q, P = case["N"] + 1, case["Nc"] + 1
        nc = _nodes(case, case["Nc"])
        return {"bytes": 2 * w * (n + nc), "flops": 2 * 2 * E * (P * P * P * Q + P * P * Q * Q + P * Q ** 3)}
    flops, factors = _ax_work(case, case["N"])
    if op == "sem_ax":
        return {"bytes": w * (factors + 2 * n), "flops": flops}
    if op == "sem_smooth":
        ax = case["order"] - (1 if case["zero"] else 0)
        return {"bytes": w * (factors * max(ax, 1) + (3 if case["zero"] else 4) * n),
                "flops": ax * flops + case["order"] * 8 * n}
    cycle = 2 * case["k"] + (1 if case["sided"] == "symmetric" else 0)
    if op == "sem_vcycle":
        return {"bytes": 8 * (factors * cycle + 3 * n), "flops": cycle * flops}
    its, nrhs = 10, case["nrhs"]
    wv = 4 if case["mixed"] else 8
    return {"bytes": its * (cycle * wv * factors + 8 * factors) + 2 * 8 * n * nrhs,
            "flops": its * (cycle + 1) * flops * nrhs}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _gll(N):
    """Gauss-Lobatto-Legendre points, weights and differentiation matrix of order N."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):     # polish the interior points: P' has simple roots
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    return x, w, _basis(x, x, True)


def _basis(nodes, at, derivative=False):
    """Lagrange basis on `nodes` (or its derivative) at the points `at`: [point][basis]."""
    n = len(nodes)
    out = np.zeros((len(at), n))
    for j in range(n):
        others = np.delete(nodes, j)
        poly = np.prod(nodes[j] - others)
        for a, y in enumerate(at):
            if derivative:
                out[a, j] = sum(np.prod(np.delete(y - others, q)) for q in range(n - 1)) / poly
            else:
                out[a, j] = np.prod(y - others) / poly
    return out


class _SemLevel:
    def __init__(self, case, N, verts):
        dev = _device()
        nex, ney, nez = case["nex"], case["ney"], case["nez"]
        self.N, self.lmax = N, LMAX_SEM[N]
        x, w, D = _gll(N)
        self.x = x
        self.D = torch.tensor(D, device=dev)
        Q = N + 1
        NX, NY, NZ = nex * N + 1, ney * N + 1, nez * N + 1
        self.n = NX * NY * NZ
        ex, ey, ez = (torch.arange(k, device=dev) for k in (nex, ney, nez))
        l = torch.arange(Q, device=dev)
        gz = (ez[:, None] * N + l).view(nez, 1, 1, Q, 1, 1)
        gy = (ey[:, None] * N + l).view(1, ney, 1, 1, Q, 1)
        gx = (ex[:, None] * N + l).view(1, 1, nex, 1, 1, Q)
        self.ids = ((gz * NY + gy) * NX + gx).reshape(-1)
        free = torch.zeros(NZ, NY, NX, dtype=torch.float64, device=dev)
        free[1:-1, 1:-1, 1:-1] = 1.0
        self.free = free.reshape(-1)
        E = nex * ney * nez
        self.shape = (E, Q, Q, Q)
        # coordinates of the trilinear elements at the GLL points, and their derivatives
        v = torch.tensor(verts, device=dev)
        c = torch.stack([torch.stack([torch.stack([v[k:nez + k, j:ney + j, i:nex + i] for i in (0, 1)], 3)
                                      for j in (0, 1)], 3) for k in (0, 1)], 3)     # [ez,ey,ex,k,j,i,3]
        c = c.reshape(E, 2, 2, 2, 3)
        H = torch.tensor(np.stack([(1 - x) / 2, (1 + x) / 2], 1), device=dev)       # [Q,2]
        X = torch.einsum("ck,bj,ai,ekjix->xecba", H, H, H, c)
        J = torch.stack([torch.stack(self._grad(X[a]), 0) for a in range(3)], 0)    # dx_a / dr_m
        cof = torch.stack([torch.stack([J[(a + 1) % 3, (m + 1) % 3] * J[(a + 2) % 3, (m + 2) % 3]
                                        - J[(a + 1) % 3, (m + 2) % 3] * J[(a + 2) % 3, (m + 1) % 3]
                                        for m in range(3)]) for a in range(3)])     # det * dr_m / dx_a
        det = sum(J[0, m] * cof[0, m] for m in range(3))
        wt = torch.tensor(w, device=dev)
        scale = wt.view(1, Q, 1, 1) * wt.view(1, 1, Q, 1) * wt.view(1, 1, 1, Q) / det
        self.G = [[sum(cof[a, m] * cof[a, q] for a in range(3)) * scale if q >= m else None for q in range(3)]
                  for m in range(3)]
        del X, J, cof
        # diagonal: the pure terms contract with D^2, the mixed ones only meet at the point itself
        D2, Dd = self.D ** 2, torch.diagonal(self.D)
        dia = (torch.einsum("la,ecbl->ecba", D2, self.G[0][0]) + torch.einsum("lb,ecla->ecba", D2, self.G[1][1])
               + torch.einsum("lc,elba->ecba", D2, self.G[2][2]))
        r, s, t = Dd.view(1, 1, 1, Q), Dd.view(1, 1, Q, 1), Dd.view(1, Q, 1, 1)
        dia = dia + 2 * (self.G[0][1] * r * s + self.G[0][2] * r * t + self.G[1][2] * s * t)
        diag = torch.zeros(self.n, dtype=torch.float64, device=dev).index_add_(0, self.ids, dia.reshape(-1))
        self.S = self.free / diag
        self.W = self.free / torch.zeros_like(diag).index_add_(0, self.ids, torch.ones_like(dia.reshape(-1)))

    def _grad(self, u):
        return (torch.einsum("al,...cbl->...cba", self.D, u), torch.einsum("bl,...cla->...cba", self.D, u),
                torch.einsum("cl,...lba->...cba", self.D, u))

    def gather(self, u):
        return u[:, self.ids].view(-1, *self.shape)

    def scatter(self, v):
        v = v.reshape(v.shape[0], -1)
        return torch.zeros(v.shape[0], self.n, dtype=v.dtype, device=v.device).index_add_(1, self.ids, v)

    def A(self, u):
        g = self._grad(self.gather(u * self.free))
        G = self.G
        w = [sum(G[min(m, q)][max(m, q)] * g[q] for q in range(3)) for m in range(3)]
        y = (torch.einsum("la,...cbl->...cba", self.D, w[0]) + torch.einsum("lb,...cla->...cba", self.D, w[1])
             + torch.einsum("lc,...lba->...cba", self.D, w[2]))
        return self.scatter(y) * self.free

    def link(self, C):
        """Interpolation from the coarser level C."""
        self.J, self.C = torch.tensor(_basis(C.x, self.x), device=self.ids.device), C

    def R(self, r):
        e = self.gather(r * self.W)
        e = torch.einsum("la,...cbl->...cba", self.J, e)
        e = torch.einsum("lb,...cla->...cba", self.J, e)
        e = torch.einsum("lc,...lba->...cba", self.J, e)
        return self.C.scatter(e) * self.C.free

    def P(self, z):
        e = self.C.gather(z * self.C.free)
        e = torch.einsum("al,...cbl->...cba", self.J, e)
        e = torch.einsum("bl,...cla->...cba", self.J, e)
        e = torch.einsum("cl,...lba->...cba", self.J, e)
        out = torch.zeros(z.shape[0], self.n, dtype=z.dtype, device=z.device)
        out[:, self.ids] = e.reshape(z.shape[0], -1)
        return out * self.free

    def solve(self, b):
        """A^{-1} b by Jacobi-PCG to far below the library's coarse tolerance."""
        r = b * self.free
        x, z = torch.zeros_like(r), self.S * r
        p, rz = z.clone(), (r * z).sum(1, keepdim=True)
        stop = 1e-28 * (r * r).sum(1, keepdim=True)
        for it in range(2000):
            q = self.A(p)
            alpha = rz / (p * q).sum(1, keepdim=True).clamp_min(1e-300)
            x, r = x + alpha * p, r - alpha * q
            if it % 8 == 7 and bool(((r * r).sum(1, keepdim=True) <= stop).all()):
                break
            z = self.S * r
            old, rz = rz, (r * z).sum(1, keepdim=True)
            p = z + rz / old.clamp_min(1e-300) * p
        return x


class _FdLevel:
    def __init__(self, m, st, lmax):
        self.m, self.st, self.lmax, self.n = m, st, lmax, m * m
        self.S = 1.0 / st[1][1]

    def A(self, u):
        m = self.m
        p = torch.nn.functional.pad(u.view(-1, m, m), (1, 1, 1, 1))
        y = 0
        for a in range(3):
            for b in range(3):
                if self.st[a][b] != 0.0:
                    y = y + self.st[a][b] * p[:, a:a + m, b:b + m]
        return y.reshape(u.shape[0], -1)

    def link(self, C):
        self.C = C
        P = np.zeros((self.m, C.m))
        for i in range(C.m):
            P[2 * i:2 * i + 3, i] = (0.5, 1.0, 0.5)
        self.J = torch.tensor(P, device=_device())

    def R(self, r):
        return torch.einsum("ya,xb,nyx->nab", self.J, self.J, r.view(-1, self.m, self.m)).reshape(r.shape[0], -1)

    def P(self, z):
        c = self.C.m
        return torch.einsum("ya,xb,nab->nyx", self.J, self.J, z.view(-1, c, c)).reshape(z.shape[0], -1)

    def solve(self, b):
        dense = self.A(torch.eye(self.n, dtype=torch.float64, device=b.device))
        return torch.linalg.solve(dense, b.T).T


def _fd_levels(m):
    h = 1.0 / (m + 1)
    K, M = np.array([-1.0, 2.0, -1.0]), np.array([0.0, 1.0, 0.0])
    st = (np.outer(M, K) + np.outer(K, M)) / h ** 2
    sizes = _fd_sizes(m)
    out = []
    for j, size in enumerate(sizes):
        out.append(_FdLevel(size, st.tolist(), LMAX_FD_FINE if j == 0 else LMAX_FD_COARSE))
        # Galerkin product with the bilinear hat: one coarse column on a patch without boundary
        hat = np.zeros((11, 11))
        hat[4:7, 4:7] = np.outer([0.5, 1.0, 0.5], [0.5, 1.0, 0.5])
        Ah = np.zeros_like(hat)
        for a in (-1, 0, 1):
            for b in (-1, 0, 1):
                Ah += st[a + 1, b + 1] * np.roll(hat, (a, b), (0, 1))
        st = np.array([[(np.roll(hat, (2 * a, 2 * b), (0, 1)) * Ah).sum() for b in (-1, 0, 1)] for a in (-1, 0, 1)])
    for F, C in zip(out, out[1:]):
        F.link(C)
    return out


def _smooth(L, b, x, order, kind, betas=None, scale=1.0):
    lam = L.lmax * scale
    r = b if x is None else b - L.A(x)
    x = torch.zeros_like(b) if x is None else x
    if kind == "1st":
        theta, delta = 0.55 * lam, 0.45 * lam
        sigma = theta / delta
        rho = 1.0 / sigma
        r = L.S * r
        d = r / theta
        for _ in range(1, order):
            x, r = x + d, r - L.S * L.A(d)
            new = 1.0 / (2.0 * sigma - rho)
            d = new * rho * d + 2.0 * new / delta * r
            rho = new
        return x + d
    if betas is None:
        betas = BETAS[order] if kind == "opt4th" else (1.0,) * order
    d = 4.0 / (3.0 * lam) * (L.S * r)
    for i in range(1, order):
        x, r = x + betas[i - 1] * d, r - L.A(d)
        d = (2 * i - 1) / (2 * i + 3) * d + (8 * i + 4) / ((2 * i + 3) * lam) * (L.S * r)
    return x + betas[order - 1] * d


def _cycle(levels, b, kind, k, sided, betas=None, scale=1.0):
    L = levels[0]
    if len(levels) == 1:
        return L.solve(b)
    if isinstance(L, _SemLevel):
        b = b * L.free
    x = _smooth(L, b, None, 2 * k if sided == "one-sided" else k, kind, betas, scale)
    x = x + L.P(_cycle(levels[1:], L.R(b - L.A(x)), kind, k, sided, betas, scale))
    return x if sided == "one-sided" else _smooth(L, b, x, k, kind, betas, scale)


def _solve(levels, b, case):
    """Flexible CG from zero, every right-hand side frozen once it has converged."""
    dot = lambda u, v: (u * v).sum(1, keepdim=True)  # noqa: E731
    M = lambda v: _cycle(levels, v, case["kind"], case["k"], case["sided"])  # noqa: E731
    r = b * levels[0].free
    x, stop = torch.zeros_like(r), 1e-16 * dot(r, r)
    z = M(r)
    p, rz = z, dot(z, r)
    active = torch.ones_like(rz)
    for _ in range(500):
        q = levels[0].A(p)
        alpha = active * rz / dot(p, q)
        x, r = x + alpha * p, r - alpha * q
        active = active * (dot(r, r) > stop)
        if not bool(active.any()):
            break
        z = M(r)
        beta = -alpha * dot(z, q) / rz
        rz = dot(z, r)
        p = z + beta * p
    return x


def exact(case, seed):
    inp = {k: torch.atleast_2d(v.double()) for k, v in _inputs(case, seed).items()}
    op, b = case["op"], inp["b"]
    if op.startswith("fd"):
        levels = _fd_levels(case["m"])
        if op == "fd_vcycle":
            return _cycle(levels, b, case["kind"], case["k"], case["sided"])[0]
        if op == "fd_smooth":
            return _smooth(levels[0], b, None if case["zero"] else inp["x0"], case["order"], case["kind"])[0]
        betas = [torch.ones((), dtype=torch.float64, device=b.device, requires_grad=True) for _ in range(case["k"])]
        scale = torch.ones((), dtype=torch.float64, device=b.device, requires_grad=True)
        e = b
        for _ in range(case["steps"]):
            e = e - _cycle(levels, levels[0].A(e), "4th", case["k"], "symmetric", betas, scale)
        each = (e * e).sum(1) / (b * b).sum(1)
        f = each.mean()
        g = torch.autograd.grad(f, [*betas, scale])
        return {"f": np.float64(f.item()), "betas": np.array([v.item() for v in g[:-1]]),
                "scale": np.float64(g[-1].item()), "each": each.detach().cpu().numpy()}
    verts = _vertices(case["nex"], case["ney"], case["nez"], seed)
    if op == "sem_coarse":
        return _SemLevel(case, 1, verts).solve(b)[0]
    if op in ("sem_vcycle", "sem_solve"):
        levels = [_SemLevel(case, N, verts) for N in _orders(case)]
        for F, C in zip(levels, levels[1:]):
            F.link(C)
        if op == "sem_vcycle":
            return _cycle(levels, b, case["kind"], case["k"], case["sided"])[0]
        x = _solve(levels, b, case)
        return x if case["nrhs"] > 1 else x[0]
    L = _SemLevel(case, case["N"], verts)
    if op == "sem_ax":
        return L.A(b)[0]
    if op == "sem_smooth":
        return _smooth(L, b * L.free, None if case["zero"] else inp["x0"], case["order"], case["kind"])[0]
    L.link(_SemLevel(case, case["Nc"], verts))
    return {"coarse": L.R(b)[0], "fine": L.P(inp["zc"])[0]}
