"""The work a program has this library do, as measurable cases.

Operators (`sem_apply`, `sem_ax` + `sem_dssum`, `sem_apply_global`) are what
every Krylov iteration and every explicit step spends its time in; the solves
(`sem_cg_solve`, `sem_batch_solve`, `sem_gmres_solve` with the Schwarz
preconditioner, and the differentiable Helmholtz solve) are the calls a flow
solver makes per time step.  Meshes are boxes [0, 2 pi]^3, deformed as in the
operator-throughput workload unless a case says otherwise.

`exact` computes the same results in plain FP64 torch from its own mesh.
"""
import math
import random

import numpy as np
import torch

import paper_2107_01243_gb300 as sem
from paper_2107_01243_gb300 import autograd

TWO_PI = 2.0 * math.pi
DEFORM = 0.1
# the largest solve exact() repeats in plain torch (local points)
EXACT_SOLVE_POINTS = 600_000


def listed():
    return [
        # one matvec of the smallest mesh in use (64 elements): launches and latency
        dict(name="apply-f64-n7-e64", kind="apply", dtype="f64", nelx=4, nely=4, nelz=4, N=7,
             h2=0.0),
        # the operator-throughput workload, 16.8 M points, both precisions
        dict(name="apply-f64-n7-e32768", kind="apply", dtype="f64", nelx=32, nely=32, nelz=32,
             N=7, h2=0.0),
        dict(name="apply-f32-n7-e32768", kind="apply", dtype="f32", nelx=32, nely=32, nelz=32,
             N=7, h2=0.0),
        # an even order (odd points per direction) on an uneven box, Helmholtz, FP32
        dict(name="apply-f32-n6-e24453", kind="apply", dtype="f32", nelx=19, nely=33, nelz=39,
             N=6, h2=1.5),
        # an even order in FP64 (IEEE arithmetic), a medium box of odd sides
        dict(name="apply-f64-n6-e7429", kind="apply", dtype="f64", nelx=17, nely=19, nelz=23,
             N=6, h2=0.0),
        # the two-call form of the operator: element operator, then gather-scatter
        dict(name="ax-dssum-f64-n5-e9177", kind="ax_dssum", dtype="f64", nelx=19, nely=21,
             nelz=23, N=5, h2=0.0),
        # the operator on unique-dof vectors (what mixed and batched solves iterate with)
        dict(name="apply-global-f32-n9-e16767", kind="apply_global", dtype="f32", nelx=23,
             nely=27, nelz=27, N=9, h2=2.0),
        # a small Poisson solve in FP64: 64 elements of the unit cube, to 1e-10
        dict(name="solve-f64-n7-e64", kind="solve", precision="f64", nelx=4, nely=4, nelz=4, N=7,
             h2=0.0, tol=1e-10),
        # a large Poisson solve, FP32 inner iterations and FP64 refinement
        dict(name="solve-mixed-n7-e32768", kind="solve", precision="mixed", nelx=32, nely=32,
             nelz=32, N=7, h2=0.0, tol=1e-10),
        # many small Helmholtz problems of several orders in one call
        dict(name="batch-16-e512-4096", kind="batch", problems=16, e_lo=512, e_hi=4096,
             tol=1e-10),
        # the pressure solve: GMRES(10) with the two-level Schwarz preconditioner
        dict(name="pressure-mixed-n7-e13824", kind="pressure", precision="mixed", nelx=24,
             nely=24, nelz=24, N=7, tol=1e-10),
        # forward and adjoint Helmholtz solve with a per-point coefficient, and its gradient
        dict(name="adjoint-f64-n7-e512", kind="adjoint", nelx=8, nely=8, nelz=8, N=7, h2=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, e_lo, e_hi, N, points=17_000_000):
    """Sides of an uneven box of about e elements (e log-uniform), at most `points` points."""
    e = min(_log_int(rng, e_lo, e_hi), max(e_lo, points // (N + 1) ** 3))
    side = e ** (1.0 / 3.0)
    nx = max(1, int(round(side * rng.uniform(0.7, 1.2))))
    ny = max(1, int(round(side * rng.uniform(0.8, 1.2))))
    nz = max(1, int(e / (nx * ny)))
    return dict(nelx=nx, nely=ny, nelz=nz)


def draw(rng: random.Random):
    kind = rng.choices(["apply", "ax_dssum", "apply_global", "solve", "batch", "pressure",
                        "adjoint"], [6, 2, 3, 3, 1, 2, 1])[0]
    if kind in ("apply", "ax_dssum"):
        N = rng.randint(3, 9)
        return dict(kind=kind, dtype=rng.choice(["f64", "f32"]), N=N,
                    h2=rng.choice([0.0, round(rng.uniform(0.1, 10.0), 3)]),
                    **_box(rng, 27, 32768, N))
    if kind == "apply_global":
        N = rng.choice([3, 5, 7, 9])
        return dict(kind=kind, dtype="f32", N=N, h2=rng.choice([0.0, round(rng.uniform(0.1, 10.0), 3)]),
                    **_box(rng, 27, 32768, N))
    if kind == "solve":
        N = rng.choice([5, 6, 7, 8, 9])
        return dict(kind=kind, precision=rng.choice(["f64", "mixed"]), N=N, tol=1e-10,
                    h2=rng.choice([0.0, round(rng.uniform(0.1, 10.0), 3)]),
                    **_box(rng, 27, 4096, N, 4_000_000))
    if kind == "batch":
        lo = _log_int(rng, 64, 512)
        return dict(kind=kind, problems=rng.randint(3, 16), e_lo=lo, e_hi=lo * rng.randint(2, 8),
                    tol=1e-10)
    if kind == "pressure":
        N = rng.choice([5, 7, 9])
        return dict(kind=kind, precision=rng.choice(["f64", "mixed"]), N=N, tol=1e-10,
                    **_box(rng, 64, 4096, N, 4_000_000))
    N = rng.choice([5, 6, 7])
    return dict(kind=kind, N=N, h2=round(rng.uniform(0.5, 2.0), 3), **_box(rng, 27, 512, N))


# ---------------------------------------------------------------- inputs
def _nel(case):
    return case["nelx"], case["nely"], case["nelz"]


def _points(nel, N):
    return nel[0] * nel[1] * nel[2] * (N + 1) ** 3


def _global_points(nel, N):
    return math.prod(N * n + 1 for n in nel)


def _is_cube(case):
    """The small Poisson solve runs on the undeformed unit cube."""
    return case["kind"] == "solve" and max(_nel(case)) <= 4


def _mesh(case):
    return ((1.0, 1.0, 1.0), 0.0) if _is_cube(case) else ((TWO_PI, TWO_PI, TWO_PI), DEFORM)


def _uniform(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, generator=g, device="cuda", dtype=dtype) * 2.0 - 1.0


def _smooth(seed, x, y, z):
    """Smooth random field: eight Fourier modes, a ~ N(0,1), k in {1..4}^3."""
    r = np.random.default_rng(seed)
    f = torch.zeros_like(x)
    for _ in range(8):
        a, k, phi = r.standard_normal(), r.integers(1, 5, 3), r.uniform(0.0, TWO_PI)
        f += float(a) * torch.sin(float(k[0]) * x + float(k[1]) * y + float(k[2]) * z + float(phi))
    return f


def _batch_problems(case, seed):
    """The batch's boxes and orders are part of the case; lambda and the sources follow the seed."""
    shape, r = np.random.default_rng(1000 + case["problems"] + case["e_lo"]), np.random.default_rng(seed)
    out = []
    for p in range(case["problems"]):
        e = int(shape.integers(case["e_lo"], case["e_hi"] + 1))
        side = e ** (1.0 / 3.0)
        nx, ny = max(1, int(side)), max(1, int(round(side)))
        out.append(dict(nel=(nx, ny, max(1, e // (nx * ny))), N=int(shape.choice([5, 7, 9])),
                        lam=float(r.uniform(0.1, 10.0)), seed=seed * 100 + p))
    return out


def _coords(h):
    return [sem.sem_get_field(h, f, torch.empty(h.n_local, dtype=torch.float64, device="cuda"))
            for f in (sem.SEM_FIELD_X, sem.SEM_FIELD_Y, sem.SEM_FIELD_Z)]


def _source(h, seed):
    """b = mask o QQ^T (B f) of a smooth random source f."""
    b = torch.empty(h.n_local, dtype=torch.float64, device="cuda")
    return sem.sem_rhs(h, _smooth(seed, *_coords(h)), b)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = _batch_problems(case, seed)
        hs = [sem.sem_setup(p["nel"], p["N"], length=(TWO_PI,) * 3, deform=DEFORM) for p in probs]
        bs = [_source(h, p["seed"]) for h, p in zip(hs, probs)]
        return dict(case=case, hs=hs, batch=sem.sem_batch_create(hs), bs=bs,
                    xs=[torch.empty_like(b) for b in bs], h2s=[p["lam"] for p in probs])
    length, deform = _mesh(case)
    h = sem.sem_setup(_nel(case), case["N"], length=length, deform=deform)
    st = dict(case=case, h=h)
    if kind in ("apply", "ax_dssum"):
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        st["u"] = _uniform(h.n_local, dtype, seed)
        st["w"] = torch.empty_like(st["u"])
    elif kind == "apply_global":
        st["u"] = _uniform(h.n_global, torch.float32, seed)
        st["w"] = torch.empty_like(st["u"])
    else:
        st["b"] = _source(h, seed)
        st["x"] = torch.empty_like(st["b"])
    if kind == "pressure":
        st["m"] = sem.sem_schwarz_create(h)
    if kind == "adjoint":
        xyz = _coords(h)
        st["h1"] = 1.0 + 0.5 * torch.tanh(_smooth(seed + 1, *xyz))
        st["target"] = _smooth(seed + 2, *xyz)
        mult = sem.sem_get_field(h, sem.SEM_FIELD_MULT, torch.empty_like(st["b"]))
        st["weight"] = 1.0 / mult
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        return sem.sem_apply(st["h"], st["u"], st["w"], h2=case["h2"])
    if kind == "ax_dssum":
        sem.sem_ax(st["h"], st["u"], st["w"], h2=case["h2"])
        return sem.sem_dssum(st["h"], st["w"])
    if kind == "apply_global":
        return sem.sem_apply_global(st["h"], st["u"], st["w"], h2=case["h2"])
    if kind == "solve":
        prec = sem.SEM_SOLVE_F64 if case["precision"] == "f64" else sem.SEM_SOLVE_MIXED
        sem.sem_cg_solve(st["h"], st["b"], st["x"], h2=case["h2"], tol=case["tol"], precision=prec)
        return st["x"]
    if kind == "batch":
        sem.sem_batch_solve(st["batch"], st["bs"], st["xs"], [1.0] * len(st["xs"]), st["h2s"],
                            tol=case["tol"])
        return st["xs"]
    if kind == "pressure":
        prec = sem.SEM_SOLVE_F64 if case["precision"] == "f64" else sem.SEM_SOLVE_MIXED
        sem.sem_gmres_solve(st["h"], st["b"], st["x"], tol=case["tol"], restart=10,
                            precond=st["m"], precision=prec)
        return st["x"]
    h1 = st["h1"].detach().requires_grad_(True)
    u = autograd.helmholtz_solve(h1, st["b"], st["h"], h2=case["h2"])
    loss = ((u - st["target"]) ** 2 * st["weight"]).sum()
    (g,) = torch.autograd.grad(loss, h1)
    return u.detach(), g


# ---------------------------------------------------------------- work
def _iterations(nel, N, h2, tol):
    """Jacobi-PCG iterations, to about a factor of two: they grow with the lattice points
    along a side and the digits asked for; a mass term takes the smoothest modes away."""
    per = 0.35 if h2 == 0.0 else 0.25
    return max(20, int(per * N * max(nel) * math.sqrt(N / 2.0) * math.log10(1.0 / tol) / 4.0))


def _operator_work(nel, N, size, h2=0.0):
    """u read, w written, six geometric factors (and the mass) read; sum-factorised flops."""
    n, words = _points(nel, N), 8 + (1 if h2 else 0)
    return n * words * size, n * (12 * (N + 1) + 11 + (3 if h2 else 0))


def _solve_work(nel, N, h2, tol, mixed):
    """Per iteration the operator and six vectors read or written on the unique points."""
    it, size = _iterations(nel, N, h2, tol), 4 if mixed else 8
    by, fl = _operator_work(nel, N, size, h2)
    vec = _global_points(nel, N)
    return it * (by + 6 * vec * size), it * (fl + 12 * vec)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_solve_work(p["nel"], p["N"], p["lam"], case["tol"], True)
                 for p in _batch_problems(case, 1)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    nel, N = _nel(case), case["N"]
    if kind in ("apply", "ax_dssum"):
        by, fl = _operator_work(nel, N, 8 if case["dtype"] == "f64" else 4, case["h2"])
    elif kind == "apply_global":
        n, g = _points(nel, N), _global_points(nel, N)
        by, fl = _operator_work(nel, N, 4, case["h2"])
        by += (g - n) * 2 * 4
    elif kind == "solve":
        by, fl = _solve_work(nel, N, case["h2"], case["tol"], case["precision"] == "mixed")
    elif kind == "pressure":
        # about 45 iterations; per iteration the operator, the local solves (six line
        # contractions on (N + 3)^3 points) and the Krylov vectors
        size = 4 if case["precision"] == "mixed" else 8
        b1, f1 = _operator_work(nel, N, size)
        g, e = _global_points(nel, N), math.prod(nel)
        by, fl = 45 * (b1 + 14 * g * size), 45 * (f1 + e * 12 * (N + 3) ** 4 + 40 * g)
    else:
        b1, f1 = _solve_work(nel, N, case["h2"], 1e-12, False)
        n = _points(nel, N)
        by, fl = 2 * b1 + 9 * 8 * n, 2 * f1 + n * (12 * (N + 1) + 15)
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------------------- the same in plain FP64 torch
def _gll(N):
    leg = np.polynomial.legendre
    c = np.eye(N + 1)[N]
    d1, d2 = leg.legder(c), leg.legder(c, 2)
    inner = np.sort(np.real(leg.legroots(d1))) if N > 1 else np.zeros(0)
    for _ in range(3):
        inner = inner - leg.legval(inner, d1) / leg.legval(inner, d2) if N > 1 else inner
    xi = np.concatenate(([-1.0], inner, [1.0]))
    ln = leg.legval(xi, c)
    diff = xi[:, None] - xi[None, :] + np.eye(N + 1)
    D = ln[:, None] / (ln[None, :] * diff)
    np.fill_diagonal(D, 0.0)
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return xi, 2.0 / (N * (N + 1) * ln ** 2), D


class _Plain:
    """Mesh, geometric factors and assembled operator on one box, all Dirichlet faces."""

    def __init__(self, nel, N, length, deform):
        dev, P = "cuda", N + 1
        xi, w, D = _gll(N)
        self.D = torch.tensor(D, device=dev)
        e = torch.arange(math.prod(nel), device=dev)
        at = [e % nel[0], (e // nel[0]) % nel[1], e // (nel[0] * nel[1])]
        shape = [(1, 1, 1, P), (1, 1, P, 1), (1, P, 1, 1)]
        t, idx = torch.tensor((xi + 1.0) / 2.0, device=dev), torch.arange(P, device=dev)
        full = (e.numel(), P, P, P)
        c, lat, self.mask = [], [], torch.ones(full, dtype=torch.float64, device=dev)
        for d in range(3):
            a = at[d].view(-1, 1, 1, 1)
            c.append(((a + t.view(shape[d])) * (length[d] / nel[d])).expand(full))
            lat.append(N * a + idx.view(shape[d]))
            self.mask = self.mask * ((lat[d] > 0) & (lat[d] < N * nel[d]))
        sx, sy, sz = (torch.sin(v) for v in c)
        self.xyz = [c[0] + deform * sy * sz, c[1] + deform * sz * sx, c[2] + deform * sx * sy]
        gx, gy = N * nel[0] + 1, N * nel[1] + 1
        self.gid = (lat[0] + gx * (lat[1] + gy * lat[2])).expand(full).reshape(-1)
        self.n_global = _global_points(nel, N)
        self.mult = self.gather(torch.ones(full, dtype=torch.float64, device=dev))
        J = [self.grad(v) for v in self.xyz]                     # J[a][b] = dx_a / dr_b
        cof = [[J[(a + 1) % 3][(b + 1) % 3] * J[(a + 2) % 3][(b + 2) % 3]
                - J[(a + 1) % 3][(b + 2) % 3] * J[(a + 2) % 3][(b + 1) % 3]
                for b in range(3)] for a in range(3)]             # det J dr_b / dx_a
        det = sum(J[0][b] * cof[0][b] for b in range(3))
        wt = torch.tensor(w, device=dev)
        W = wt.view(1, 1, 1, P) * wt.view(1, 1, P, 1) * wt.view(1, P, 1, 1)
        self.B = W * det
        self.G = {(b, d): W / det * sum(cof[a][b] * cof[a][d] for a in range(3))
                  for b in range(3) for d in range(b, 3)}

    def grad(self, u):
        return (torch.einsum("il,ekjl->ekji", self.D, u), torch.einsum("jl,ekli->ekji", self.D, u),
                torch.einsum("kl,elji->ekji", self.D, u))

    def gather(self, w):
        """QQ^T w."""
        g = torch.zeros(self.n_global, dtype=torch.float64, device=w.device)
        return g.index_add_(0, self.gid, w.reshape(-1))[self.gid].view(w.shape)

    def flux(self, u):
        g, G = self.grad(u), self.G
        return [sum(G[min(b, d), max(b, d)] * g[d] for d in range(3)) for b in range(3)]

    def local(self, u, h1, h2):
        f = [h1 * v for v in self.flux(u)]
        w = (torch.einsum("li,ekjl->ekji", self.D, f[0]) + torch.einsum("lj,ekli->ekji", self.D, f[1])
             + torch.einsum("lk,elji->ekji", self.D, f[2]))
        return w + h2 * self.B * u

    def apply(self, u, h1=1.0, h2=0.0):
        return self.mask * self.gather(self.local(u, h1, h2))

    def diagonal(self, h1, h2):
        D, G, P = self.D, self.G, self.D.shape[0]
        D2, d = D * D, torch.diagonal(D)
        out = (torch.einsum("li,ekjl->ekji", D2, h1 * G[0, 0]) + torch.einsum("lj,ekli->ekji", D2, h1 * G[1, 1])
               + torch.einsum("lk,elji->ekji", D2, h1 * G[2, 2]))
        di, dj, dk = d.view(1, 1, 1, P), d.view(1, 1, P, 1), d.view(1, P, 1, 1)
        out = out + 2.0 * h1 * (G[0, 1] * di * dj + G[0, 2] * di * dk + G[1, 2] * dj * dk)
        return self.gather(out + h2 * self.B)

    def solve(self, b, h1=1.0, h2=0.0, tol=1e-14, maxit=4000):
        """Jacobi-PCG, far beyond the tolerances of the cases."""
        minv = self.mask / self.diagonal(h1, h2)
        x, r = torch.zeros_like(b), b.clone()
        z = minv * r
        p, rz, stop = z.clone(), (r * z / self.mult).sum(), tol * (b * b / self.mult).sum().sqrt()
        for it in range(maxit):
            w = self.apply(p, h1, h2)
            a = rz / (p * w / self.mult).sum()
            x += a * p
            r -= a * w
            if it % 16 == 15 and bool((r * r / self.mult).sum().sqrt() <= stop):
                break
            z = minv * r
            new = (r * z / self.mult).sum()
            p, rz = z + (new / rz) * p, new
        return x

    def source(self, seed):
        return self.mask * self.gather(self.B * _smooth(seed, *self.xyz))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for p in _batch_problems(case, seed):
            if _points(p["nel"], p["N"]) > EXACT_SOLVE_POINTS // 2:
                out.append(None)
                continue
            m = _Plain(p["nel"], p["N"], (TWO_PI,) * 3, DEFORM)
            out.append(m.solve(m.source(p["seed"]), h2=p["lam"]).reshape(-1))
        return out
    nel, N = _nel(case), case["N"]
    if kind in ("solve", "pressure", "adjoint") and _points(nel, N) > EXACT_SOLVE_POINTS:
        return None
    m = _Plain(nel, N, *_mesh(case))
    if kind in ("apply", "ax_dssum"):
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        u = _uniform(_points(nel, N), dtype, seed).double()
        return m.apply(u.view(m.mask.shape), h2=case["h2"]).reshape(-1)
    if kind == "apply_global":
        u = _uniform(m.n_global, torch.float32, seed).double()
        w = m.apply(u[m.gid].view(m.mask.shape), h2=case["h2"]).reshape(-1)
        return torch.zeros(m.n_global, dtype=torch.float64, device="cuda").index_copy_(0, m.gid, w)
    b = m.source(seed)
    if kind in ("solve", "pressure"):
        return m.solve(b, h2=case.get("h2", 0.0)).reshape(-1)
    h1, h2 = 1.0 + 0.5 * torch.tanh(_smooth(seed + 1, *m.xyz)), case["h2"]
    u = m.solve(b, h1, h2)
    lam = m.solve(m.mask * m.gather(2.0 * (u - _smooth(seed + 2, *m.xyz)) / m.mult), h1, h2)
    g = -sum(a * f for a, f in zip(m.grad(lam), m.flux(u)))
    return u.reshape(-1), g.reshape(-1)
