"""The work that a program has this library do, as cases to be timed and compared.

A case is one call (or one short sequence of calls) of the package's public entry points on a
box of hexahedral elements: the assembled operator of an outer Krylov iteration, the operators
and the Schwarz smoother of the p-multigrid levels, the dealiased advection term and its
characteristics substep, whole solves, and the differentiated solve. Meshes are boxes of
Ex x Ey x Ez elements in a shuffled storage order, as an unstructured mesh reader delivers
them, and fields are drawn on the GPU from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2104_05829_gb300 import SemContext
from paper_2104_05829_gb300.autograd import helmholtz_solve

ALL_FACES = "x0 x1 y0 y1 z0 z1"


def listed():
    return [
        # the operator of a small solve (4^3 elements, all-Dirichlet Poisson): launches and latency count
        dict(name="ax_4x4x4_n7", kind="ax", ex=4, ey=4, ez=4, N=7, prec="fp64", warp=0.0, h2=0.0, nodal=False, faces=ALL_FACES, field="smooth"),
        # the throughput workload: Helmholtz operator on the warped 32^3 box, larger than L2
        dict(name="ax_32x32x32_n7", kind="ax", ex=32, ey=32, ez=32, N=7, prec="fp64", warp=0.1, h2=0.5, nodal=False, faces=ALL_FACES, field="random"),
        # the operator of a differentiated Helmholtz solve: nodal diffusion coefficient, odd element counts, order 5
        dict(name="ax_31x29x33_n5_nodal", kind="ax", ex=31, ey=29, ez=33, N=5, prec="fp64", warp=0.1, h2=1.0, nodal=True, faces=ALL_FACES, field="smooth"),
        # the high-order end of the order sweep with the FP32-pair option
        dict(name="ax_26x26x26_n9_pairs", kind="ax", ex=26, ey=26, ez=26, N=9, prec="pairs", warp=0.1, h2=0.5, nodal=False, faces=ALL_FACES, field="random"),
        # the fine-level operator of the mixed-precision V-cycle (BF16 factors) on the 24^3 pressure mesh
        dict(name="level_ax_24x24x24_n7_bf16g", kind="level_ax", ex=24, ey=24, ez=24, N=7, prec="bf16g", warp=0.1, h2=0.0, faces="x0"),
        # the Schwarz smoother's local solves on the 24^3 pressure mesh
        dict(name="asm_24x24x24_n7_fp32", kind="asm", ex=24, ey=24, ez=24, N=7, prec="fp32", warp=0.1, h2=0.0, faces="x0"),
        # the nonlinear term of a momentum step: three components in full precision
        dict(name="advect_24x24x24_n7_fp64", kind="advect", ex=24, ey=24, ez=24, N=7, prec="fp64", warp=0.1, ncomp=3),
        # the same term for two scalars in FP32, odd element counts, another order
        dict(name="advect_17x19x13_n6_fp32", kind="advect", ex=17, ey=19, ez=13, N=6, prec="fp32", warp=0.1, ncomp=2),
        # one Runge-Kutta substep of the characteristics scheme on a velocity field
        dict(name="char_16x16x16_n7_fp64p", kind="char", ex=16, ey=16, ez=16, N=7, prec="fp64p", warp=0.1, ncomp=3),
        # the pressure solve of a time step: flexible CG + p-multigrid, FP32 V-cycle, FP32-pair outer operator
        dict(name="solve_24x24x24_n7_pmg", kind="solve", ex=24, ey=24, ez=24, N=7, precond="pmg", prec="fp32", outer_pairs=True, smoother="jacobi", warp=0.1, h2=0.0, tol=1e-8, faces="x0"),
        # the small manufactured Poisson solve by Jacobi-PCG: a chain of short launches
        dict(name="solve_4x4x4_n7_jacobi", kind="solve", ex=4, ey=4, ez=4, N=7, precond="jacobi", prec="fp64", outer_pairs=False, smoother="jacobi", warp=0.0, h2=0.0, tol=1e-10, faces=ALL_FACES),
        # a training step on the solution: forward solve with a nodal coefficient, adjoint solve and both gradients
        dict(name="adjoint_12x12x12_n7", kind="adjoint", ex=12, ey=12, ez=12, N=7, precond="pmg", prec="fp32", outer_pairs=False, smoother="jacobi", warp=0.1, h2=1.0, tol=1e-10, faces=ALL_FACES),
    ]


def _shape(rng, N, lo, hi):
    """Elements per direction of a box of about lo..hi local points (log-uniform), sides within a factor of two."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi))) / (N + 1) ** 3
    side = max(1.0, n ** (1.0 / 3.0))
    e = [max(1, round(side * rng.uniform(0.75, 1.33))) for _ in range(3)]
    while e[0] * e[1] * e[2] * (N + 1) ** 3 > hi:
        e[e.index(max(e))] -= 1
    return dict(ex=e[0], ey=e[1], ez=e[2])


def draw(rng):
    kind = rng.choice(["ax", "ax", "ax", "level_ax", "asm", "advect", "advect", "char", "solve", "solve", "adjoint"])
    warp = rng.choice([0.1, 0.1, 0.05])
    if kind == "ax":
        N = rng.choice([7, 7, 7, 3, 5, 9, 11, rng.randint(2, 11)])
        return dict(kind=kind, N=N, **_shape(rng, N, 2 ** 15, 2 ** 24), prec=rng.choice(["fp64", "fp64", "pairs"]), warp=warp,
                    h2=rng.choice([0.0, 0.5, 1.0]), nodal=rng.random() < 0.25, faces=rng.choice([ALL_FACES, "x0", "x0 y1 z0"]),
                    field=rng.choice(["random", "smooth"]))
    if kind == "level_ax":
        N = rng.choice([7, 7, 3, 5, 9, rng.randint(2, 11)])
        return dict(kind=kind, N=N, **_shape(rng, N, 2 ** 15, 2 ** 23), prec=rng.choice(["fp32", "bf16g"]), warp=warp,
                    h2=rng.choice([0.0, 0.5]), faces=rng.choice([ALL_FACES, "x0"]))
    if kind == "asm":
        N = rng.choice([7, 7, 3, 5, rng.randint(2, 8)])
        return dict(kind=kind, N=N, **_shape(rng, N, 2 ** 15, 24 ** 3 * 512), prec=rng.choice(["fp32", "bf16g"]), warp=warp,
                    h2=rng.choice([0.0, 0.5]), faces=rng.choice([ALL_FACES, "x0"]))
    if kind in ("advect", "char"):
        N = rng.choice([7, 7, 5, rng.randint(2, 8)])
        return dict(kind=kind, N=N, **_shape(rng, N, 2 ** 15, (24 ** 3 if kind == "advect" else 16 ** 3) * 512),
                    prec=rng.choice(["fp64", "fp64p", "fp32"]), warp=warp, ncomp=rng.choice([1, 2, 3]))
    N = rng.choice([7, 7, 5, rng.randint(3, 9)])
    pmg = kind == "adjoint" or rng.random() < 0.65
    hi = 12 ** 3 * 512 if kind == "adjoint" else (20 ** 3 * 512 if pmg else 8 ** 3 * 512)
    smoother = "asm" if kind == "solve" and pmg and rng.random() < 0.4 else "jacobi"
    return dict(kind=kind, N=N, **_shape(rng, N, 2 ** 14, hi), precond="pmg" if pmg else "jacobi",
                prec=rng.choice(["fp32", "bf16g", "fp64"]) if pmg else "fp64", outer_pairs=rng.random() < 0.5, smoother=smoother,
                warp=warp, h2=1.0 if kind == "adjoint" else rng.choice([0.0, 0.5]), tol=1e-10 if kind == "adjoint" or not pmg else 1e-8,
                faces=rng.choice([ALL_FACES, "x0"]))


# ---- one-dimensional rules ---------------------------------------------------------------------

def _gll(N):
    """GLL nodes and weights of order N."""
    c = np.zeros(N + 1)
    c[N] = 1.0
    leg = np.polynomial.legendre
    x = np.concatenate(([-1.0], np.sort(leg.legroots(leg.legder(c)).real), [1.0])) if N > 1 else np.array([-1.0, 1.0])
    for _ in range(4):  # Newton on P_N' at the interior nodes, P_N'' from Legendre's equation
        if N > 1:
            p, d = leg.legval(x[1:-1], c), leg.legval(x[1:-1], leg.legder(c))
            x[1:-1] -= d * (1 - x[1:-1] ** 2) / (2 * x[1:-1] * d - N * (N + 1) * p)
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (N * (N + 1) * leg.legval(x, c) ** 2)


def _cardinal(nodes, at):
    """J[a, b]: cardinal polynomial b on the nodes at point a."""
    J = np.ones((len(at), len(nodes)))
    for b in range(len(nodes)):
        for c in range(len(nodes)):
            if c != b:
                J[:, b] *= (at - nodes[c]) / (nodes[b] - nodes[c])
    return J


def _deriv(x):
    """D[a, b]: derivative of cardinal polynomial b on the nodes x at node a."""
    n = len(x)
    lam = np.array([1.0 / np.prod([x[b] - x[c] for c in range(n) if c != b]) for b in range(n)])
    D = np.zeros((n, n))
    for a in range(n):
        for b in range(n):
            if a != b:
                D[a, b] = lam[b] / lam[a] / (x[a] - x[b])
        D[a, a] = -D[a].sum()
    return D


# ---- the mesh and the context a program keeps ----------------------------------------------------

class _Box:
    """A box mesh: coordinates, lattice position and Dirichlet flag of every local point, shaped [E, k, j, i]."""

    def __init__(self, ex, ey, ez, N, warp, faces):
        self.shape, self.N, self.E = (ex, ey, ez), N, ex * ey * ez
        dev = "cuda"
        order = torch.as_tensor(np.random.RandomState(0).permutation(self.E), device=dev)
        self.el = el = [order % ex, (order // ex) % ey, order // (ex * ey)]
        xi, self.rho = _gll(N)
        t = torch.as_tensor((xi + 1.0) / 2.0, device=dev)
        a = torch.arange(N + 1, device=dev)
        views = [(1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1)]
        full = (self.E, N + 1, N + 1, N + 1)
        self.ijk = [(el[d].view(-1, 1, 1, 1) * N + a.view(views[d])) for d in range(3)]
        self.side = [n * N + 1 for n in self.shape]
        self.lattice = (self.ijk[0] + self.side[0] * (self.ijk[1] + self.side[1] * self.ijk[2])).expand(full).reshape(-1)
        x = [(el[d].view(-1, 1, 1, 1) + t.view(views[d])) / self.shape[d] for d in range(3)]
        s = warp * torch.sin(math.pi * x[0]) * torch.sin(math.pi * x[1]) * torch.sin(math.pi * x[2])
        self.x = [(v + s).expand(full).contiguous() for v in x]
        m = torch.zeros(full, dtype=torch.bool, device=dev)
        for f in faces.split():
            d = "xyz".index(f[0])
            m |= self.ijk[d] == (0 if f[1] == "0" else self.side[d] - 1)
        self.dirichlet, self.faces = m, faces.split()
        self.n_lattice = self.side[0] * self.side[1] * self.side[2]

    def on_nodes(self, values):
        """Local points of one value per lattice node."""
        return values[self.lattice]

    def sum_copies(self, w):
        g = torch.zeros(self.n_lattice, dtype=w.dtype, device=w.device)
        return g.index_add_(0, self.lattice, w)[self.lattice]


@functools.lru_cache(maxsize=1)
def _box(ex, ey, ez, N, warp, faces):
    return _Box(ex, ey, ez, N, warp, faces)


@functools.lru_cache(maxsize=1)
def _context(ex, ey, ez, N, warp, faces, copies, smoother):
    """The context of a mesh: set up once by a program and used for every call that follows."""
    box = _box(ex, ey, ez, N, warp, faces)
    host = [v.cpu().numpy() for v in box.x]
    return SemContext(*host, (box.lattice + 1).cpu().numpy(), box.dirichlet.to(torch.uint8).cpu().numpy(), N,
                      prec_copies=copies, smoother=smoother)


_FP32, _BF16G, _PAIRS = 1, 2, 4   # the factor copies a context is asked for


def _mesh_of(case):
    box = (case["ex"], case["ey"], case["ez"], case["N"], case["warp"], case.get("faces", ""))
    copies = {"fp32": _FP32, "bf16g": _FP32 | _BF16G, "pairs": _PAIRS}.get(case["prec"], 0)
    if case.get("outer_pairs"):
        copies |= _PAIRS
    return _box(*box), box + (copies, case.get("smoother", "jacobi"))


def _smooth(box, gen, modes=8, kmax=4):
    """A sum of cosine modes with random wave vectors, amplitudes and phases."""
    v = torch.zeros_like(box.x[0])
    k = torch.randint(-kmax, kmax + 1, (modes, 3), generator=gen, device="cuda").tolist()
    a = torch.randn(modes, generator=gen, device="cuda", dtype=torch.float64).tolist()
    p = (2 * math.pi * torch.rand(modes, generator=gen, device="cuda", dtype=torch.float64)).tolist()
    for m in range(modes):
        v += a[m] * math.sqrt(2.0 / modes) * torch.cos(math.pi * (k[m][0] * box.x[0] + k[m][1] * box.x[1] + k[m][2] * box.x[2]) + p[m])
    return v.reshape(-1)


def _random(box, gen, normal=False):
    make = torch.randn if normal else torch.rand
    v = make(box.n_lattice, generator=gen, device="cuda", dtype=torch.float64)
    return box.on_nodes(v - v.mean() if normal else 2.0 * v - 1.0)


def _inputs(case, seed):
    """The fields of a case, in FP64 (those of an FP32 call hold FP32 values)."""
    box, _ = _mesh_of(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    free = (~box.dirichlet).reshape(-1).to(torch.float64)
    kind, d = case["kind"], {}
    if kind == "ax":
        d["u"] = free * (_smooth(box, gen) if case["field"] == "smooth" else _random(box, gen))
        if case["nodal"]:
            d["h1"] = torch.exp(0.5 * _smooth(box, gen))
    elif kind in ("level_ax", "asm"):
        d["u"] = free * _random(box, gen, normal=kind == "asm")
    elif kind in ("advect", "char"):
        d["c"] = torch.stack([_smooth(box, gen) for _ in range(3)])
        d["u"] = torch.stack([_smooth(box, gen) for _ in range(case["ncomp"])])
    elif kind == "solve":
        d["b"] = free * _random(box, gen, normal=True)
    else:
        d["f"] = _smooth(box, gen)
        d["h1"] = torch.exp(0.5 * _smooth(box, gen))
        d["gu"] = _smooth(box, gen)
    if case["prec"] in ("fp32", "bf16g") and kind in ("level_ax", "asm", "advect", "char"):
        d = {k: v.to(torch.float32).to(torch.float64) for k, v in d.items()}
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    _, key = _mesh_of(case)
    ctx = _context(*key)
    kind = case["kind"]
    if case["prec"] in ("fp32", "bf16g") and kind in ("level_ax", "asm", "advect", "char"):
        d = {k: v.to(torch.float32) for k, v in d.items()}
    s = dict(case=case, ctx=ctx, **{k: v.contiguous() for k, v in d.items()})
    if kind in ("ax", "level_ax", "asm", "advect", "char"):
        s["w"] = torch.empty_like(s["u"])
    elif kind == "solve":
        s["w"] = torch.empty_like(s["b"])
    # what a context builds on its first call of a kind (cubature factors, Schwarz data, workspaces)
    # is part of what a program has in hand
    if not getattr(ctx, "_warm", False) and kind in ("asm", "advect", "char"):
        run(s)
        ctx._warm = True
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "ax":
        return ctx.ax(s["u"], s["w"], h1=1.0, h2=case["h2"], h1_L=s.get("h1"), assemble=True, pairs=case["prec"] == "pairs")
    if kind == "level_ax":
        return ctx.level_ax(0, s["u"], s["w"], h1=1.0, h2=case["h2"], prec=case["prec"], assemble=True)
    if kind == "asm":
        return ctx.asm_apply(0, s["u"], s["w"], h1=1.0, h2=case["h2"], prec=case["prec"])
    if kind == "advect":
        return ctx.advect(s["c"], s["u"], s["w"], assemble=True, prec=case["prec"])
    if kind == "char":
        # the scheme advances a copy: the field of the earlier time level is used again by the next step
        s["w"].copy_(s["u"])
        return ctx.char_advance(s["c"], s["w"], 0.0, 1e-3, 1, prec=case["prec"])
    if kind == "solve":
        u, _ = ctx.solve(s["b"], h1=1.0, h2=case["h2"], tol=case["tol"], maxit=2000, precond=case["precond"], prec=case["prec"],
                         rhs="assembled", u=s["w"], outer_pairs=case["outer_pairs"])
        return u
    f, h1 = s["f"].detach().requires_grad_(True), s["h1"].detach().requires_grad_(True)
    u = helmholtz_solve(ctx, f, h1, h2=case["h2"], tol=case["tol"], maxit=2000, precond=case["precond"], prec=case["prec"],
                        outer_pairs=case["outer_pairs"])
    df, dh1 = torch.autograd.grad(u, (f, h1), s["gu"])
    return u.detach(), df, dh1


def work(case):
    NP = case["N"] + 1
    E = case["ex"] * case["ey"] * case["ez"]
    n = E * NP ** 3
    kind = case["kind"]
    ax_flops = E * (12 * NP ** 4 + 17 * NP ** 3)
    if kind == "ax":
        return dict(bytes=n * (72 + (8 if case["nodal"] else 0)), flops=ax_flops)
    if kind == "level_ax":
        return dict(bytes=n * (36 if case["prec"] == "fp32" else 22), flops=ax_flops)
    if kind == "asm":
        return dict(bytes=n * 12, flops=E * 12 * (NP + 2) ** 4)
    if kind in ("advect", "char"):
        q, size = (3 * NP + 1) // 2, 4 if case["prec"] == "fp32" else 8
        interp = 2 * (NP ** 3 * q + NP ** 2 * q ** 2 + NP * q ** 3)
        flops = E * (3 * (interp + 6 * q ** 3) + case["ncomp"] * (2 * interp + 6 * q ** 4 + 6 * q ** 3))
        b = E * size * (9 * q ** 3 + (3 + 2 * case["ncomp"]) * NP ** 3)
        steps = 4 if kind == "char" else 1   # a Runge-Kutta substep evaluates the term four times
        return dict(bytes=b * steps, flops=flops * steps)
    # a solve applies the outer operator once an iteration and, with p-multigrid, four fine-level
    # operators of the V-cycle; iteration counts are those of these tolerances
    if case["precond"] == "jacobi":
        its, per = 60, n * (72 + 40)
        return dict(bytes=its * per, flops=its * ax_flops)
    per = n * (72 + 40 + 4 * {"fp32": 36, "bf16g": 22, "fp64": 72}[case["prec"]])
    its = 15 if kind == "solve" else 2 * 20
    return dict(bytes=its * per, flops=its * 5 * ax_flops)


# ---- the same in plain 64-bit torch --------------------------------------------------------------

def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _lines(M, v, axis):
    """Matrix M on the i (axis 0), j (1) or k (2) lines of v [..., k, j, i]."""
    v = v.movedim(-1 - axis, -1)
    return (v @ M.T).movedim(-1, -1 - axis)


def _grad(D, v):
    return [_lines(D, v, a) for a in range(3)]


class _Exact:
    """A = R QQ^T (D^T h1 G D + h2 B) of a box in 64 bits."""

    def __init__(self, case):
        self.case, self.box = case, _mesh_of(case)[0]
        box, N = self.box, case["N"]
        xi, rho = _gll(N)
        self.xi, self.D = xi, _t(_deriv(xi))
        self.free = (~box.dirichlet).to(torch.float64)
        rho = _t(rho)
        w3 = rho.view(-1, 1, 1) * rho.view(1, -1, 1) * rho
        inv, det = self.metric(self.D, box.x)
        self.B = w3 * det
        self.G = [[sum(inv[m][p] * inv[n][p] for p in range(3)) * self.B if n >= m else None for n in range(3)] for m in range(3)]

    @staticmethod
    def metric(D, x):
        """dr_d/dx_m as a table [d][m], and the Jacobian."""
        J = [_grad(D, v - v[:, :1, :1, :1]) for v in x]   # J[m][d] = dx_m / dr_d
        adj = [[J[(m + 1) % 3][(d + 1) % 3] * J[(m + 2) % 3][(d + 2) % 3] - J[(m + 1) % 3][(d + 2) % 3] * J[(m + 2) % 3][(d + 1) % 3]
                for m in range(3)] for d in range(3)]
        det = sum(J[m][0] * adj[0][m] for m in range(3))
        return [[adj[d][m] / det for m in range(3)] for d in range(3)], det

    def shaped(self, v):
        return v.view(self.box.E, *(3 * [self.case["N"] + 1]))

    def flux(self, u):
        g = _grad(self.D, u)
        return [sum(self.G[min(m, n)][max(m, n)] * g[n] for n in range(3)) for m in range(3)]

    def apply(self, u, h1, h2):
        u = self.shaped(u)
        w = h2 * self.B * u
        for m, f in enumerate(self.flux(u)):
            w = w + _lines(self.D.T, f if h1 is None else h1 * f, m)
        return self.free.reshape(-1) * self.box.sum_copies(w.reshape(-1))

    def diagonal(self, h1, h2):
        one = torch.ones_like(self.B) if h1 is None else h1
        d, D = h2 * self.B, self.D
        dd = D.diagonal()
        view = [dd, dd.view(-1, 1), dd.view(-1, 1, 1)]
        for m in range(3):
            d = d + _lines((D * D).T.contiguous(), one * self.G[m][m], m)
            for n in range(m + 1, 3):
                d = d + 2.0 * one * self.G[m][n] * view[m] * view[n]
        return self.box.sum_copies(d.reshape(-1))

    def solve(self, b, h1, h2, tol=3e-14, maxit=6000):
        """Conjugate gradients with the diagonal, on replicated vectors (one owner copy in the products)."""
        copies = self.box.sum_copies(torch.ones_like(b))
        own = self.free.reshape(-1) / copies
        inv = self.free.reshape(-1) / self.diagonal(h1, h2)
        x, r = torch.zeros_like(b), b.clone()
        z = inv * r
        p, rz = z.clone(), torch.dot(own * r, z)
        stop = tol * torch.dot(own * b, b).sqrt()
        for it in range(maxit):
            w = self.apply(p, h1, h2)
            a = rz / torch.dot(own * p, w)
            x += a * p
            r -= a * w
            if it % 8 == 7 and bool(torch.dot(own * r, r).sqrt() <= stop):
                break
            z = inv * r
            new = torch.dot(own * r, z)
            p = z + (new / rz) * p
            rz = new
        return x

    # -- the dealiased advection term
    def advection(self):
        N, box = self.case["N"], self.box
        z, w = np.polynomial.legendre.leggauss((3 * (N + 1) + 1) // 2)
        self.I, self.Dq, self.wq = _t(_cardinal(self.xi, z)), _t(_deriv(z)), _t(w)

    def to_gauss(self, v):
        return _lines(self.I, _lines(self.I, _lines(self.I, v, 0), 1), 2)

    def advect(self, c, u):
        c, u = [self.shaped(v) for v in c], [self.shaped(v) for v in u]
        out = [torch.empty_like(v) for v in u]
        w3 = self.wq.view(-1, 1, 1) * self.wq.view(1, -1, 1) * self.wq
        for e in range(0, self.box.E, 2048):
            sl = slice(e, e + 2048)
            inv, det = self.metric(self.Dq, [self.to_gauss(v[sl] - v[sl, :1, :1, :1]) for v in self.box.x])
            cq = [self.to_gauss(v[sl]) for v in c]
            ch = [sum(inv[d][m] * cq[m] for m in range(3)) * det * w3 for d in range(3)]
            for v, o in zip(u, out):
                g = _grad(self.Dq, self.to_gauss(v[sl]))
                q = sum(ch[d] * g[d] for d in range(3))
                T = self.I.T.contiguous()
                o[sl] = _lines(T, _lines(T, _lines(T, q, 2), 1), 0)
        return torch.stack([self.box.sum_copies(v.reshape(-1)) for v in out])

    # -- the overlapping Schwarz smoother
    def schwarz(self, r, h2):
        box, N = self.box, self.case["N"]
        M, E = N + 3, box.E
        rho = box.rho
        K = _deriv(self.xi).T @ np.diag(rho) @ _deriv(self.xi)
        sides = []   # side types of every element: 0 neighbour, 1 Dirichlet, 2 Neumann
        for d in range(3):
            ends = []
            for side, at in ((0, 0), (1, box.shape[d] - 1)):
                t = 1 if "xyz"[d] + str(side) in box.faces else 2
                ends.append(torch.where(box.el[d] == at, t, 0))
            sides.append(ends)
        S = np.zeros((9, M, M))
        lam = np.ones((9, M))
        for left in range(3):
            for right in range(3):
                A, B = np.zeros((3 * N + 1,) * 2), np.zeros(3 * N + 1)
                for el, there in ((0, left == 0), (1, True), (2, right == 0)):
                    if there:
                        A[el * N:el * N + N + 1, el * N:el * N + N + 1] += K
                        B[el * N:el * N + N + 1] += rho
                keep = [s for s in range(-1, N + 2) if not (s == -1 and left or s == 0 and left == 1 or s == N and right == 1 or s == N + 1 and right)]
                g = np.array(keep) + N
                q = 1.0 / np.sqrt(B[g])
                lm, Q = np.linalg.eigh(q[:, None] * A[np.ix_(g, g)] * q)
                S[3 * left + right][np.array(keep) + 1, :len(keep)] = q[:, None] * Q
                lam[3 * left + right, :len(keep)] = lm
        S, lam = _t(S), _t(lam)
        X = torch.stack(box.x)
        length = []
        for d in range(3):
            X_ = X.movedim(-1 - d, -1)
            length.append((X_[..., N] - X_[..., 0]).square().sum(0).sqrt().mean((-1, -2)))
        # lattice position of every slot of the (N+3)^3 boxes, kept where the slot is the element's own or in a face layer
        a = torch.arange(-1, N + 2, device="cuda")
        views = [(1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1)]
        pos = [box.el[d].view(-1, 1, 1, 1) * N + a.view(views[d]) for d in range(3)]
        inside, outer = torch.ones((E, M, M, M), dtype=torch.bool, device="cuda"), torch.zeros((E, M, M, M), dtype=torch.int8, device="cuda")
        for d in range(3):
            inside &= (pos[d] >= 0) & (pos[d] < box.side[d])
            outer += ((a == -1) | (a == N + 1)).view(views[d]).to(torch.int8)
        keep = inside & (outer <= 1)
        node = torch.where(keep, pos[0] + box.side[0] * (pos[1] + box.side[1] * pos[2]), 0).reshape(-1)
        keep = keep.to(torch.float64)
        glob = torch.zeros(box.n_lattice, dtype=torch.float64, device="cuda")
        glob[box.lattice] = r
        v = keep * glob[node].view(keep.shape)
        mats = [S[3 * sides[d][0] + sides[d][1]] for d in range(3)]
        eig = [(2.0 / length[d]).square()[:, None] * lam[3 * sides[d][0] + sides[d][1]] for d in range(3)]
        v = torch.einsum("ema,ekjm->ekja", mats[0], v)
        v = torch.einsum("emb,ekmi->ekbi", mats[1], v)
        v = torch.einsum("emc,emji->ecji", mats[2], v)
        den = eig[2][:, :, None, None] + eig[1][:, None, :, None] + eig[0][:, None, None, :] + h2
        v = torch.where(den != 0, v / torch.where(den != 0, den, 1.0), 0.0) * (8.0 / (length[0] * length[1] * length[2])).view(-1, 1, 1, 1)
        v = torch.einsum("ecm,emji->ecji", mats[2], v)
        v = torch.einsum("ebm,ekmi->ekbi", mats[1], v)
        v = torch.einsum("eam,ekjm->ekja", mats[0], v)
        z = torch.zeros_like(glob).index_add_(0, node, (keep * v).reshape(-1))
        count = torch.zeros_like(glob).index_add_(0, node, keep.reshape(-1))
        return self.free.reshape(-1) * (z / count.clamp(min=1.0))[box.lattice]


def exact(case, seed):
    kind, n = case["kind"], case["ex"] * case["ey"] * case["ez"] * (case["N"] + 1) ** 3
    if kind in ("solve", "adjoint") and n > 1_500_000:
        return None   # thousands of plain iterations on a large box take too long
    d, X = _inputs(case, seed), _Exact(case)
    h1 = X.shaped(d["h1"]) if "h1" in d else None
    if kind in ("ax", "level_ax"):
        return X.apply(d["u"], h1, case["h2"])
    if kind == "asm":
        return X.schwarz(d["u"], case["h2"])
    if kind == "solve":
        return X.solve(d["b"], None, case["h2"])
    if kind == "adjoint":
        free = X.free.reshape(-1)
        u = X.solve(free * X.box.sum_copies((X.B * X.shaped(d["f"])).reshape(-1)), h1, case["h2"])
        lam = X.solve(free * X.box.sum_copies(d["gu"]), h1, case["h2"])
        gl, fu = _grad(X.D, X.shaped(lam)), X.flux(X.shaped(u))
        return u, X.B.reshape(-1) * lam, -sum(g * f for g, f in zip(gl, fu)).reshape(-1)
    X.advection()
    if kind == "advect":
        return X.advect(d["c"], d["u"])
    mass, h, w = X.box.sum_copies(X.B.reshape(-1)), 1e-3, d["u"]
    slope = lambda v: -X.advect(d["c"], v) / mass  # noqa: E731
    k1 = slope(w)
    k2 = slope(w + 0.5 * h * k1)
    k3 = slope(w + 0.5 * h * k2)
    k4 = slope(w + h * k3)
    return w + (h / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
