"""The digit advection operator on thin elements with a wind along them: the products of the directions are alike while the metric of
one is many times the other's."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, relmax

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# FP64 passes: about 2 (N+1) + 3 nq terms one behind the other, the derivative's row sums up to 40 of the field: 56 2^-53 40 = 2.5e-13;
# pair calls: their 3e-11 bar
TOL = dict(fp64=2.5e-13, fp64p=3e-11)
LD = np.longdouble


def _legendre(n, x):
    p, q = np.ones_like(x), x
    for k in range(1, n):
        p, q = q, ((2 * k + 1) * x * q - k * p) / LD(k + 1)
    return q, n * (x * q - p) / (x * x - 1)


def _rules(N, n):
    """GLL nodes of order N, n Gauss nodes and weights: Newton's method in extended precision."""
    x = O.gll(N)[0].astype(LD)
    z = np.polynomial.legendre.leggauss(n)[0].astype(LD)
    for _ in range(4):
        p, d = _legendre(N, x[1:-1])
        x[1:-1] -= d * (1 - x[1:-1] ** 2) / (2 * x[1:-1] * d - N * (N + 1) * p)
        p, d = _legendre(n, z)
        z -= p / d
    return x, z, 2 / ((1 - z * z) * _legendre(n, z)[1] ** 2)


def _cardinal(x, z):
    J = np.ones((len(z), len(x)), dtype=LD)
    for b in range(len(x)):
        for c in range(len(x)):
            if c != b:
                J[:, b] *= (z - x[c]) / (x[b] - x[c])
    return J


def _derivative(x):
    lam = np.array([1 / np.prod([x[b] - x[c] for c in range(len(x)) if c != b]) for b in range(len(x))], dtype=LD)
    D = np.array([[lam[b] / lam[a] / (x[a] - x[b]) if a != b else 0 for b in range(len(x))] for a in range(len(x))], dtype=LD)
    return D - np.diag(D.sum(1))


def _apply(M, v, axis):
    return np.moveaxis(np.moveaxis(v, axis, -1) @ M.T, -1, axis)


def _extended(mesh, c, u):
    """C(c) u element by element in extended precision. (The oracle's FP64 metric costs 2.4e-13 on the thinnest elements here.)"""
    x, z, w = _rules(mesh["N"], (3 * (mesh["N"] + 1) + 1) // 2)
    I, D = _cardinal(x, z), _derivative(z)
    gauss = lambda v: _apply(I, _apply(I, _apply(I, v.astype(LD), 3), 2), 1)
    X = [gauss(mesh[q] - mesh[q][:, :1, :1, :1]) for q in "xyz"]
    J = [[_apply(D, X[m], 3 - d) for d in range(3)] for m in range(3)]
    cof = lambda d, m: (J[(m + 1) % 3][(d + 1) % 3] * J[(m + 2) % 3][(d + 2) % 3]
                        - J[(m + 1) % 3][(d + 2) % 3] * J[(m + 2) % 3][(d + 1) % 3])
    cq, uq = [gauss(f) for f in c], gauss(u)
    w3 = w[:, None, None] * w[:, None] * w
    v = sum(w3 * cof(d, m) * cq[m] * _apply(D, uq, 3 - d) for d in range(3) for m in range(3))
    return _apply(I.T, _apply(I.T, _apply(I.T, v, 1), 2), 3).ravel()


@pytest.mark.parametrize("N", [4, 5, 6, 7])
@pytest.mark.parametrize("k", [0, 5, 7, 9, 13, 20, 30])
def test_thin_elements(N, k):
    mesh = dict(si.box_mesh((2, 3, 2), N, warp=0.1, perm_seed=0))
    x, y, z = mesh["x"], mesh["y"], mesh["z"]
    thin = 2.0 ** -k
    mesh["y"] = y * thin
    ctx = ctx_for(mesh, prec_copies=0)
    c = np.stack([np.sin(np.pi * x) * np.cos(y), thin * np.cos(2 * x) * z, 1 + 0.3 * np.sin(3 * x * y)])
    u = np.exp(x) * np.sin(3 * y + z)
    ref = _extended(mesh, c, u)
    for prec, tol in TOL.items():
        w = H(ctx.advect(torch.stack([T(f) for f in c]), T(u), prec=prec))
        assert relmax(w, ref) < tol
    ctx.close()
