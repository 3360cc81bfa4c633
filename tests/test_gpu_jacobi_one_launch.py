"""Jacobi-PCG of small meshes in one cooperative launch (csrc/jacobi_dig.cu) against the same iteration as a chain of
kernels, which a context with a short spin limit keeps."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, global_from_L
from paper_2104_05829_gb300 import _lib

pytestmark = pytest.mark.gpu

CASES = [   # shape, N, Dirichlet faces, nodal h1, h2, pairs
    ((1, 1, 1), 7, ("x0",), False, 0.5, False),
    ((3, 2, 2), 4, ("x0",), True, 0.0, False),
    ((2, 3, 2), 5, ("x0", "y1", "z0"), False, 0.0, False),
    ((4, 3, 2), 6, ("x0", "x1", "y0", "y1", "z0", "z1"), True, 1.0, False),
    ((4, 4, 4), 7, ("x0", "x1", "y0", "y1", "z0", "z1"), False, 0.0, True),
    ((8, 8, 9), 7, ("x0",), False, 0.5, False),     # 576 elements: nearly every block the device holds
    ((9, 9, 9), 7, ("x0",), False, 0.5, False),     # 729: the chain of kernels on both sides
]


@pytest.mark.parametrize("shape, N, faces, nodal, h2, pairs", CASES)
def test_against_the_chain_of_kernels(shape, N, faces, nodal, h2, pairs):
    mesh = si.box_mesh(shape, N, warp=0.1, perm_seed=1, dirichlet=faces)
    lev = O.level_from_mesh(mesh)
    one, chain = ctx_for(mesh, prec_copies=4), ctx_for(mesh, prec_copies=4, spin_limit=1 << 20)
    b = T(si.gaussian_assembled_rhs(mesh, 0))
    h1 = T(np.exp(0.5 * si.smooth_random_field(mesh, 5))) if nodal else None
    x0 = T(H(one.solve(b, h1_L=h1, h2=h2, tol=0.0, maxit=2, rhs="assembled", raise_on_error=False)[0]))

    def run(ctx, **kw):
        x, info = ctx.solve(b, h1_L=h1, h2=h2, rhs="assembled", outer_pairs=pairs, raise_on_error=False, **kw)
        return H(x), info

    # a few iterations: the two differ by roundings only (sums of at most 4e5 terms of one sign in (p, A p) and (r, z):
    # 4e5^0.5 2^-53 each, 30 of them, growing by less than the 1e2 by which CG's coefficients vary here)
    for start in (None, x0):
        kw = dict(tol=0.0, maxit=5) if start is None else dict(tol=0.0, maxit=5, x0=start)
        (xa, ia), (xb, ib) = run(one, **kw), run(chain, **kw)
        assert ia["iters"] == ib["iters"] == 5 and ia["status"] == ib["status"] == _lib.SEM_ENOTCONV
        assert np.abs(xa - xb).max() <= 30 * 4e5 ** 0.5 * 2.0 ** -53 * 1e2 * np.abs(xb).max()
        assert abs(ia["relres"] - ib["relres"]) <= 1e-9 * ib["relres"]
    # to convergence: the solution's own residual (tol, and the recurrence's drift from it: 2^-53 times a condition number
    # of up to 1e5 to 1e6)
    (xa, ia), (xb, ib) = run(one, tol=1e-10, maxit=4000), run(chain, tol=1e-10, maxit=4000)
    assert ia["status"] == ib["status"] == _lib.SEM_OK
    assert abs(ia["iters"] - ib["iters"]) <= 1 + ib["iters"] // 100
    w = H(one.ax(T(xa), h1_L=h1, h2=h2))
    bg = lev.mask(global_from_L(lev, H(b)))
    assert np.linalg.norm(bg - lev.mask(global_from_L(lev, w))) <= 3e-10 * np.linalg.norm(bg)
    # nothing to do, and no iteration allowed
    assert run(one, tol=1e-10, maxit=0)[1]["status"] == _lib.SEM_ENOTCONV
    x, info = one.solve(T(0 * H(b)), h1_L=h1, h2=h2, tol=1e-10, rhs="assembled")
    assert info["iters"] == 0 and not np.any(H(x))
    one.close()
    chain.close()


def test_a_matrix_that_is_not_positive_ends_with_a_breakdown():
    mesh = si.box_mesh((2, 2, 2), 7, warp=0.0, perm_seed=0, dirichlet=("x0",))
    b = T(si.gaussian_assembled_rhs(mesh, 0))
    for limit in (1 << 31, 1 << 20):
        ctx = ctx_for(mesh, prec_copies=0, spin_limit=limit)
        _, info = ctx.solve(b, h1=-1.0, h2=0.0, tol=1e-10, rhs="assembled", raise_on_error=False)
        assert info["status"] == _lib.SEM_EBREAKDOWN and info["iters"] == 0
        ctx.close()
