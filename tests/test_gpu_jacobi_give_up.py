"""The one-launch Jacobi-PCG where a grid barrier gives up: the solve goes on with the chain of kernels, from where it was. And which of
the two ran, seen by the last bits: the forms add in different orders."""
import numpy as np
import pytest

import sem_inputs as si
from gpu_common import H, T, ctx_for
from paper_2104_05829_gb300 import _lib

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ONE, CHAIN, GIVES_UP = 1 << 31, 1 << 20, 0     # spin limits


def _solve(mesh, limit, x0=False, **kw):
    ctx = ctx_for(mesh, prec_copies=0, spin_limit=limit)
    b = T(si.gaussian_assembled_rhs(mesh, 0))
    start = dict(x0=T(0.25 * H(b))) if x0 else {}
    x, info = ctx.solve(b, h2=0.5, rhs="assembled", raise_on_error=False, **start, **kw)
    again, _ = ctx.solve(b, h2=0.5, rhs="assembled", raise_on_error=False, **start, **kw)
    assert torch.equal(x, again)       # the context stays usable, and a repetition gives the same bits
    ctx.close()
    return x, info


@pytest.mark.parametrize("shape, N, one", [((4, 4, 4), 7, True), ((8, 8, 9), 7, True), ((5, 4, 3), 4, True), ((6, 3, 3), 6, True),
                                           ((9, 9, 9), 7, False)])
@pytest.mark.parametrize("x0", [False, True])
def test_give_up_and_which_form_ran(shape, N, one, x0):
    mesh = si.box_mesh(shape, N, warp=0.1, perm_seed=1, dirichlet=("x0",))
    kw = dict(tol=0.0, maxit=20, x0=x0)
    (xo, io), (xc, ic), (xg, ig) = (_solve(mesh, limit, **kw) for limit in (ONE, CHAIN, GIVES_UP))
    assert io["iters"] == ic["iters"] == ig["iters"] == 20
    assert io["status"] == ic["status"] == ig["status"] == _lib.SEM_ENOTCONV
    assert torch.equal(xo, xc) == (not one)
    # every launch's first barrier finds a block missing: the chain from the start, with its bits
    assert torch.equal(xg, xc) and ig["relres"] == ic["relres"]
    # to convergence
    (xo, io), (xc, ic), (xg, ig) = (_solve(mesh, limit, tol=1e-10, maxit=4000, x0=x0) for limit in (ONE, CHAIN, GIVES_UP))
    assert io["status"] == ic["status"] == ig["status"] == _lib.SEM_OK
    assert torch.equal(xg, xc) and ig["iters"] == ic["iters"]


def test_one_element_has_nobody_to_wait_for():
    mesh = si.box_mesh((1, 1, 1), 7, warp=0.1, perm_seed=0, dirichlet=("x0",))
    (xo, io), (xg, ig) = (_solve(mesh, limit, tol=1e-10, maxit=4000) for limit in (ONE, GIVES_UP))
    assert io["status"] == ig["status"] == _lib.SEM_OK and io["iters"] == ig["iters"] and torch.equal(xo, xg)
