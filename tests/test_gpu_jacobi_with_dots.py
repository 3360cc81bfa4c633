"""A dot product of the same context on another stream while a one-launch Jacobi-PCG is under way: neither disturbs the other."""
import threading
import time

import pytest

import sem_inputs as si
from gpu_common import T, ctx_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_dot_products_during_a_solve():
    mesh = si.box_mesh((6, 6, 6), 7, warp=0.1, perm_seed=1, dirichlet=("x0",))
    ctx = ctx_for(mesh, prec_copies=0)
    b, v = T(si.gaussian_assembled_rhs(mesh, 0)), T(si.uniform_field(mesh, 2))
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    kw = dict(tol=0.0, maxit=1024, rhs="assembled", raise_on_error=False)   # one launch of some 18 ms
    x, info = ctx.solve(b, stream=mine, **kw)
    want = ctx.dot(v, v, stream=other)
    during = 0
    for _ in range(5):
        got, called = [], threading.Event()
        u = torch.empty_like(b)
        torch.cuda.synchronize()

        def work():
            torch.cuda.set_device(0)
            called.set()
            got.append(ctx.solve(b, u=u, stream=mine, **kw)[1])

        t = threading.Thread(target=work)
        t.start()
        called.wait()
        time.sleep(0.004)    # the launch is under way: what comes before it shares the reductions' scratch
        for _ in range(10):
            assert ctx.dot(v, v, stream=other) == want
            during += t.is_alive()
        t.join()
        assert got[0] == info and torch.equal(u, x)
    assert during > 0
    ctx.close()
