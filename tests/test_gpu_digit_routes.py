"""Which kernel answers which call. Fields scaled by 2^1000 are computed with FP64 instructions and scale exactly, so a call that FP64
instructions answer anyway gives the same bits, and one in digits, whose roundings are others, does not."""
import pytest

import sem_inputs as si
from gpu_common import T, ctx_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(2, 12))
def test_operator(N):
    mesh = si.box_mesh((3, 2, 2), N, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=4)
    u = T(si.uniform_field(mesh, 1, continuous=False))
    w, pairs = ctx.ax(u, h2=0.5, assemble=False), ctx.ax(u, h2=0.5, assemble=False, pairs=True)
    far = ctx.ax(u * 2.0 ** 1000, h2=0.5, assemble=False) * 2.0 ** -1000
    part = torch.zeros_like(u)
    ctx.ax_elements(2, 7, u, part, h2=0.5)
    assert torch.equal(w, far) == (N < 4)
    assert torch.equal(w, pairs) == (N in (7, 11))
    assert torch.equal(part.view(12, -1)[2:7], w.view(12, -1)[2:7])
    assert torch.equal(ctx.level_ax(0, u, h1=1.0, h2=0.5, prec="fp64", assemble=False), w)
    ctx.close()


@pytest.mark.parametrize("N", range(2, 9))
def test_advection(N):
    mesh = si.box_mesh((3, 2, 2), N, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    c = torch.stack([T(si.uniform_field(mesh, q)) for q in range(3)])
    u = T(si.uniform_field(mesh, 5))
    w, pairs = ctx.advect(c, u), ctx.advect(c, u, prec="fp64p")
    far = ctx.advect(c, u * 2.0 ** 900) * 2.0 ** -900
    assert torch.equal(w, far) == (N not in (4, 5, 6, 7))
    assert torch.equal(w, pairs) == (N in (5, 6, 7))
    ctx.close()
