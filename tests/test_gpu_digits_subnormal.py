"""Fields of subnormal numbers, whose high words are all zero, through the digit operators: computed in FP64, not taken for zero."""
import numpy as np
import pytest

import sem_inputs as si
from gpu_common import T, ctx_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL = 2.0 ** -1074


def up(t):
    return t * 2.0 ** 1000 * 2.0 ** 60


def down(t):
    return t * 2.0 ** -1000 * 2.0 ** -60


@pytest.mark.parametrize("N", [4, 7, 8, 9, 10, 11])
def test_operator(N):
    mesh = si.box_mesh((2, 1, 2), N, warp=0.0, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    u = T(np.round(1e6 * si.uniform_field(mesh, 3))) * SMALL     # whole multiples of the smallest number
    # the mass term alone: B u, a multiple of the smallest number, rounded once
    assert torch.equal(ctx.ax(u, h1=0.0, h2=1e6, assemble=False), down(ctx.ax(up(u), h1=0.0, h2=1e6, assemble=False)))
    # the stiffness: each of some 6 (N+1) operations may round to a multiple of the smallest number
    w, ref = ctx.ax(u, h1=1e3, assemble=False), down(ctx.ax(up(u), h1=1e3, assemble=False))
    assert torch.any(w != 0)
    # G of these elements is below 1, the rows of D^T sum to at most N^2, and h1 comes last
    assert float((w - ref).abs().max()) <= 1e3 * 6 * (N + 1) * N ** 2 * SMALL
    ctx.close()


@pytest.mark.parametrize("N", [4, 7])
def test_advection(N):
    mesh = si.box_mesh((2, 1, 2), N, warp=0.0, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    c = torch.stack([T(si.uniform_field(mesh, q)) for q in range(3)])
    u = T(np.round(1e8 * si.uniform_field(mesh, 5))) * SMALL
    for a, b in ((c, u), (torch.stack([u, 2 * u, 0 * u]), c[0].contiguous())):
        w = ctx.advect(a, b)
        assert torch.any(w != 0)
        ref = down(ctx.advect(up(a) if a is not c else a, b if a is not c else up(b)))
        # the passes' some 100 roundings, row sums up to 40 three times over
        assert float((w - ref).abs().max()) <= 100 * 40 * 8 * SMALL
    ctx.close()
