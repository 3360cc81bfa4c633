"""The element operator in integer digits (csrc/ax_dig.cu): orders with padded lines and planes, nodal h1, the
elements that go to the FP64 form, scaling, alignment."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, relmax

pytestmark = pytest.mark.gpu

# 63-bit digits leave only the FP64 roundings of the oracle's sums (about 3 (N+1) terms twice over) and of the result:
# 6 (N+1) 2^-53 of the terms, which are up to 2^3 times the result's maximum on random u
TOL = 6 * 8 * 2.0 ** -53 * 8


def _oracle(lev, u, h1, h2):
    return O.ax_local(u, lev.G, lev.B, lev.D, h1, h2)


@pytest.mark.parametrize("N", [4, 5, 6, 7])
@pytest.mark.parametrize("nodal", [False, True])
def test_orders_and_coefficients(N, nodal):
    mesh = si.box_mesh((3, 2, 1), N, warp=0.1, perm_seed=1)
    lev = O.level_from_mesh(mesh)
    ctx = ctx_for(mesh, prec_copies=4)
    u = si.uniform_field(mesh, 3, continuous=False)
    h1 = np.exp(0.5 * si.smooth_random_field(mesh, 5)) if nodal else 0.7
    for h2 in (0.0, 1.3):
        ref = _oracle(lev, u, h1, h2)
        for pairs in (False, True):
            w = H(ctx.ax(T(u), h1=1.0 if nodal else h1, h1_L=T(h1) if nodal else None, h2=h2, assemble=False, pairs=pairs))
            assert relmax(w, ref.ravel()) < (TOL if not pairs or N == 7 else 5e-12)
    ctx.close()


@pytest.mark.parametrize("N", [4, 5, 6, 7])
def test_fixed_point_and_fp64_form_agree_at_every_kind_of_point(N):
    """u 2^1000 is computed in FP64 from the same factors; the results at vertices, edges and faces, some hundred to ten
    times smaller than inside, agree with the fixed-point ones relative to their own size."""
    mesh = si.box_mesh((2, 2, 2), N, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    u = si.uniform_field(mesh, 9, continuous=False) * 2.0 ** -10
    shape = (8, N + 1, N + 1, N + 1)
    w = H(ctx.ax(T(u), assemble=False)).reshape(shape)
    ref = H(ctx.ax(T(u * 2.0 ** 1000), assemble=False)).reshape(shape) * 2.0 ** -1000
    end = (np.arange(N + 1) % N == 0).astype(int)
    ends = end[:, None, None] + end[None, :, None] + end[None, None, :]
    for kind in range(4):
        at = np.broadcast_to(ends == kind, shape)
        assert relmax(w[at], ref[at]) < TOL
    ctx.close()


@pytest.mark.parametrize("N", [5, 7])
def test_scale_zero_and_alignment(N):
    mesh = si.box_mesh((2, 1, 3), N, warp=0.05, perm_seed=2)
    ctx = ctx_for(mesh, prec_copies=0)
    u = si.uniform_field(mesh, 4)
    w = H(ctx.ax(T(u), assemble=False))
    for k in (-600, -40, 1, 500):      # a power of two goes through exactly
        assert np.array_equal(H(ctx.ax(T(u * 2.0 ** k), assemble=False)), w * 2.0 ** k)
    assert not np.any(H(ctx.ax(T(0.0 * u), h2=1.0, assemble=False)))
    shifted = T(np.concatenate([[0.0], u.ravel()]))[1:]
    assert np.array_equal(H(ctx.ax(shifted, assemble=False)), w)
    ctx.close()


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-300, 1e300])
def test_elements_outside_fixed_point(value):
    """An element that fixed point cannot hold is computed in FP64, its neighbours are not touched."""
    mesh = si.box_mesh((2, 2, 1), 7, warp=0.1, perm_seed=0)
    lev = O.level_from_mesh(mesh)
    ctx = ctx_for(mesh, prec_copies=0)
    u = si.uniform_field(mesh, 6, continuous=False)
    plain = H(ctx.ax(T(u), h2=0.5, assemble=False)).reshape(4, -1)
    u2 = u.copy()
    if np.isfinite(value):
        u2[1] *= value
        ref = _oracle(lev, u2, 1.0, 0.5).reshape(4, -1)
    else:
        u2[1, 3, 4, 5] = value
    w = H(ctx.ax(T(u2), h2=0.5, assemble=False)).reshape(4, -1)
    assert np.array_equal(w[[0, 2, 3]], plain[[0, 2, 3]])
    if np.isfinite(value):
        assert relmax(w[1], ref[1]) < TOL
    else:
        bad = ~np.isfinite(w[1].reshape(8, 8, 8))
        assert bad[3, 4].all() and bad[3, :, 5].all() and bad[:, 4, 5].all()
    ctx.close()
