"""The element operator in integer digits at 8 <= N <= 11 (csrc/ax_dig_eo.cu): even and odd numbers of points, nodal h1,
the elements that go to the FP64 form, scaling."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, relmax

pytestmark = pytest.mark.gpu

# as for the lower orders: 6 (N+1) 2^-53 of the terms, which are up to 2^3 times the result's maximum on random u
TOL = 6 * 12 * 2.0 ** -53 * 8


@pytest.mark.parametrize("N", [8, 9, 10, 11])
@pytest.mark.parametrize("nodal", [False, True])
def test_orders_and_coefficients(N, nodal):
    mesh = si.box_mesh((3, 1, 2), N, warp=0.1, perm_seed=1)
    lev = O.level_from_mesh(mesh)
    ctx = ctx_for(mesh, prec_copies=4)
    # the library's own factors: the oracle's differ by the roundings of D x, up to some N^2 2^-53, which is not looked at here
    F = ctx.geom(0).reshape(-1, 7, N + 1, N + 1, N + 1)
    G, B = [F[:, c] for c in range(6)], F[:, 6]
    u = si.uniform_field(mesh, 3, continuous=False)
    h1 = np.exp(0.5 * si.smooth_random_field(mesh, 5)) if nodal else 0.7
    for h2 in (0.0, 1.3):
        ref = O.ax_local(u.reshape(B.shape), G, B, lev.D, np.reshape(h1, B.shape) if nodal else h1, h2)
        for pairs in (False, True):
            w = H(ctx.ax(T(u), h1=1.0 if nodal else h1, h1_L=T(h1) if nodal else None, h2=h2, assemble=False, pairs=pairs))
            assert relmax(w, ref.ravel()) < (TOL if not pairs or N == 11 else 5e-12)
    ctx.close()


@pytest.mark.parametrize("N", [8, 9, 10, 11])
def test_scale_zero_and_elements_of_the_fp64_form(N):
    mesh = si.box_mesh((2, 2, 1), N, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    u = si.uniform_field(mesh, 9, continuous=False) * 2.0 ** -10
    w = H(ctx.ax(T(u), h2=0.5, assemble=False))
    for k in (-300, 0, 300):    # fixed point scales with u, bit for bit
        assert np.array_equal(H(ctx.ax(T(u * 2.0 ** k), h2=0.5, assemble=False)), w * 2.0 ** k)
    assert not np.any(H(ctx.ax(T(0 * u), assemble=False)))
    # beyond the exponents of fixed point: computed in FP64, the same to rounding at every point's own size
    far = H(ctx.ax(T(u * 2.0 ** 1000), h2=0.5, assemble=False)) * 2.0 ** -1000
    assert relmax(far, w) < TOL
    # an Inf or NaN stays in its element
    v = u.ravel().copy()
    v[3] = np.inf
    bad = H(ctx.ax(T(v), h2=0.5, assemble=False)).reshape(4, -1)
    assert not np.all(np.isfinite(bad[0])) and np.array_equal(bad[1:], w.reshape(4, -1)[1:])
    ctx.close()


def test_pair_calls_take_the_digits_of_a_large_mesh():
    mesh = si.box_mesh((13, 13, 13), 9, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=4)
    u = T(si.uniform_field(mesh, 2, continuous=False))
    assert np.array_equal(H(ctx.ax(u, h2=0.5, assemble=False)), H(ctx.ax(u, h2=0.5, assemble=False, pairs=True)))
    ctx.close()
