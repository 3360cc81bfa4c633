"""The digit element operators with a nodal h1 of high contrast inside an element: points that see only small values of h1 keep
the accuracy of those values."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, relmax

pytestmark = pytest.mark.gpu

# FP64's roundings on random u: 6 (N+1) 2^-53 of the terms, which are up to 2^3 times the result's maximum; h1 itself varies by
# e^(2 * 0.5 * 3) = 2^4.4 over the points compared, and the terms with it
TOL = 6 * 12 * 2.0 ** -53 * 8 * 2.0 ** 4.4


def _contrast(mesh, N, low):
    """h1 = low exp(g / 2), but exp(g / 2) along the edge j = k = 0 of every element."""
    h1 = np.exp(0.5 * np.clip(si.smooth_random_field(mesh, 5), -3, 3))
    edge = np.zeros((N + 1,) * 3, dtype=bool)
    edge[0, 0, :] = True
    return np.where(edge, h1, low * h1)


@pytest.mark.parametrize("N", [4, 5, 6, 7, 8, 9, 10, 11])
@pytest.mark.parametrize("low", [2.0 ** -6, 2.0 ** -12, 2.0 ** -40, 2.0 ** -300, 0.0])
def test_small_values_beside_large_ones(N, low):
    mesh = si.box_mesh((3, 2, 2), N, warp=0.1, perm_seed=1)
    ctx = ctx_for(mesh, prec_copies=4)
    F = ctx.geom(0).reshape(-1, 7, N + 1, N + 1, N + 1)
    G, B = [F[:, c] for c in range(6)], F[:, 6]
    D = O.level_from_mesh(mesh).D
    h1 = _contrast(mesh, N, low).reshape(B.shape)
    u = si.uniform_field(mesh, 3, continuous=False)
    ref = O.ax_local(u.reshape(B.shape), G, B, D, h1, 0.0).reshape(B.shape)
    for pairs in (False, True) if N in (7, 11) else (False,):
        w = H(ctx.ax(T(u), h1_L=T(h1), assemble=False, pairs=pairs)).reshape(B.shape)
        assert relmax(w, ref) < TOL
        # w at a point takes h1 on the three lines through it: with j, k > 0 none of them meets the edge
        for e in range(mesh["E"]):
            if low:
                assert relmax(w[e, 1:, 1:], ref[e, 1:, 1:]) < TOL
            else:
                assert not np.any(w[e, 1:, 1:])
    ctx.close()


@pytest.mark.parametrize("low", [1.0, 2.0 ** -10])
def test_one_launch_solve_with_elements_of_the_fp64_form(low):
    mesh = si.box_mesh((3, 3, 2), 7, warp=0.1, perm_seed=1, dirichlet=("x0",))
    one, chain = ctx_for(mesh, prec_copies=0), ctx_for(mesh, prec_copies=0, spin_limit=1 << 20)
    b = T(si.gaussian_assembled_rhs(mesh, 0))
    h1 = T(_contrast(mesh, 7, low))
    xa, xb = (H(c.solve(b, h1_L=h1, h2=0.5, tol=0.0, maxit=5, rhs="assembled", raise_on_error=False)[0]) for c in (one, chain))
    # sums of at most 4e5 terms of one sign, 30 of them, growing by less than the 1e2 by which the coefficients of the iteration
    # vary, and by the contrast
    assert np.abs(xa - xb).max() <= 30 * 4e5 ** 0.5 * 2.0 ** -53 * 1e2 / low * np.abs(xb).max()
    one.close()
    chain.close()


@pytest.mark.parametrize("N", [7, 11])
def test_pair_calls_keep_48_bits_of_small_values(N):
    """h1 spans 2^12 and a little: within what a pair call leaves in digits."""
    mesh = si.box_mesh((3, 2, 2), N, warp=0.1, perm_seed=1)
    ctx = ctx_for(mesh, prec_copies=4)
    u = T(si.uniform_field(mesh, 3, continuous=False))
    low = 2.0 ** -12
    edge = np.zeros((N + 1,) * 3, dtype=bool)
    edge[0, 0, :] = True
    ramp = np.broadcast_to(1.0 + np.arange(N + 1) / (2.0 * N + 2.0), mesh["x"].shape)   # 1 to 1.5: one binade
    h1 = T(np.where(edge, ramp, low * ramp))
    ref, w = (H(ctx.ax(u, h1_L=h1, assemble=False, pairs=p)).reshape(mesh["x"].shape) for p in (False, True))
    for e in range(mesh["E"]):
        # the terms' 2^-48, as for FP64's 2^-53 above
        assert relmax(w[e, 1:, 1:], ref[e, 1:, 1:]) < 6 * 12 * 2.0 ** -48 * 8 * 1.5
    # a pair call takes the digits there, the FP64 call the FP64 form
    assert not np.array_equal(w, ref)
    ctx.close()
