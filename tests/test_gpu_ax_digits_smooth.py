"""The digit element operators on fields whose fluxes are equal at mirror points (linear, quadratic and smooth ones), where
the sums of an even-odd line come closest to the bound of the fixed-point form; element by element against the FP64 form."""
import numpy as np
import pytest

import sem_inputs as si
from gpu_common import T, ctx_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# The FP64 form's own roundings on smooth data: 6 (N+1) 2^-53 of the terms of its sums, up to 2^3 times the largest result for
# terms of one size, and a derivative's terms are up to its row sum (below N^2 = 121) times the derivative
TOL = 6 * 12 * 2.0 ** -53 * 8 * 121


def _fp64_form(ctx, u, **kw):
    """Beyond the exponents of fixed point every element is computed in FP64."""
    return ctx.ax(u * 2.0 ** 1000, assemble=False, **kw) * 2.0 ** -1000


def _worst(w, ref, E):
    w, ref = w.view(E, -1), ref.view(E, -1)
    return float(((w - ref).abs().amax(1) / ref.abs().amax(1)).max())


@pytest.mark.parametrize("N", [4, 7, 8, 9, 10, 11])
@pytest.mark.parametrize("shape", [(2, 2, 2), (2, 3, 5)])
@pytest.mark.parametrize("nodal", [False, True])
def test_slopes_over_a_binade(N, shape, nodal):
    mesh = si.box_mesh(shape, N, warp=0.0, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=4)
    x, y, z = mesh["x"] - 0.5, mesh["y"] - 0.5, mesh["z"] - 0.5
    h1 = T(np.full(x.shape, 0.7)) if nodal else None
    kw = dict(h1=1.0 if nodal else 0.7, h1_L=h1, h2=0.0)
    for f in (x, y - z, x * x + 0.25 * z):
        u = T(f)
        ref = _fp64_form(ctx, u, **kw)
        for s in np.linspace(1.0, 2.0, 400, endpoint=False):
            for pairs in (False, True) if N in (7, 11) else (False,):
                w = ctx.ax(u * float(s), assemble=False, pairs=pairs, **kw)
                assert _worst(w, ref * float(s), mesh["E"]) < TOL, (s, pairs)
    ctx.close()


@pytest.mark.parametrize("N, side", [(7, 13), (8, 10), (9, 13), (10, 10), (11, 9)])
@pytest.mark.parametrize("nodal", [False, True])
def test_smooth_fields_on_some_thousand_elements(N, side, nodal):
    mesh = si.box_mesh((side,) * 3, N, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=4)
    h1 = T(np.exp(0.5 * si.smooth_random_field(mesh, 50))) if nodal else None
    for seed in range(8):
        u = T(si.smooth_random_field(mesh, seed))
        ref = _fp64_form(ctx, u, h1_L=h1, h2=0.5)
        for pairs in (False, True) if N in (7, 9, 11) else (False,):
            w = ctx.ax(u, h1_L=h1, h2=0.5, assemble=False, pairs=pairs)
            assert _worst(w, ref, mesh["E"]) < TOL, (seed, pairs)
    ctx.close()
