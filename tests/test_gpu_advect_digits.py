"""The dealiased advection operator in integer digits (csrc/advect_dig.cu): scaling, zero data, single components
against several, elements that go to the FP64 form."""
import numpy as np
import pytest

import oracle as O
import sem_inputs as si
from gpu_common import H, T, ctx_for, relmax

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the oracle's FP64 passes: about 2 (N+1) + 3 nq terms one behind the other, the derivative's row sums up to 40 of the
# field: 56 2^-53 40 = 2.5e-13
TOL = 2.5e-13


def _fields(mesh, n, seed):
    return [si.uniform_field(mesh, seed + q) for q in range(n)]


def _flat(fields):
    return torch.stack([T(f) for f in fields])


@pytest.mark.parametrize("N", [4, 5, 6, 7])
@pytest.mark.parametrize("prec", ["fp64", "fp64p"])
def test_components_scale_and_zero(N, prec):
    mesh = si.box_mesh((3, 1, 2), N, warp=0.1, perm_seed=1)
    lev = O.level_from_mesh(mesh)
    ctx = ctx_for(mesh, prec_copies=0)
    c, u = _fields(mesh, 3, 1), _fields(mesh, 2, 5)
    cub = O.cubature_setup(lev)
    w = ctx.advect(_flat(c), _flat(u), prec=prec)
    for q in range(2):
        assert relmax(H(w[q]), O.advect_local(lev, cub, np.stack(c), u[q]).ravel()) < (TOL if N > 4 or prec == "fp64" else 3e-11)
        assert torch.equal(ctx.advect(_flat(c), T(u[q]), prec=prec), w[q])
    if N > 4 or prec == "fp64":
        for k in (-300, 7):      # powers of two go through exactly
            assert torch.equal(ctx.advect(_flat(c), _flat(u) * 2.0 ** k, prec=prec), w * 2.0 ** k)
            assert torch.equal(ctx.advect(_flat(c) * 2.0 ** k, _flat(u), prec=prec), w * 2.0 ** k)
    assert not torch.any(ctx.advect(_flat(c) * 0.0, _flat(u), prec=prec))
    assert not torch.any(ctx.advect(_flat(c), _flat(u) * 0.0, prec=prec))
    ctx.close()


@pytest.mark.parametrize("value", [np.inf, np.nan, 2.0 ** 900])
@pytest.mark.parametrize("where", ["wind", "field"])
def test_elements_outside_fixed_point(value, where):
    mesh = si.box_mesh((2, 2, 1), 6, warp=0.1, perm_seed=0)
    ctx = ctx_for(mesh, prec_copies=0)
    c, u = _fields(mesh, 3, 1), _fields(mesh, 2, 5)
    plain = H(ctx.advect(_flat(c), _flat(u))).reshape(2, 4, -1)
    bad = c[1] if where == "wind" else u[1]
    scale = np.isfinite(value)
    if scale:
        (c if where == "wind" else u)[:] = [np.where(np.arange(4).reshape(4, 1, 1, 1) == 2, f * value, f)
                                           for f in (c if where == "wind" else u)]
    else:
        bad[2, 3, 1, 4] = value
    w = H(ctx.advect(_flat(c), _flat(u))).reshape(2, 4, -1)
    assert np.array_equal(w[:, [0, 1, 3]], plain[:, [0, 1, 3]])
    if scale:
        assert relmax(w[:, 2] / value, plain[:, 2]) < TOL
    else:
        assert not np.isfinite(w[1, 2]).any()
        assert np.isfinite(w[0, 2]).all() == (where == "field")
    ctx.close()
