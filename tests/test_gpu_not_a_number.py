"""Quotients that are not numbers, which finite states reach: the limiter ignores a 0 / 0 from
slopes whose products underflow, as the oracle does."""
import numpy as np
import pytest

import oracle as O
from igks_inputs import fields as F
from igks_inputs import meshgen as G

from _parity import assert_close

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.mark.parametrize("beside", [0, 1])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("limiter", [1, 2])
def test_limiter_of_slopes_that_underflow(limiter, sign, beside):
    """One cell's momentum differs from its neighbours' by 1e-120: at that extremum the
    Venkatakrishnan quotient is 0 / 0 with venkat_k = 0. (beside: a mesh that makes the group
    large, whose gradients are formed by one thread per cell.)"""
    from paper_1709_00803_gb300 import igks
    m, fl = G.cavity(12), F.cavity_flow()
    fl.limiter, fl.venkat_k = limiter, 0.0
    W = np.repeat(np.array([1.0, 0.0, 0.0, 50.0, 0.0])[:, None], m.n_cells, axis=1)
    W[1, 66] = sign * 1e-120
    ctx = igks.Context()
    for q, f in [(m, fl)] + [(G.cavity(100), F.cavity_flow())] * beside:
        ctx.set_flow(ctx.mesh_upload(q), f)
    for k in range(1 + beside):
        ctx.init_freestream(k)
    ctx.set_fields(0, W)
    ora = O.Oracle(m, fl)
    ora.set_W(W)
    ctx.iterate(1); ora.iterate(1)
    phi = ctx.get_array(0, "phi")
    assert np.isfinite(phi).all()
    assert_close("phi", phi, ora.get(O.ORA_PHI), TOL)
    assert_close("W", ctx.get_fields(0), ora.get(O.ORA_W), TOL)
    ctx.destroy()
