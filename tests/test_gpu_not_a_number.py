"""Quotients and residuals that are not numbers, which finite states reach: the limiter ignores a
0 / 0 from slopes whose products underflow, as the oracle does, and the maximum norm is that of
the residuals that are numbers."""
import numpy as np
import pytest

import oracle as O
from igks_inputs import fields as F
from igks_inputs import meshgen as G

from _parity import assert_close, seeded

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


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_maximum_norm_ignores_what_is_not_a_number(precision):
    """Jumps of the velocity at Mach 8 reconstruct to pressures below zero and leave some
    residuals without a value; both kinds share blocks of the residual kernel."""
    torch = pytest.importorskip("torch")
    from paper_1709_00803_gb300 import igks
    m = G.tiny_quads(12, 10, skew=0.3, seed=3, bcs=("symmetry", "farfield"))
    fl = F.turbulent_plate_flow()
    fl.sa_on, fl.mach, fl.reynolds = 0, 8.0, 1e4
    ctx = igks.Context(precision=precision)
    s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
    W = seeded(m, fl, 71, amp=0.0)
    mx = W[1] * np.where(np.arange(m.n_cells) % 12 < 4, 1 + 0.5 * np.random.default_rng(1).uniform(-1, 1, m.n_cells), 1)
    W[3] += 0.5 * (mx ** 2 - W[1] ** 2) / W[0]          # the same pressure everywhere
    W[1] = mx
    ctx.set_fields(s, W)
    rc, st = ctx.iterate(1)
    res, area = ctx.get_array(s, "res")[0], ctx.get_array(s, "geom_cell")[0]
    ctx.destroy()
    some = [np.isnan(res[k:k + 64]).any() and np.isfinite(res[k:k + 64]).any() for k in range(0, m.n_cells, 64)]
    assert all(some)
    assert rc == igks.DIVERGED
    assert st[0]["res_inf"] == np.nanmax(np.abs(res))
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    r, a = torch.tensor(res, device="cuda"), torch.tensor(area, device="cuda")
    igks.residual_norms_noalloc(r.data_ptr(), a.data_ptr(), m.n_cells, out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    assert float(out.cpu()[0]) == st[0]["res_inf"]
