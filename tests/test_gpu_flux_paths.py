"""The flux's branches: normal velocities inside the tail table (up to six standard deviations
of the Maxwellian) and beyond it, against the oracle at the FP64
parity bar; and limited gradients, which pass from the gradient kernel to the flux, with the
solves split into groups on streams of their own (bitwise equal to one group)."""
import numpy as np
import pytest

import oracle as O
from igks_inputs import fields as F
from igks_inputs import meshgen as G

from _parity import assert_close, make_pair, seeded

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mach", [0.05, 1.0, 2.5, 5.0, 8.0])
def test_flux_over_normal_mach_numbers(mach, precision):
    """Mach 5 puts |U| at 5.9 standard deviations (the last table nodes), 8 at 9.5 (beyond).
    A box with a symmetry plane and free stream around: no wall or outflow, whose ghosts have
    no flux at supersonic speeds (negative pressure behind the reconstruction)."""
    m = G.tiny_quads(12, 10, skew=0.3, seed=3, bcs=("symmetry", "farfield"))
    fl = F.turbulent_plate_flow()
    fl.sa_on, fl.mach, fl.reynolds = 0, mach, 1e4
    ctx, sid, ora = make_pair(m, fl, seeded(m, fl, 71, amp=0.002), precision=precision)
    ctx.iterate(1); ora.iterate(1)
    assert_close("flux", ctx.get_array(sid, "flux"), ora.get(O.ORA_FLUX), TOL)


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_limited_solves_in_groups_bitwise_equal_one_group(precision):
    from paper_1709_00803_gb300 import igks
    cases = [(G.naca_scaled(0.02, 0.4, 0.12, 3000 + 700 * k, k), F.naca_flow(0.2 + 0.1 * k)) for k in range(4)]
    for _, fl in cases[2:]:
        fl.limiter = F.LIMITER_VENKAT
    ref = None
    for groups in (1, 2, 4):
        ctx = igks.Context(precision=precision, sweep_mode=1, groups=groups, check_every=4)
        for m, fl in cases:
            ctx.set_flow(ctx.mesh_upload(m), fl)
        for k, (m, fl) in enumerate(cases):
            ctx.init_freestream(k)
            ctx.set_fields(k, seeded(m, fl, 80 + k, amp=0.02))
        ctx.iterate(9)
        out = [ctx.get_fields(k) for k in range(len(cases))]
        ctx.destroy()
        ref = ref or out
        for a, b in zip(out, ref):
            assert np.array_equal(a, b), groups
