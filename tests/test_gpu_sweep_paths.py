"""The narrow sweeps' paths against the one-launch-per-level sweeps, bitwise: every schedule
applies a cell's stencil entries in the same order with the same explicitly rounded
operations, so the increments and the state must be the same bits. The meshes reach levels
wider than the staged records (records read from global memory), neighbours that left the
shared-memory ring (the seam of an O-mesh), more levels than the shared-memory table holds,
levels wider than one round of a block, and stencils larger than a record with ghosts before
and after interior neighbours."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu


def _multicolour():
    from paper_1709_00803_gb300 import igks
    m = G.cavity(40)
    return m.renumbered(igks.order_cells(m, igks.ORDER_MULTICOLOR)[0])


CASES = {
    "two_levels_of_800": (_multicolour, F.cavity_flow),
    "o_mesh_seam": (lambda: G.naca_scaled(0.02, 0.4, 0.12, 9000, 1), F.naca_flow),
    "2101_levels": (lambda: G.flat_plate_quads(2100, 2, 1.1), F.laminar_plate_flow),
    "levels_of_150": (lambda: G.cavity(150), F.cavity_flow),
    "polygons": (lambda: G.refined_cavity(permute_seed=11), F.cavity_flow),
}


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_narrow_sweeps_bitwise_equal_level_launches(name, precision):
    from paper_1709_00803_gb300 import igks
    mk, flow_fn = CASES[name]
    m, fl = mk(), flow_fn()
    W0 = F.perturbed_state(m, fl, seed=61, amp=0.02)
    ref = None
    for mode, cluster, threads in ((2, 1, 0), (1, 1, 256), (1, 1, 32), (1, 2, 256)):
        ctx = igks.Context(precision=precision, sweep_mode=mode, sweep_cluster=cluster, sweep_threads=threads)
        s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
        ctx.set_fields(s, W0)
        ctx.iterate(2)
        out = [ctx.get_array(s, "dwstar"), ctx.get_array(s, "dw"), ctx.get_fields(s)]
        ctx.destroy()
        if ref is None:
            ref = out
        for a, b in zip(out, ref):
            assert np.array_equal(a, b), (mode, cluster, threads, np.abs(a - b).max())
