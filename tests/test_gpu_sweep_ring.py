"""Narrow sweeps of meshes whose levels are wider than the shared-memory ring, bitwise against
the one-launch-per-level sweeps; asked for, and as the default of a context in which a deep
mesh makes the schedule narrow for all."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

from test_sweep_ring import MESHES

pytestmark = pytest.mark.gpu

FLOWS = {"multicolour_plate": F.turbulent_plate_flow, "multicolour_airfoil_3936": F.naca_flow,
         "multicolour_airfoil_8120": F.naca_flow}
NAMES = ["multicolour_plate", "multicolour_airfoil_3936", "multicolour_airfoil_8120", "polygons_60", "polygons_100"]


def _run(solves, precision, iters=3, **opt):
    from paper_1709_00803_gb300 import igks
    ctx = igks.Context(precision=precision, **opt)
    for m, fl in solves:
        ctx.set_flow(ctx.mesh_upload(m), fl)
    for k, (m, fl) in enumerate(solves):
        ctx.init_freestream(k)
        ctx.set_fields(k, F.perturbed_state(m, fl, seed=61 + k, amp=0.02))
    ctx.iterate(iters)
    out = [ctx.get_array(0, "dwstar"), ctx.get_array(0, "dw"), ctx.get_fields(0)]
    ctx.destroy()
    return out


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", NAMES)
def test_levels_wider_than_the_ring_bitwise(name, precision):
    solve = (MESHES[name](), FLOWS.get(name, F.cavity_flow)())
    ref = _run([solve], precision, sweep_mode=2)
    assert all(np.isfinite(a).all() for a in ref)
    for cluster, threads in ((1, 256), (1, 128), (1, 64), (2, 256)):
        out = _run([solve], precision, sweep_mode=1, sweep_cluster=cluster, sweep_threads=threads)
        for a, b in zip(out, ref):
            assert np.array_equal(a, b), (cluster, threads, np.abs(a - b).max())


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_shallow_mesh_beside_a_deep_one_bitwise(precision):
    shallow = (MESHES["multicolour_plate"](), F.turbulent_plate_flow())
    deep = (G.plate_scaled(5003, 1), F.turbulent_plate_flow())
    for a, b in zip(_run([shallow, deep], precision), _run([shallow], precision, sweep_mode=2)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("groups", [1, 2, 5])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_broad_and_thin_solves_in_one_context(precision, groups):
    """Solves of few broad levels (clusters) between solves of many thin ones (a block each), in
    groups that hold either kind or both: the bits of each solve alone, and the launches of each kind."""
    from paper_1709_00803_gb300 import igks
    broad = (MESHES["multicolour_plate"](), F.turbulent_plate_flow())
    thin = (G.plate_scaled(2000, 1), F.turbulent_plate_flow())
    solves = [broad, thin, thin, broad, broad]
    alone = {id(s): _run([s], precision, iters=5)[2] for s in (broad, thin)}
    ctx = igks.Context(precision=precision, groups=groups, check_every=2)
    for m, fl in solves:
        ctx.set_flow(ctx.mesh_upload(m), fl)
    for k, (m, fl) in enumerate(solves):
        ctx.init_freestream(k)
        ctx.set_fields(k, F.perturbed_state(m, fl, seed=61, amp=0.02))
    # nine kernels a group and two sweeps for each kind in it; of two groups the second is the last solve
    assert ctx.launches_per_iteration() == {1: 13, 2: 13 + 11, 5: 5 * 11}[groups]
    ctx.iterate(5)
    for k, s in enumerate(solves):
        assert np.array_equal(ctx.get_fields(k), alone[id(s)])
    ctx.destroy()
