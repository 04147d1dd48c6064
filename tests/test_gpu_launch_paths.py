"""The iteration's kernels launched one behind the other in every way the context knows:
chained (one group, no events), with events between the kernels, without graphs, several
iterations in one graph, and in groups on streams. The launches change nothing but when a
kernel starts, so all give the same bits."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu


def _wide(n):
    from paper_1709_00803_gb300 import igks
    m = G.cavity(n)
    return m.renumbered(igks.order_cells(m, igks.ORDER_MULTICOLOR)[0])


MESHES = {"narrow": (lambda: [G.cavity(33), G.cavity(21)], F.cavity_flow),
          "wide": (lambda: [_wide(33), _wide(20)], F.cavity_flow),
          "plates": (lambda: [G.plate_scaled(1500, 1), G.plate_scaled(900, 2)], F.turbulent_plate_flow)}


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", list(MESHES))
def test_launch_paths_bitwise(name, precision, scheme):
    from paper_1709_00803_gb300 import igks
    mk, flow_fn = MESHES[name]
    meshes, ref = mk(), None
    for opt in (dict(timing=1), dict(), dict(use_graph=0), dict(check_every=3), dict(groups=2),
                dict(groups=2, use_graph=0)):
        ctx = igks.Context(precision=precision, **opt)
        for m in meshes:
            fl = flow_fn()
            fl.scheme = scheme
            ctx.set_flow(ctx.mesh_upload(m), fl)
        for k, m in enumerate(meshes):
            ctx.init_freestream(k)
            ctx.set_fields(k, F.perturbed_state(m, flow_fn(), seed=7 + k, amp=0.02))
        ctx.iterate(7)
        out = [ctx.get_fields(k) for k in range(len(meshes))]
        ctx.destroy()
        if ref is None:
            ref = out
        for a, b in zip(out, ref):
            assert np.isfinite(b).all()
            assert np.array_equal(a, b), (opt, np.abs(a - b).max())


@pytest.mark.parametrize("first", [0, 1])
def test_scheme_changed_after_build(first):
    """A context whose solves are all explicit launches no sweeps; changing a scheme between
    iterations changes the launches with it."""
    from paper_1709_00803_gb300 import igks
    m, out = G.cavity(24), []
    for use_graph in (1, 0):
        ctx = igks.Context(precision=igks.PREC_MIXED, use_graph=use_graph)
        sid = ctx.mesh_upload(m)
        for step, scheme in enumerate((first, 1 - first, first)):
            fl = F.cavity_flow()
            fl.scheme = scheme
            ctx.set_flow(sid, fl)
            if not step:
                ctx.init_freestream(sid)
                ctx.set_fields(sid, F.perturbed_state(m, fl, seed=2, amp=0.02))
            ctx.iterate(3)
            info = ctx.mesh_info(sid)               # few levels: one launch per level
            sweeps = 1 + info["levels_fwd"] + info["levels_bwd"]
            assert ctx.launches_per_iteration() == 8 + (0 if scheme == 1 and use_graph else sweeps)
        out.append(ctx.get_fields(sid))
        ctx.destroy()
    assert np.array_equal(out[0], out[1])
