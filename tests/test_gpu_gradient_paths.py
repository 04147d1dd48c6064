"""Gradients, limiter and time step with four threads per cell (small groups) against one
thread per cell (the same solve beside a mesh that makes the group large): the same bits."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu

MESHES = {
    "hybrid_plate": (lambda: G.plate_scaled(1003, 1), F.turbulent_plate_flow),
    "o_mesh": (lambda: G.naca_scaled(0.0, 0.0, 0.12, 4000, 3), F.naca_flow),
    "polygons": (lambda: G.refined_cavity(permute_seed=11), F.cavity_flow),
    "one_row": (lambda: G.flat_plate_quads(7, 1, 1.1), F.laminar_plate_flow),
}


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("name", list(MESHES))
def test_four_threads_per_cell_bitwise(name, limiter):
    from paper_1709_00803_gb300 import igks
    mk, flow_fn = MESHES[name]
    m, fl = mk(), flow_fn()
    fl.limiter = limiter
    W0 = F.perturbed_state(m, fl, seed=3, amp=0.02)
    out = []
    for beside in (0, 1):
        ctx = igks.Context(precision=igks.PREC_FP64)
        meshes = [(m, fl)] + [(G.cavity(100), F.cavity_flow())] * beside
        for q, f in meshes:
            ctx.set_flow(ctx.mesh_upload(q), f)
        for k in range(len(meshes)):
            ctx.init_freestream(k)
        ctx.set_fields(0, W0)
        _, st = ctx.iterate(1)
        out.append([ctx.get_array(0, n) for n in ("grad", "phi", "lambda_c", "res")] + [ctx.get_fields(0), st[0]["dt"]])
        ctx.destroy()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
