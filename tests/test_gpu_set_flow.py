"""igks_set_flow on a context that has iterated: a changed scheme leaves what the context holds
as it is, the times of the last iteration's kernels among it, whether or not the launches
change with the scheme; the iterations that follow are those of a fresh context."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solves,groups", [(1, 1), (2, 1), (2, 2)])
def test_scheme_change_keeps_kernel_times(solves, groups):
    from paper_1709_00803_gb300 import igks
    meshes = [G.cavity(24), G.cavity(17)][:solves]

    def context(schemes):
        ctx = igks.Context(timing=1, groups=groups)
        for m, scheme in zip(meshes, schemes):
            fl = F.cavity_flow()
            fl.scheme = scheme
            ctx.set_flow(ctx.mesh_upload(m), fl)
        for k, m in enumerate(meshes):
            ctx.init_freestream(k)
            ctx.set_fields(k, F.perturbed_state(m, F.cavity_flow(), seed=k, amp=0.02))
        return ctx

    ctx = context([0] * solves)
    ctx.iterate(2)
    before = ctx.kernel_times()
    W, sc = [ctx.get_fields(k) for k in range(solves)], [ctx.get_scalars(k) for k in range(solves)]
    fl = F.cavity_flow()
    fl.scheme = 1
    ctx.set_flow(0, fl)
    assert ctx.kernel_times() == before
    ctx.iterate(3)
    assert ctx.kernel_times() != before
    fresh = context([1, 0][:solves])
    for k in range(solves):
        fresh.set_fields(k, W[k])
        fresh.set_scalars(k, sc[k])
    fresh.iterate(3)
    for k in range(solves):
        assert np.array_equal(ctx.get_fields(k), fresh.get_fields(k))
    assert ctx.launches_per_iteration() == fresh.launches_per_iteration()
    ctx.destroy(); fresh.destroy()
