"""Launch configurations: what igks_autotune returns and the untuned default's flux block can
be applied, change no bits, and anything else is refused."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_flux_blocks_bitwise_and_others_refused(precision):
    from paper_1709_00803_gb300 import igks
    m, fl = G.laminar_plate(), F.laminar_plate_flow()
    W0, out = F.perturbed_state(m, fl, seed=4, amp=0.02), []
    for block in (0, 32, 64, 128):
        ctx = igks.Context(precision=precision)
        s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
        launch = dict(sweep_threads=256, sweep_mode=1, sweep_cluster=1, groups=1)
        if block:
            ctx.set_launch(dict(launch, flux_block=block))
        else:
            choice = ctx.autotune(1)
            assert choice["flux_block"] in (32, 64, 128)
            ctx.set_launch(choice)
        for bad in (0, 16, 48, 96, 256):
            with pytest.raises(igks.IgksError) as e:
                ctx.set_launch(dict(launch, flux_block=bad))
            assert e.value.code == igks.EINVAL
        ctx.set_fields(s, W0)
        ctx.iterate(3)
        out.append(ctx.get_fields(s))
        ctx.destroy()
    for a in out[1:]:
        assert np.array_equal(a, out[0])
