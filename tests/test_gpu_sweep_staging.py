"""Record staging of the narrow sweeps in solves with some levels wider than the buffers: every
level's records are brought into shared memory as far as they fit. Bitwise against the
one-launch-per-level sweeps on a mesh of wide levels before (forward) and behind (backward) a
hundred thin ones, on levels around the buffers' and the ring's sizes, and on two levels only; and a copy
that never lands is noticed in such solves as in others."""
import numpy as np
import pytest

from igks_inputs import fields as F
from igks_inputs import meshgen as G

pytestmark = pytest.mark.gpu


def _half_multicolour(n, swap):
    """A cavity whose first half (swap: second half) of cells is numbered by colours."""
    from paper_1709_00803_gb300 import igks
    m = G.cavity(n)
    half = m.n_cells // 2
    col = igks.order_cells(m, igks.ORDER_MULTICOLOR)[0]
    lo, hi = np.arange(half), np.arange(half, m.n_cells)
    return m.renumbered(np.concatenate([lo, col[col >= half]] if swap else [col[col < half], hi]))


def _rows_by_parity(nx, ny):
    """Every row's even cells, then its odd ones: two levels of nx / 2 cells a row."""
    row = np.concatenate([np.arange(0, nx, 2), np.arange(1, nx, 2)])
    return G.flat_plate_quads(nx, ny, 1.1).renumbered((np.arange(ny)[:, None] * nx + row).ravel())


MESHES = {
    "wide_then_thin": lambda: _half_multicolour(90, False),
    "less_wide_then_thin": lambda: _half_multicolour(60, False),
    "thin_then_wide": lambda: _half_multicolour(90, True),
    "levels_of_500": lambda: _rows_by_parity(1000, 20),
    "levels_of_1000": lambda: _rows_by_parity(2000, 12),
    "levels_of_380": lambda: G.flat_plate_quads(420, 380, 1.01),
    "levels_of_600": lambda: G.cavity(600),
    "two_levels_of_9800": lambda: G.cavity(140).renumbered(
        np.argsort(np.add(*np.divmod(np.arange(140 * 140), 140)) % 2, kind="stable")),
}
PLATES = ("levels_of_380", "levels_of_500", "levels_of_1000")


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", list(MESHES))
def test_staged_levels_bitwise_and_starved_copy_noticed(name, precision):
    from paper_1709_00803_gb300 import igks
    m, fl = MESHES[name](), F.laminar_plate_flow() if name in PLATES else F.cavity_flow()
    W0 = F.perturbed_state(m, fl, seed=5, amp=0.01)
    ref = None
    for mode, threads in ((2, 0), (1, 256), (1, 64)):
        ctx = igks.Context(precision=precision, sweep_mode=mode, sweep_threads=threads)
        s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
        ctx.set_fields(s, W0)
        ctx.iterate(2)
        out = [ctx.get_array(s, "dwstar"), ctx.get_array(s, "dw"), ctx.get_fields(s)]
        ctx.destroy()
        ref = ref or out
        for a, b in zip(out, ref):
            assert np.isfinite(a).all()
            assert np.array_equal(a, b), (mode, threads, np.abs(a - b).max())
    ctx = igks.Context(precision=precision, sweep_mode=1, wait_limit=4096, starve_test=1, check_every=1)
    s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
    ctx.set_fields(s, W0)
    rc, st = ctx.iterate(1)
    info = ctx.mesh_info(s)
    if m.n_cells > 512 * max(info["levels_fwd"], info["levels_bwd"]):   # in clusters: no copies to wait for
        assert rc == igks.OK and name.startswith(("levels_of_500", "levels_of_1000", "two_levels"))
        ctx.destroy()
        return
    assert rc == igks.TIMEOUT and st[s]["state"] == igks.TIMEOUT
    assert np.array_equal(ctx.get_fields(s), W0)
    ctx.destroy()
