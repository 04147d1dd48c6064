"""The shared-memory ring of the narrow sweeps on meshes with levels wider than the ring (host
logic, no GPU). Position q of a sweep writes ring slot q % ring, and the cells of a level are
worked on in no order. So a stencil entry may name a ring slot only if nothing else that
writes this slot lies in the neighbour's own level, in the reader's or between them; a side
slot only if the neighbour's level is finished two levels before the reader's."""
import ctypes as C

import numpy as np
import pytest

from igks_inputs import meshgen as G


def _multicolour(m):
    from paper_1709_00803_gb300 import igks
    return m.renumbered(igks.order_cells(m, igks.ORDER_MULTICOLOR)[0])


MESHES = {
    "multicolour_plate": lambda: _multicolour(G.plate_scaled(5003, 1)),
    "multicolour_airfoil_3936": lambda: _multicolour(G.naca_scaled(0.0, 0.0, 0.12, 4000, 3)),
    "multicolour_airfoil_8120": lambda: _multicolour(G.naca_scaled(0.0, 0.0, 0.12, 8000, 3)),
    "polygons_60": lambda: G.refined_cavity(60, permute_seed=11),
    "polygons_100": lambda: G.refined_cavity(100, permute_seed=11),
    "multicolour_cavity": lambda: _multicolour(G.cavity(70)),
    "o_mesh": lambda: G.naca_scaled(0.02, 0.4, 0.12, 9000, 1),
}


def schedule(m, precision, forward):
    """Levels, order, stencil lists and ring size of the library's narrow schedule."""
    from paper_1709_00803_gb300 import igks
    n, ip = m.n_cells, igks._ip
    fc = np.ascontiguousarray(m.face_cells, dtype=np.int32).ravel()
    fb = np.ascontiguousarray(m.face_bc, dtype=np.int32)
    lvl, ptr = np.zeros(n + 1, np.int32), np.zeros(n + 1, np.int32)
    order, j, slot = np.zeros(n, np.int32), np.zeros(2 * m.n_faces, np.int32), np.zeros(2 * m.n_faces, np.int32)
    nl, ring = C.c_int32(), C.c_int32()
    rc = igks.lib().igks_sweep_schedule_(n, m.n_faces, ip(fc), ip(fb), precision, int(forward), ip(lvl), C.byref(nl),
                                         ip(order), ip(ptr), ip(j), ip(slot), C.byref(ring))
    assert rc == igks.OK
    return lvl[:nl.value + 1], order, ptr, j[:ptr[-1]], slot[:ptr[-1]], ring.value


@pytest.mark.parametrize("forward", [True, False])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", list(MESHES))
def test_ring_slots_are_written_by_the_neighbour_alone(name, precision, forward):
    m = MESHES[name]()
    lvl, order, ptr, j, slot, ring = schedule(m, precision, forward)
    n = m.n_cells
    assert sorted(order.tolist()) == list(range(n)) and lvl[0] == 0 and lvl[-1] == n
    pos = np.empty(n, np.int64)
    pos[order] = np.arange(n)
    level = np.searchsorted(lvl, np.arange(n), side="right") - 1          # of a position
    reader = np.repeat(np.arange(n), np.diff(ptr))
    q = pos[np.maximum(j, 0)]
    inring = (j >= 0) & (slot >= 0) & (slot < ring)
    assert np.array_equal(slot[inring], q[inring] % ring)
    # the nearest positions that share the slot: behind the reader's level, before the neighbour's
    assert not (inring & (q + ring < lvl[level[reader] + 1])).any()
    assert not (inring & (q - ring >= lvl[level[q]])).any()
    side = (j >= 0) & (slot >= ring)
    assert (level[q[side]] <= level[reader[side]] - 3).all()
    own = level[reader[side]].astype(np.int64) * 1000 + slot[side]
    assert np.unique(own).size == own.size                                # one neighbour a side slot and level
    assert (level[q[j >= 0]] < level[reader[j >= 0]]).all()


def test_levels_wider_than_the_ring_are_among_the_meshes():
    wide = {1024: 0, 2048: 0}
    for mk in MESHES.values():
        m = mk()
        for precision in (0, 1):
            lvl, *_, ring = schedule(m, precision, True)
            wide[ring] += np.diff(lvl).max() > ring
    assert wide[1024] >= 4 and wide[2048] >= 2
