"""fdtd_step_timed runs and times the kernels fdtd_step takes, on the default
tile too, and leaves the same bits."""
import ctypes as C

import pytest
import torch

from paper_2102_12978_gb300 import fdtd

pytestmark = pytest.mark.gpu


def _grids(walls, route):
    out = []
    for _ in range(2):
        g = fdtd.Grid(fdtd.make_grid_desc(50, 44, 12, 6, 0.06, 0.06, 0.06, z_walls=walls, npml_z=3 if walls else 0))
        if walls:
            g.set_wall_source(theta=0.4, w0=0.5, ramp=0.1, plane=3)
        else:
            g.set_source(theta=0.35, r_center=10.0, ramp=0.1)
        g.debug_set_route(route)
        out.append(g)
    return out


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("route,steps,entries", [(1, 2, 1), (1, 8, 1), (1, 7, 3), (1, 1, 2), (2, 8, 2), (2, 7, 2)])
def test_default_tile(walls, route, steps, entries):
    a, b = _grids(walls, route)
    a.step(steps + 3)
    ms = b.step_timed(steps)
    assert len(ms) == entries and all(t > 0 for t in ms)
    b.step(3)
    assert a.n == b.n
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c)), c
    assert torch.equal(a.fluence(), b.fluence())


def test_odd_count_without_room_for_three_entries():
    a, b = _grids(False, 1)
    ms, n = (C.c_float * 2)(), C.c_int()
    fdtd.check(fdtd.lib().fdtd_step_timed(C.c_void_p(b.handle), 7, ms, 2, C.byref(n)), "fdtd_step_timed")
    assert n.value == 2 and ms[0] > 0 and ms[1] > 0
    a.step(7)
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c)), c
