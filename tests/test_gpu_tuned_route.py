"""The tuner has the default tile's way of running among its candidates, so
that a tuned grid is no slower than one left alone; the window order it adds
changes no result."""
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W
from tests.gpu_cases import gpu_grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sheet,walls", [(True, True), (False, True), (True, False)])
def test_tuned_grid_with_walls_keeps_the_two_step_kernel(sheet, walls):
    """Boxes on which the pairs of steps take two thirds of the cell passes'
    time (260 x 240 x 128 cells): the tuner keeps them."""
    d = fdtd.make_grid_desc(260, 240, 128, 6, 0.05, 0.05, 0.05, z_walls=walls)
    g = fdtd.Grid(d)
    if sheet:
        g.set_wall_source(theta=0.4, w0=0.7, ramp=0.2, plane=1)
    assert g.debug_route() == 1
    g.step(3)
    before = [g.field(c) for c in range(6)] + [g.fluence()]
    assert g.autotune(6) == (5, 4, 128)
    assert g.debug_route() == 1
    assert g.n == 3
    for c in range(6):
        assert torch.equal(g.field(c), before[c])
    assert torch.equal(g.fluence(), before[6])


def test_tuned_grid_on_the_cell_passes_stays_there():
    """Where the estimate picks the cell passes the default tile is no candidate of its own."""
    g = fdtd.Grid(fdtd.make_grid_desc(64, 48, 12, 6, 0.05, 0.05, 0.05, z_walls=True, npml_z=4))
    assert g.debug_route() == 2
    assert g.autotune(4)[0] == 5 and g.debug_route() == 2


@pytest.mark.parametrize("shape,npml", [((100, 90, 9), 8), ((70, 41, 2), 6), ((330, 390, 5), 8), ((24, 20, 1), 4)])
def test_whole_windows_first_changes_no_result(shape, npml):
    """Tile (7, 16, 3) against (7, 16, 1), also after the ranges were measured
    (measured ranges hold every window)."""
    nx, ny, nz = shape
    w = W.small(nx=nx, ny=ny, nz=nz, npml=npml, r_center=min(nx, ny) / 2 - npml - 3, steps=12, ramp=0.3)
    runs = []
    for lz, measure in ((1, False), (3, False), (3, True), (2, True)):
        g = gpu_grid(w, "f32", tile=(7, 16, lz))
        g.step(4)
        if measure:
            g.measure_balance()
        g.step(8)
        if measure:
            g.set_balance(0.4, 0.2)
        g.step(6)
        runs.append([g.field(c) for c in range(6)] + [g.fluence()])
    for other in runs[1:]:
        for x, y in zip(runs[0], other):
            assert torch.isfinite(x).all() and torch.equal(x, y)
