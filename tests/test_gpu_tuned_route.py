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


def _batch(shapes, walls=False):
    gs = []
    for nx, ny, nz in shapes:
        g = fdtd.Grid(fdtd.make_grid_desc(nx, ny, nz, 6, 0.05, 0.05, 0.05, z_walls=walls))
        if walls:
            g.set_wall_source(theta=0.4, w0=0.7, ramp=0.2, plane=1)
        else:
            g.set_source(theta=0.35, r_center=min(nx, ny) / 2 - 10, ramp=0.2)
        gs.append(g)
    return gs, fdtd.Batch(gs)


@pytest.mark.parametrize("walls", [False, True])
def test_tuned_batch_is_no_slower_than_an_untuned_one(walls):
    """Uneven grids on which the untuned batch's split of the SMs or, with
    walls, its two-step kernel beats the modes that can be chosen (1.1 to 1.5
    times): within 8 % of the untuned time after tuning."""
    shapes = [(420, 400, 40), (420, 400, 40), (160, 150, 40), (96, 90, 40)] if not walls else [(200, 200, 60)] * 3
    times = []
    for tune in (False, True):
        gs, b = _batch(shapes, walls)
        if tune:
            b.autotune(steps=4)
        b.step(64)
        b.sync()
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = 1e9
        for _ in range(5):
            e[0].record(gs[0].stream)
            b.step(64)
            e[1].record(gs[0].stream)
            b.sync()
            best = min(best, e[0].elapsed_time(e[1]))
        times.append(best)
        b.close()
    assert times[1] <= 1.08 * times[0], times


def test_a_mode_chosen_for_one_grid_leaves_the_others_alone():
    """The others keep their route, their shares of the SMs and the bits of the cell passes."""
    shapes = [(160, 150, 24), (140, 150, 24), (150, 140, 24)]
    ref, alone = _batch(shapes)
    alone.close()
    gs, b = _batch(shapes)
    ctas, routes = fdtd.batch_routes([g.desc for g in gs])
    assert routes.tolist() == [1, 1, 1]
    b.set_grid_mode(1, fdtd.BATCH_MODE_CELL8)
    assert [b.grid_mode(q) for q in range(3)] == [0, 1, 0]
    assert [b.grid_ctas(q) for q in range(3)] == ctas.tolist()
    b.step(70)
    b.sync()
    for g, x in zip(ref, gs):
        g.set_tile(5, 4, 1)
        g.step(70)
        for c in range(6):
            assert torch.equal(g.field(c), x.field(c)), c
        assert torch.equal(g.fluence(), x.fluence())
    b.close()
