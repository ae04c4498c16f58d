"""A grid on its default tile takes its pairs of FP32 steps with the two-step
kernel.  The fields and the fluence are those of the cell passes (tile variant
5, chosen explicitly), bit for bit: both round every operation the same way.
Sizes lie at the edges of the kernel's windows (24 columns, 20 rows), with odd
and even widths and CPML depths, thin and tall boxes, z walls with and without
a z CPML, every source, and odd step counts."""
import numpy as np
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pair(shape, npml, steps, walls=False, npml_z=0, antenna=None, sheet=None, fluence=True, seed=3, **pml):
    """The same grid twice from the same random state: default tile, cell passes."""
    nx, ny, nz = shape
    init = W.random_state((nz, ny, nx), seed=seed)
    init[1][:, :, 0] = 0; init[2][:, :, 0] = 0     # tangential E on the walls
    init[0][:, 0, :] = 0; init[2][:, 0, :] = 0
    if walls:
        init[0][0] = 0; init[1][0] = 0
    out = []
    for tile in (None, (5, 4, 1)):
        d = fdtd.make_grid_desc(nx, ny, nz, npml, 1 / 16, 1 / 18, 1 / 17, precision="f32", fluence=fluence,
                                z_walls=walls, npml_z=npml_z, **pml)
        g = fdtd.Grid(d)
        if tile:
            g.set_tile(*tile)
        assert g.tile()[0] == 5
        if antenna:
            g.set_source(**antenna)
        if sheet:
            g.set_wall_source(**sheet)
        for c in range(6):
            g.set_field(c, init[c])
        for n in steps:
            g.step(n)
        g.sync()
        out.append(g)
    a, b = out
    assert a.n == b.n == sum(steps)
    for c in range(6):
        x, y = a.field(c), b.field(c)
        assert torch.isfinite(x).all()
        assert torch.equal(x, y), (c, (x - y).abs().max().item())
    if fluence:
        assert torch.equal(a.fluence(), b.fluence())
    return a, b


@pytest.mark.parametrize("shape,npml", [((2, 2, 1), 0), ((4, 4, 2), 1), ((23, 19, 3), 3), ((24, 20, 4), 5),
                                        ((25, 25, 5), 6), ((47, 39, 6), 7), ((48, 40, 7), 10), ((49, 41, 33), 8),
                                        ((97, 61, 9), 6), ((70, 130, 3), 0), ((130, 24, 12), 6), ((31, 200, 2), 4), ((400, 270, 4), 6),
                                        ((505, 330, 3), 8)])
def test_periodic_boxes(shape, npml):
    _pair(shape, npml, (6, 5))


@pytest.mark.parametrize("shape,npml,npml_z", [((24, 20, 2), 3, 0), ((25, 41, 12), 5, 5), ((49, 39, 13), 6, 3), ((345, 330, 14), 5, 2),
                                               ((48, 61, 40), 4, 8), ((96, 22, 9), 0, 2), ((33, 33, 200), 6, 16)])
def test_z_walled_boxes(shape, npml, npml_z):
    sheet = dict(theta=0.4, w0=0.7, envelope="cw", ramp=0.2, plane=max(1, npml_z))
    _pair(shape, npml, (8, 3), walls=True, npml_z=npml_z, sheet=sheet)


@pytest.mark.parametrize("kw", [dict(m=0), dict(m=2, pol="circ+", thickness=3.0), dict(m=1, pol="z", mode="TM"),
                                dict(m=1, pol="x", inject="tangential")])
def test_antenna(kw):
    src = dict(theta=0.35, r_center=24.0, thickness=1.0, ramp=0.1)
    src.update(kw)
    _pair((96, 83, 10), 8, (7, 8), antenna=src)


def test_antenna_and_sheet_in_a_periodic_box():
    _pair((60, 47, 11), 6, (6, 6), antenna=dict(theta=0.35, r_center=14.0, ramp=0.1),
          sheet=dict(theta=0.4, w0=0.5, envelope="gauss", T=0.7, T0=0.3, plane=0))


def test_stretched_shells_without_fluence():
    _pair((50, 44, 9), 7, (9,), fluence=False, pml_kappa_max=3.0, pml_alpha_max=0.1)


def test_checkpoint_between_the_routes():
    """A state saved on one route and loaded on the other goes on bit for bit
    (the E-side psi changes copy with every two-step launch)."""
    a, b = _pair((49, 41, 14), 6, (4, 3), walls=True, npml_z=4, sheet=dict(plane=4, ramp=0.2))
    sa, sb = a.save_state(), b.save_state()
    a.load_state(sb)
    b.load_state(sa)
    a.step(6)
    b.step(6)
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c))
    assert torch.equal(a.fluence(), b.fluence())


@pytest.mark.parametrize("npml_z,before", [(3, 2), (5, 4), (3, 3)])
def test_z_walled_state_holds_the_current_psi(npml_z, before):
    """A pair of steps leaves the z shells' E psi in the other copy; a state saved
    there goes on alike in a grid that stands on the first copy, and back."""
    shape = (26, 23, 40 * npml_z + 3)
    a, _ = _pair(shape, 4, (before,), walls=True, npml_z=npml_z)
    b, _ = _pair(shape, 4, (4,), walls=True, npml_z=npml_z, seed=5)
    state, other = a.save_state(), b.save_state()
    a.step(5)
    b.load_state(state)
    b.step(5)
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c)), c
    assert torch.equal(a.fluence(), b.fluence())
    a.load_state(other)
    b.load_state(other)
    a.step(3)
    b.step(3)
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c)), c


def test_batch_after_steps_and_a_state_loaded_into_a_batched_grid():
    """A batch reads the E-side psi copy its grids are at, also after a state
    of the other copy is loaded into a batched grid."""
    w = W.small(nx=50, ny=44, nz=8, npml=6, r_center=11.0, ramp=0.2)
    d = fdtd.make_grid_desc(w.nx, w.ny, w.nz, w.npml, w.dx, w.dx, w.dz, precision="f32")
    src = dict(theta=w.theta, r_center=w.r_center, ramp=w.ramp)
    ref, g = fdtd.Grid(d), fdtd.Grid(d)
    ref.set_tile(5, 4, 1)
    for x in (ref, g):
        x.set_source(**src)
    g.step(2)
    early = g.save_state()
    g.step(2)
    batch = fdtd.Batch([g])
    batch.step(64)
    g.load_state(early)
    batch.step(66)
    batch.sync()
    ref.step(2 + 66)
    for c in range(6):
        assert torch.equal(ref.field(c), g.field(c))
    assert np.array_equal(ref.fluence().cpu().numpy(), g.fluence().cpu().numpy())
    batch.close()
