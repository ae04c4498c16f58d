"""The two-step kernel on the default tile against the cell passes, bit for bit,
with the route set and checked on both sides: the boxes of the tests are too
small for the rule to pick the two-step kernel for all of them, above all the
ones with a z CPML.  Sizes lie at the edges of the kernel's windows (24 columns,
20 rows), of its z shells (shells that meet, one plane between them), with the
sheet inside and beside a shell, with and without a fluence."""
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _grid(route, shape, npml, npml_z=None, sheet=None, antenna=None, fluence=True, seed=3, **pml):
    nx, ny, nz = shape
    walls = npml_z is not None
    init = W.random_state((nz, ny, nx), seed=seed)
    init[1][:, :, 0] = 0; init[2][:, :, 0] = 0     # tangential E on the walls
    init[0][:, 0, :] = 0; init[2][:, 0, :] = 0
    if walls:
        init[0][0] = 0; init[1][0] = 0
    g = fdtd.Grid(fdtd.make_grid_desc(nx, ny, nz, npml, 1 / 16, 1 / 18, 1 / 17, fluence=fluence, z_walls=walls,
                                      npml_z=npml_z or 0, **pml))
    if antenna:
        g.set_source(**antenna)
    if sheet is not None:
        g.set_wall_source(theta=0.4, w0=0.7, envelope="cw", ramp=0.2, plane=sheet)
    for c in range(6):
        g.set_field(c, init[c])
    g.debug_set_route(route)
    assert g.debug_route() == route
    return g


def _equal(a, b, fluence=True):
    assert a.n == b.n
    for c in range(6):
        x, y = a.field(c), b.field(c)
        assert torch.isfinite(x).all()
        assert torch.equal(x, y), (c, (x - y).abs().max().item())
    if fluence:
        assert torch.equal(a.fluence(), b.fluence())


WALLED = [
    # shape, npml, npml_z, sheet plane
    ((24, 20, 4), 3, 1, 1), ((25, 41, 12), 5, 5, 5), ((49, 39, 13), 6, 3, 2), ((48, 61, 40), 4, 8, None),
    ((96, 22, 9), 0, 2, 8), ((33, 33, 70), 6, 16, 16), ((47, 21, 6), 3, 2, 3), ((70, 44, 34), 7, 16, 33),
    ((130, 85, 11), 8, 1, 9), ((31, 20, 7), 0, 0, 6), ((200, 170, 5), 6, 1, 1),
]


@pytest.mark.parametrize("fluence", [True, False])
@pytest.mark.parametrize("shape,npml,npml_z,sheet", WALLED)
def test_z_walled_boxes(shape, npml, npml_z, sheet, fluence):
    a, b = (_grid(r, shape, npml, npml_z, sheet, fluence=fluence) for r in (1, 2))
    for g in (a, b):
        for n in (8, 3, 2):
            g.step(n)
    _equal(a, b, fluence)


def test_z_walls_with_stretched_shells():
    kw = dict(pml_kappa_max=3.0, pml_alpha_max=0.1)
    a, b = (_grid(r, (50, 44, 21), 7, 5, 5, **kw) for r in (1, 2))
    for g in (a, b):
        g.step(9)
    _equal(a, b)


@pytest.mark.parametrize("fluence", [True, False])
@pytest.mark.parametrize("shape,npml", [((26, 22, 1), 0), ((50, 41, 2), 6), ((230, 130, 3), 8), ((8, 8, 400), 2),
                                        ((28, 21, 150), 5)])
def test_thin_and_narrow_periodic_boxes(shape, npml, fluence):
    """Boxes the rule leaves on the cell passes."""
    a, b = (_grid(r, shape, npml, fluence=fluence) for r in (1, 2))
    for g in (a, b):
        g.step(7)
    _equal(a, b, fluence)


@pytest.mark.parametrize("npml_z,before", [(3, 2), (5, 4), (16, 3), (1, 6)])
def test_states_cross_the_routes(npml_z, before):
    """A state saved where the second copy of the z shells' E psi is current
    goes on alike on the cell passes, and one of theirs on the two-step kernel."""
    shape = (26, 23, 2 * npml_z + 9)
    a, b = (_grid(r, shape, 4, npml_z, npml_z) for r in (1, 2))
    for g in (a, b):
        g.step(before)
    sa, sb = a.save_state(), b.save_state()
    a.load_state(sb)
    b.load_state(sa)
    for g in (a, b):
        g.step(7)
    _equal(a, b)
    a.load_state(sa)
    b.load_state(sa)
    for g in (a, b):
        g.step(4)
    _equal(a, b)


@pytest.mark.parametrize("fluence", [True, False])
@pytest.mark.parametrize("steps", [130, 70, 7])
def test_batch_on_the_two_step_kernel(steps, fluence):
    """Two replays of the graph and the remainders, z-walled grids with a z CPML
    and the sheet beside antenna grids: the table-driven kernels against single
    grids on the cell passes."""
    antenna = dict(m=1, theta=0.35, r_center=10.0, ramp=0.1)
    boxes = [dict(shape=(50, 41, 16), npml=6, npml_z=4, sheet=4), dict(shape=(48, 44, 9), npml=6, antenna=antenna),
             dict(shape=(26, 61, 7), npml=3, npml_z=1), dict(shape=(44, 45, 11), npml=5, antenna=antenna, sheet=3),
             dict(shape=(30, 25, 8), npml=4, npml_z=3, sheet=7)]
    ref = [_grid(2, fluence=fluence, **kw) for kw in boxes]
    gs = [_grid(1, fluence=fluence, **kw) for kw in boxes]
    b = fdtd.Batch(gs)
    b.step(steps)
    b.sync()
    for r, g in zip(ref, gs):
        r.step(steps)
        _equal(g, r, fluence)
    b.close()


def test_route_is_refused_where_it_cannot_be():
    g = fdtd.Grid(fdtd.make_grid_desc(16, 16, 4, 2, 0.05, 0.05, 0.05, precision="f64"))
    assert g.debug_route() == 2
    for call in (lambda: g.debug_set_route(1), lambda: g.debug_set_route(3)):
        with pytest.raises(fdtd.FDTDError) as e:
            call()
        assert e.value.status == fdtd.FDTD_EINVAL
    f = fdtd.Grid(fdtd.make_grid_desc(16, 16, 4, 2, 0.05, 0.05, 0.05))
    b = fdtd.Batch([f])
    with pytest.raises(fdtd.FDTDError) as e:
        f.debug_set_route(1)
    assert e.value.status == fdtd.FDTD_ESTATE
    b.close()
