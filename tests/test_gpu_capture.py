"""Steps on the default tile captured into the caller's graph: replays of an
even number of steps advance the state like that many steps each, whichever
kernels the route takes."""
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,walls", [("f32", False), ("f32", True), ("f64", False)])
@pytest.mark.parametrize("steps", [2, 4, 6, 8])
def test_replays_advance_the_state(precision, walls, steps):
    nx, ny, nz = 50, 44, 12
    d = fdtd.make_grid_desc(nx, ny, nz, 6, 1 / 16, 1 / 18, 1 / 17, precision=precision, z_walls=walls)
    init = W.random_state((nz, ny, nx), seed=9)
    init[1][:, :, 0] = 0; init[2][:, :, 0] = 0     # tangential E on the walls
    init[0][:, 0, :] = 0; init[2][:, 0, :] = 0
    if walls:
        init[0][0] = 0; init[1][0] = 0
    stream = torch.cuda.Stream()
    g, ref = fdtd.Grid(d, stream=stream), fdtd.Grid(d)
    ref.set_tile(5, 4, 1)
    for x in (g, ref):
        for c in range(6):
            x.set_field(c, init[c])
        x.step(3)
        x.sync()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        g.step(steps)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    ref.step(3 * steps)
    for c in range(6):
        assert torch.equal(g.field(c), ref.field(c)), c
    assert torch.equal(g.fluence(), ref.fluence())
    g.step(5)             # and plain steps go on from there
    ref.step(5)
    for c in range(6):
        assert torch.equal(g.field(c), ref.field(c)), c
