"""An expired device wait reaches the caller: the kernels with bounded waits
raise the grid's error word, and the calls that wait for the device report it.
The word is written from the host here, where a kernel would have raised it."""
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W
from tests.gpu_cases import gpu_grid

pytestmark = pytest.mark.gpu


def _raise_word(g, value=1):
    """Write the grid's error word: the last 256 bytes of its arena."""
    at = g._arena_ptr - g.arena.data_ptr() + fdtd.fdtd_required_bytes(g.desc) - 256
    torch.cuda.synchronize()
    g.arena[at:at + 4].view(torch.int32).fill_(value)
    torch.cuda.synchronize()


def _times_out(call):
    with pytest.raises(fdtd.FDTDError) as e:
        call()
    assert e.value.status == fdtd.FDTD_ETIMEOUT


@pytest.mark.parametrize("grids,bad", [(1, 0), (3, 2), (67, 63), (67, 66)])
def test_batch_sync_reports_a_grids_expired_wait(grids, bad):
    w = W.small(nx=32, ny=30, nz=4, npml=4, r_center=7.0, ramp=1.0)
    gs = [gpu_grid(w, "f32") for _ in range(grids)]
    b = fdtd.Batch(gs)
    b.step(2)
    b.sync()
    _raise_word(gs[bad])
    _times_out(b.sync)
    b.sync()              # reported once
    gs[bad].sync()
    b.close()


def test_word_raised_by_a_batch_on_another_stream():
    """A batch runs its grids on the first one's stream.  A grid with a stream
    of its own cannot wait for them, so a look at its word that comes before
    the batch's kernels raise it is not the last one."""
    w = W.small(nx=32, ny=30, nz=4, npml=4, r_center=7.0, ramp=1.0)
    d = fdtd.make_grid_desc(w.nx, w.ny, w.nz, w.npml, w.dx, w.dx, w.dz, courant=w.courant, precision="f32")
    other = torch.cuda.Stream()
    a, g = gpu_grid(w, "f32"), fdtd.Grid(d, stream=other)
    b = fdtd.Batch([a, g])
    b.step(4)
    b.close()
    g.sync()              # reads zero: nothing has expired yet
    _raise_word(g)
    _times_out(g.sync)
    g.sync()


@pytest.mark.parametrize("tile", [None, (7, 16, 1), (1, 8, 4)])
def test_word_raised_by_a_replayed_graph(tile):
    """Steps captured into the caller's graph run when it is replayed, which
    the grid does not see."""
    w = W.small(nx=32, ny=30, nz=4, npml=4, r_center=7.0, ramp=1.0)
    d = fdtd.make_grid_desc(w.nx, w.ny, w.nz, w.npml, w.dx, w.dx, w.dz, courant=w.courant, precision="f32")
    stream = torch.cuda.Stream()
    g = fdtd.Grid(d, stream=stream)
    if tile:
        g.set_tile(*tile)
    g.step(4)
    g.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        g.step(4)
    g.sync()
    graph.replay()
    _raise_word(g)
    _times_out(g.sync)
    g.sync()
    _raise_word(g)        # and after the next replay
    _times_out(g.sync)
