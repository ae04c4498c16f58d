"""Read-outs into device arrays of any alignment and row length, and through
the host, against each other: the field copy and the fluence reducer take
16-byte accesses where row length and destination allow them."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2102_12978_gb300 import fdtd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(2, 2, 1), (5, 3, 2), (32, 9, 4), (33, 7, 5), (34, 6, 3), (200, 45, 9), (257, 12, 3)])
def test_device_and_host_readouts_agree(precision, shape):
    nx, ny, nz = shape
    g = fdtd.Grid(fdtd.make_grid_desc(nx, ny, nz, 0, 0.05, 0.05, 0.05, precision=precision))
    gen = np.random.default_rng(nx)
    init = [gen.standard_normal((nz, ny, nx)) for _ in range(6)]
    for c in range(6):
        g.set_field(c, init[c])
    for c in range(6):
        assert torch.equal(g.field(c), torch.as_tensor(init[c]).to(g.dtype).cuda())
    g.step(3)
    n = nx * ny * nz
    host = np.zeros(n, np.float64)
    fdtd.fdtd_fluence(g.handle, host.ctypes.data, False, False)
    assert np.array_equal(g.fluence().cpu().numpy().ravel(), host) and host.any()
    for shift in (0, 1, 3):        # elements off a 16-byte boundary
        buf = torch.full((n + 8,), 7.0, dtype=g.dtype, device="cuda")
        fdtd.fdtd_get_field(g.handle, 1, buf.data_ptr() + shift * buf.element_size(), True)
        assert torch.equal(buf[shift:shift + n].view(nz, ny, nx), g.field(1))
        assert (buf[:shift] == 7).all() and (buf[shift + n:] == 7).all()
        flu = torch.full((n + 8,), 7.0, dtype=torch.float64, device="cuda")
        fdtd.fdtd_fluence(g.handle, flu.data_ptr() + 8 * shift, True, False)
        assert np.array_equal(flu[shift:shift + n].cpu().numpy(), host)
        assert (flu[:shift] == 7).all() and (flu[shift + n:] == 7).all()


def test_fluence_of_tiny_and_large_terms():
    """Accumulators from denormal to large values convert as the host does."""
    g = fdtd.Grid(fdtd.make_grid_desc(64, 8, 4, 0, 0.05, 0.05, 0.05, precision="f32"))
    scale = torch.logspace(-24, 12, 64).view(1, 1, 64)
    for c in range(6):
        g.set_field(c, scale * (1.0 + 0.1 * c) * torch.ones(g.shape))
    g.step(2)
    dev = g.fluence().cpu().numpy()
    host = np.zeros(g.shape)
    fdtd.check(fdtd.lib().fdtd_fluence(C.c_void_p(g.handle), C.c_void_p(host.ctypes.data), 0, 0), "fdtd_fluence")
    assert np.array_equal(dev, host, equal_nan=True)   # (the largest squares overflow FP32)
    buf = g.save_state().cpu().numpy().tobytes()
    acc = np.frombuffer(buf, dtype=np.float32)           # the accumulator's bits are in the state
    vals = dev[dev > 0].astype(np.float32)
    assert np.isin(vals[:16], acc).any()
