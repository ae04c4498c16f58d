"""A read-out is written by a kernel only where all of it lies inside the
destination's allocation; every other destination goes through the runtime's
copy, which checks the range itself."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2102_12978_gb300 import fdtd

pytestmark = pytest.mark.gpu


def test_direct_output_stays_inside_the_allocation():
    torch.cuda.synchronize()
    driver = C.CDLL("libcuda.so.1")
    size = 8 << 20
    base = C.c_uint64()
    assert driver.cuMemAlloc_v2(C.byref(base), C.c_size_t(size)) == 0
    try:
        p = base.value
        g = fdtd.Grid(fdtd.make_grid_desc(16, 12, 4, 0, 0.05, 0.05, 0.05))
        assert g.debug_direct_output(p, size, 8)
        assert not g.debug_direct_output(p, size + 1, 8)
        assert g.debug_direct_output(p + size - 64, 64, 8)
        assert not g.debug_direct_output(p + size - 64, 65, 8)
        assert not g.debug_direct_output(p + 4, 64, 8) and g.debug_direct_output(p + 4, 64, 4)
        host = np.zeros(64)
        assert not g.debug_direct_output(host.ctypes.data, 64, 8)
        # a field that just fits is written to the allocation's last byte
        n = 16 * 12 * 4
        x = torch.arange(n, dtype=torch.float32, device="cuda").view(4, 12, 16)
        g.set_field(0, x)
        dst = p + size - 4 * n
        fdtd.fdtd_get_field(g.handle, 0, dst, True)
        out = np.zeros(n, np.float32)
        assert driver.cuMemcpyDtoH_v2(out.ctypes.data_as(C.c_void_p), C.c_uint64(dst), C.c_size_t(4 * n)) == 0
        assert np.array_equal(out, np.arange(n, dtype=np.float32))
        g.close()
    finally:
        torch.cuda.synchronize()
        driver.cuMemFree_v2(base)
