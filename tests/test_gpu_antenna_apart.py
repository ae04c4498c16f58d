"""FP64 grids add the antenna's terms inside the cell passes or in a pass of
their own, by the warps that hold antenna columns; the bits are the same.  A
batch keeps them inside: single grids on both sides of the line against it."""
import numpy as np
import pytest
import torch

from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W
from tests.gpu_cases import gpu_grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,r,thick,apart", [((48, 40, 16), 10.0, 1.0, False), ((96, 90, 40), 14.0, 3.0, False),
                                                 ((50, 50, 300), 16.0, 1.0, True), ((96, 96, 64), 24.0, 20.0, True),
                                                 ((70, 64, 90), 18.0, 8.0, False), ((70, 64, 91), 18.0, 8.0, True)])
def test_inside_and_apart_agree(shape, r, thick, apart):
    nx, ny, nz = shape
    w = W.small(nx=nx, ny=ny, nz=nz, npml=6, r_center=r, thickness=thick, ramp=0.2)
    a, b = gpu_grid(w, "f64"), gpu_grid(w, "f64")
    s, keep = fdtd.make_annulus_desc(m=w.m, theta=w.theta, pol=w.pol, mode=w.mode, E0=w.E0, r_center=r, thickness=thick)
    mask = fdtd.source_coefficients(a.desc, s)[1] & 0x3f
    rows = np.zeros((ny, -(-nx // 32) * 32), bool)
    rows[:, :nx] = mask != 0
    warps = int(rows.reshape(ny, -1, 32).any(axis=2).sum())
    assert (warps * nz >= 8000) == apart, warps * nz
    batch = fdtd.Batch([b])
    a.step(6)
    batch.step(6)
    batch.sync()
    for c in range(6):
        assert torch.equal(a.field(c), b.field(c)), c
    assert torch.equal(a.fluence(), b.fluence())
    batch.close()
