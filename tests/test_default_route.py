"""Which kernel a pair of FP32 steps takes on the default tile: the one estimated
to be faster.  The boxes are ones where the two differ by more than 15 %, with
both times as measured on a GB300 (us per step)."""
import pytest

from paper_2102_12978_gb300 import fdtd

# (nx, ny, nz, npml), npml_z (None: z-periodic), sheet, fluence, two-step kernel, cell passes
BOXES = [
    # planes too few to pay for a window's start
    ((1024, 1024, 1, 6), None, False, True, 57.4, 20.5), ((1024, 1024, 2, 6), None, False, False, 54.8, 28.2),
    ((2048, 2048, 1, 16), None, False, True, 224.0, 78.8), ((560, 560, 3, 6), None, False, True, 27.7, 20.5),
    ((400, 400, 4, 0), None, False, True, 18.5, 14.4), ((2048, 2048, 2, 6), None, False, True, 260.6, 179.9),
    # enough of them
    ((560, 560, 12, 6), None, False, True, 55.8, 75.0), ((2048, 2048, 6, 6), None, False, True, 398.0, 542.0),
    ((1024, 1024, 8, 6), None, False, False, 94.2, 111.6), ((332, 332, 46, 6), None, False, False, 47.2, 80.4),
    ((256, 256, 128, 16), None, False, True, 109.9, 174.2), ((512, 512, 64, 16), None, False, True, 179.7, 335.0),
    # narrow boxes: windows mostly past the walls, or filling them
    ((32, 32, 1024, 6), None, False, True, 35.9, 25.1), ((26, 26, 4096, 6), None, False, True, 121.0, 91.0),
    ((20, 20, 4096, 5), None, False, True, 37.9, 68.8), ((100, 100, 1024, 6), None, False, True, 150.9, 270.7),
    ((24, 1024, 256, 6), None, False, True, 75.9, 174.6), ((16, 2048, 64, 4), None, False, False, 34.0, 66.6),
    ((16, 16, 4096, 4), None, False, True, 33.0, 50.4), ((160, 160, 12, 6), None, False, True, 10.3, 12.9),
    # z walls and sheets
    ((560, 560, 2, 6), 0, False, True, 29.8, 20.2), ((560, 560, 6, 6), 1, False, False, 66.3, 33.9),
    ((360, 360, 6, 6), 1, False, True, 33.9, 20.5), ((64, 64, 640, 6), 16, False, True, 92.4, 69.7),
    ((1024, 1024, 12, 6), 2, False, False, 259.0, 205.6), ((411, 411, 192, 16), 16, False, True, 508.0, 684.0),
    ((340, 340, 192, 16), 4, False, True, 358.9, 464.5), ((40, 1024, 120, 6), 3, False, True, 104.6, 182.1),
    ((205, 205, 800, 6), 0, False, True, 472.7, 749.7), ((200, 200, 800, 6), 4, False, True, 469.7, 713.8),
    ((332, 332, 46, 6), None, True, True, 78.5, 108.4), ((560, 560, 3, 6), None, True, True, 30.8, 20.6),
]


@pytest.mark.parametrize("box,npml_z,sheet,fluence,two,cells", BOXES)
def test_the_faster_kernel_is_taken(box, npml_z, sheet, fluence, two, cells):
    nx, ny, nz, npml = box
    d = fdtd.make_grid_desc(nx, ny, nz, npml, 0.05, 0.05, 0.05, fluence=fluence, z_walls=npml_z is not None,
                            npml_z=npml_z or 0)
    est_two, est_cells = fdtd.route_us(d, sheet)
    assert (est_two < est_cells) == (two < cells), (est_two, est_cells)


def test_estimates_grow_with_the_box_and_shrink_with_the_ctas():
    """No size wraps or divides by nothing: one plane, one window, the tallest
    and the widest box of the 2^31-element limit."""
    for shape in ((2, 2, 1), (2, 2, 30000000), (40000, 50000, 1), (8, 8, 16384), (1200, 1200, 1400)):
        for walls in (False, True):
            if walls and shape[2] < 2:
                continue
            d = fdtd.make_grid_desc(*shape, 0, 0.05, 0.05, 0.05, z_walls=walls)
            t, c = fdtd.route_us(d)
            assert 0 < t < 1e9 and 0 < c < 1e9
            assert fdtd.route_us(d, ctas=8)[0] > t
    with pytest.raises(fdtd.FDTDError):
        fdtd.route_us(d, ctas=0)


# grids of a batch, fluence, which of them take the two-step kernel in the graph (None: either, the times are close)
BATCHES = [
    ([(64, 64, 32, 8)], True, [2]), ([(64, 64, 3, 6)] * 8, True, [2] * 8), ([(332, 332, 3, 6)] * 2, True, [2] * 2),
    ([(32, 32, 1024, 6)] * 4, True, [2] * 4), ([(48, 40, 16, 6)] * 16, True, [2] * 16),
    ([(24, 24, 8, 4)] * 40, True, [2] * 40), ([(96, 96, 16, 16)] * 12, True, [1] * 12),
    ([(160, 160, 40, 8)] * 4, False, [1] * 4), ([(332, 332, 46, 6)] * 2, False, [1] * 2),
    ([(n, n, 64, 16) for n in (640, 320, 160, 96) for _ in range(2)], True, [1] * 8),
    ([(560, 560, 2, 6), (320, 320, 64, 16)], True, [2, 1]),
]


@pytest.mark.parametrize("boxes,fluence,routes", BATCHES)
def test_grids_of_a_batch(boxes, fluence, routes):
    """Both ways of each batch were measured (us per step; csrc/batch.cu)."""
    descs = [fdtd.make_grid_desc(*b, 0.05, 0.05, 0.05, fluence=fluence) for b in boxes]
    ctas, got = fdtd.batch_routes(descs)
    assert got.tolist() == routes
    assert all(8 <= c <= 152 for c in ctas)
    for b, c in zip(boxes, ctas):
        windows = -(-b[0] // 24) * -(-b[1] // 20)
        assert c == 152 or windows < 152      # grids of many windows have every SM
