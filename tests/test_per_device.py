"""What the two-step kernel sets up once per process it sets up once per device:
a kernel's opt-in to more shared memory holds on the device it was made on."""
import pytest

from paper_2102_12978_gb300 import fdtd


@pytest.mark.parametrize("devices,results,values", [
    ([0, 0, 0], [2, 5, 5], [2, 2, 2]),                    # one device: set up once
    ([0, 1, 0, 1, 7], [1, 2, 9, 9, 3], [1, 2, 1, 2, 3]),  # every device has its own
    ([3, 3, 3], [0, 4, 9], [-1, 4, 4]),                   # a set-up that failed runs again
    ([63, 64, 64, -1], [1, 2, 3, 4], [1, 2, 3, 4]),       # past the table: set up on each call
])
def test_each_device_is_set_up(devices, results, values):
    assert fdtd.per_device(devices, results).tolist() == values
