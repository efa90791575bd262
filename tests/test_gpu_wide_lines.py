"""The fused large-CFL sweep at the edges of its line lengths (threads and column
blocks change at 32, 64, 128, 256, 512, 1024, 2048 and 4096 cells), partial
column blocks and rows, and Courant numbers of many periods, against the
oracle's CEC_SL."""
import pytest
import torch

from gpu_helpers import assert_parity
from paper_1606_06117_gb300 import _lib as sl
from test_gpu_wide import case, oracle_of

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1, 1), (2, 3, 1), (32, 5, 7), (33, 2, 40), (64, 65, 9), (128, 3, 17), (129, 4, 70), (256, 2, 8),
          (257, 2, 9), (512, 1, 10), (513, 3, 3), (1, 1024, 6), (1, 1025, 5), (1, 2048, 3), (1, 2049, 2), (1, 4096, 3),
          (2, 1, 4096), (1, 3, 2049), (70, 41, 187)]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("cmax", [3.5, 700.0])
@pytest.mark.parametrize("shape", SHAPES)
def test_lines_of_every_length_match_the_oracle(shape, cmax, dtype):
    phi, vel, sp, dt, courant = case(shape, cmax, sum(shape), dtype)
    for parity in (0, 1):
        out = sl.advect_wide(phi, vel, dt, sp, "CEC", parity)
        torch.cuda.synchronize()
        assert sl.sl_device_status() == 0
        assert_parity(out.cpu().numpy(), oracle_of(phi, courant, "CEC", parity), dtype, f"{shape} {cmax} {parity}")


def test_a_number_that_cannot_be_used_keeps_the_cell_among_far_departures():
    phi, vel, sp, dt, courant = case((6, 9, 50), 90.0, 1, "f32")
    vel[0, 2, 3, 4] = float("inf")
    vel[1, 2, 3, 4] = float("nan")
    courant[0, 2, 3, 4] = courant[1, 2, 3, 4] = 0.0
    out = sl.advect_wide(phi, vel, dt, sp, "CEC", 0)
    torch.cuda.synchronize()
    assert sl.sl_device_status() == sl.DEV_CFL
    assert_parity(out.cpu().numpy(), oracle_of(phi, courant, "CEC", 0), "f32")
