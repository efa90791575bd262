"""Split CEC steps with double arithmetic at the edges of their tiles: column
tiles of 32 x 16 (32 x 4 on small planes), 16-byte and element-wise staging,
shares of few planes, one to three cells along an axis."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_parity, oracle_step, random_case
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu
DEV = "cuda"
SHAPES = [(1, 1, 1), (2, 3, 5), (13, 16, 32), (7, 17, 33), (30, 15, 31), (5, 33, 66), (40, 48, 64),
          (4, 32), (5, 33), (3, 2), (64, 96), (17, 130), (600, 520)]


@pytest.mark.parametrize("dtype", ["f64", "f32_d64"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("parity", [0, 1])
def test_double_steps_match_the_oracle_at_tile_edges(shape, dtype, parity):
    phi, vel, sp, dt = random_case(shape, seed=sum(shape) + parity, dtype=dtype)
    vel.view(-1)[::7] = 0.0                       # C = 0, and exactly 1 and -1
    vel[0].view(-1)[::11] = sp[0] / dt
    vel[0].view(-1)[5::13] = -sp[0] / dt
    out = sl.advect(phi.to(DEV), vel.to(DEV), dt, sp, "CEC", parity, delta64=dtype == "f32_d64")
    torch.cuda.synchronize()
    sl.sl_device_status()                         # a rounded Courant number may pass 1 by one unit
    assert_parity(out.cpu().numpy(), oracle_step(phi, vel, sp, dt, "CEC", parity), dtype, f"{shape} {parity}")


def test_float_storage_keeps_denormals_and_infinities():
    """Float values widen exactly: denormal fields step as the oracle does, and
    an infinity stays in the cells its stencil reaches."""
    shape = (6, 9, 40)
    phi, vel, sp, dt = random_case(shape, seed=3, dtype="f32_d64")
    tiny = (phi * 1e-42).contiguous()
    out = sl.advect(tiny.to(DEV), vel.to(DEV), dt, sp, "CEC", 0, delta64=True).cpu().double().numpy()
    ref = oracle_step(tiny, vel, sp, dt, "CEC", 0)
    assert np.abs(out - ref).max() <= 3 * 2.0 ** -149          # three float roundings, half a unit each, at most
    phi[2, 4, 20] = float("inf")
    out = sl.advect(phi.to(DEV), vel.to(DEV), dt, sp, "CEC", 0, delta64=True).cpu()
    far = torch.ones(shape, dtype=torch.bool)
    far[:, 1:8, 17:24] = False
    assert torch.isfinite(out[far]).all() and not torch.isfinite(out[2, 4, 20])
