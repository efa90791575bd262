"""Unsplit steps in 3D on grids of one to nine planes, whose CTAs take the planes of a
tile from the first one on below eight planes and from a tile-dependent one from
eight on: many tiles, in every type, against the oracle."""
import pytest
import torch

from gpu_helpers import assert_parity, oracle_step, random_case
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64", "f32_d64"])
@pytest.mark.parametrize("scheme", ["CIR", "FEC", "BEC"])
@pytest.mark.parametrize("nz", [1, 2, 7, 8, 9])
def test_thin_grids_match_the_oracle(nz, scheme, dtype):
    shape = (nz, 130, 516)
    phi, vel, sp, dt = random_case(shape, seed=nz, dtype=dtype)
    out = sl.advect(phi.cuda(), vel.cuda(), dt, sp, scheme, delta64=dtype == "f32_d64")
    torch.cuda.synchronize()
    assert sl.sl_device_status() == 0
    assert_parity(out.cpu().numpy(), oracle_step(phi, vel, sp, dt, scheme, 0), dtype, f"{scheme} {nz}")
