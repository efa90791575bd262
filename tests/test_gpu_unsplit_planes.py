"""FP32 FEC / BEC steps on wide grids of few planes, on both sides of the rule that
gives them to one kernel or the other: bit for bit what a buffer one float off 16
bytes gets, which takes the other kernel, and against the oracle."""
import pytest
import torch

import test_gpu_unsplit32 as U
from gpu_helpers import assert_parity, oracle_step, random_case
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,shape", [("FEC", (5, 512, 512)), ("FEC", (3, 300, 300)), ("FEC", (20, 300, 220)),
                                          ("BEC", (8, 512, 512)), ("BEC", (1, 1024, 512)), ("BEC", (9, 300, 320)),
                                          ("BEC", (10, 300, 320))])
def test_both_kernels_give_the_same_bits_on_few_planes(scheme, shape):
    U.test_both_kernels_give_the_same_bits(scheme, shape)


@pytest.mark.parametrize("scheme", ["FEC", "BEC"])
@pytest.mark.parametrize("shape", [(1, 300, 300), (3, 300, 300), (9, 300, 304)])
def test_few_planes_match_the_oracle(scheme, shape):
    phi, vel, sp, dt = random_case(shape, seed=sum(shape), dtype="f32")
    out = sl.advect(phi.cuda(), vel.cuda(), dt, sp, scheme)
    torch.cuda.synchronize()
    assert sl.sl_device_status() == 0
    assert_parity(out.cpu().numpy(), oracle_step(phi, vel, sp, dt, scheme, 0), "f32", f"{scheme} {shape}")
