"""FP32 CIR / FEC / BEC steps in 3D on any size and alignment: the edges of the
32 x 16 column tiles and of the equal shares, against the oracle; and bit for
bit against the kernel that serves large grids of whole 16-byte chunks."""
import pytest
import torch

from gpu_helpers import assert_parity, oracle_step, random_case
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu
DEV = "cuda"
SHAPES = [(1, 1, 1), (2, 1, 3), (3, 16, 32), (5, 17, 33), (4, 15, 31), (9, 32, 64), (7, 49, 97), (300, 5, 7)]


@pytest.mark.parametrize("scheme", ["CIR", "FEC", "BEC"])
@pytest.mark.parametrize("shape", SHAPES)
def test_steps_match_the_oracle_at_tile_edges(shape, scheme):
    phi, vel, sp, dt = random_case(shape, seed=sum(shape), dtype="f32")
    vel.view(-1)[::7] = 0.0
    out = sl.advect(phi.to(DEV), vel.to(DEV), dt, sp, scheme)
    torch.cuda.synchronize()
    assert sl.sl_device_status() == 0
    assert_parity(out.cpu().numpy(), oracle_step(phi, vel, sp, dt, scheme, 0), "f32", f"{scheme} {shape}")


@pytest.mark.parametrize("scheme,shape", [("FEC", (96, 256, 256)), ("BEC", (160, 256, 256)), ("CIR", (152, 256, 256))])
def test_both_kernels_give_the_same_bits(scheme, shape):
    """A buffer one float off 16 bytes takes the other kernel."""
    phi, vel, sp, dt = random_case(shape, seed=5, dtype="f32")
    n = phi.numel()
    buf = torch.empty(n + 1, dtype=torch.float32, device=DEV)
    buf[1:] = phi.view(-1).to(DEV)
    vel, dims = vel.to(DEV), list(shape[::-1])
    out, ref = (torch.empty(n, dtype=torch.float32, device=DEV) for _ in range(2))
    sl.sl_advect(out, buf.data_ptr() + 4, vel, 3, dims, sp, dt, sl.SCHEMES[scheme], sl.F32)
    sl.sl_advect(ref, phi.to(DEV), vel, 3, dims, sp, dt, sl.SCHEMES[scheme], sl.F32)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
