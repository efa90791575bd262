"""FP32 CEC steps on grids that are no whole column tiles: the edges of the tiles
and of the copied rows, every alignment, one to four fields, shares of any
number of planes; and bit for bit the tensor-map path's result where both can
serve a grid."""
import pytest
import torch

from gpu_helpers import assert_parity, oracle_step, random_case
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu
DEV = "cuda"
SHAPES = [(8, 1, 1), (9, 3, 2), (8, 31, 33), (11, 33, 31), (10, 32, 36), (17, 65, 60), (40, 5, 7), (8, 2, 100), (300, 4, 4)]


@pytest.mark.parametrize("parity", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_steps_match_the_oracle_at_tile_edges(shape, parity):
    phi, vel, sp, dt = random_case(shape, seed=sum(shape) + parity, dtype="f32")
    vel.view(-1)[::7] = 0.0
    out = sl.advect(phi.to(DEV), vel.to(DEV), dt, sp, "CEC", parity)
    torch.cuda.synchronize()
    assert sl.sl_device_status() == 0
    assert_parity(out.cpu().numpy(), oracle_step(phi, vel, sp, dt, "CEC", parity), "f32", f"{shape} {parity}")


@pytest.mark.parametrize("parity", [0, 1])
def test_both_ways_of_staging_give_the_same_bits(parity):
    shape = (20, 64, 96)
    phi, vel, sp, dt = random_case(shape, seed=9, dtype="f32")
    n, vel, dims = phi.numel(), vel.to(DEV), [96, 64, 20]
    ref = sl.advect(phi.to(DEV), vel, dt, sp, "CEC", parity)
    buf = torch.empty(n + 1, dtype=torch.float32, device=DEV)
    buf[1:] = phi.view(-1).to(DEV)          # one float off 16 bytes: copied element by element
    out = torch.empty(n, dtype=torch.float32, device=DEV)
    sl.sl_advect(out, buf.data_ptr() + 4, vel, 3, dims, sp, dt, sl.CEC, sl.F32, parity)
    torch.cuda.synchronize()
    assert torch.equal(out.view(shape), ref)


@pytest.mark.parametrize("nx", [36, 37])
def test_shares_and_field_groups_keep_the_bits(tmp_path, nx):
    shape = (24, 41, nx)
    _, vel, sp, dt = random_case(shape, seed=4, dtype="f32")
    vel = vel.to(DEV)
    fields = [torch.randn(shape, device=DEV) for _ in range(6)]
    for parity in (0, 1):
        refs = [sl.advect(f, vel, dt, sp, "CEC", parity) for f in fields]
        for tz in (0, 1, 5, 24):
            if tz:
                p = tmp_path / "shape.txt"
                p.write_text(f"{nx} 41 24 {sl.CEC} {sl.F32} 2 32 32 {tz} 0 1\n")
                sl.sl_tuning_load(str(p))
            store, outs = torch.stack(fields), torch.empty((6,) + shape, device=DEV)
            sl.sl_advect_multi(list(outs), list(store), vel, 3, [nx, 41, 24], sp, dt, sl.CEC, sl.F32, parity)
            torch.cuda.synchronize()
            sl.sl_tuning_clear()
            for o, r in zip(outs, refs):
                assert torch.equal(o, r), (tz, parity)
    assert sl.sl_device_status() == 0


# (nz, ny, nx): no tile row, one and three tile rows away from the periodic seam in y, at either seam in x
# and between them; one field and groups of fields
@pytest.mark.parametrize("fields", [1, 3])
@pytest.mark.parametrize("shape", [(8, 32, 64), (9, 64, 96), (12, 96, 64), (10, 160, 128)])
def test_boxes_of_inner_and_seam_tiles_give_the_bits_of_the_copies(shape, fields):
    nz, ny, nx = shape
    phi, vel, sp, dt = random_case(shape, seed=sum(shape), dtype="f32")
    n, vel, dims = phi.numel(), vel.to(DEV), [nx, ny, nz]
    store = torch.randn((fields,) + shape, device=DEV)
    store[0] = phi.to(DEV)
    for parity in (0, 1):
        outs = torch.empty((fields,) + shape, device=DEV)
        sl.sl_advect_multi(list(outs), list(store), vel, 3, dims, sp, dt, sl.CEC, sl.F32, parity)
        for f in range(fields):
            buf = torch.empty(n + 1, dtype=torch.float32, device=DEV)
            buf[1:] = store[f].view(-1)     # one float off 16 bytes: copied element by element
            ref = torch.empty(n, dtype=torch.float32, device=DEV)
            sl.sl_advect(ref, buf.data_ptr() + 4, vel, 3, dims, sp, dt, sl.CEC, sl.F32, parity)
            torch.cuda.synchronize()
            assert torch.equal(outs[f].view(-1), ref), (parity, f)
    assert sl.sl_device_status() == 0
