"""FP32 CIR / FEC / BEC steps on x-y planes of more than 2^30 cells (their byte
offsets take 33 bits; planes of up to 2^31 - 1 cells are accepted): every cell is
written, and the rows around the periodic seam, where the cells beyond the 2^30th
meet the first ones, agree with the oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_parity
from oracle import oracle as O
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu
DEV = "cuda"
N = 32770            # rows of no 16-byte multiple; N * N = 2^30 + 131076


def band(t, r0, r1):
    """Rows [r0, r1) of the last but one axis, modulo its length, in float64 on the host."""
    rows = torch.arange(r0, r1, device=t.device) % t.shape[-2]
    return t.index_select(-2, rows).double().cpu().numpy()


def test_planes_beyond_2_to_the_30_cells():
    if torch.cuda.mem_get_info()[0] < 30 * 2 ** 30:
        pytest.skip("needs 30 GB of device memory")
    gen = torch.Generator(device=DEV).manual_seed(1)
    phi = torch.empty((1, N, N), device=DEV).uniform_(-1.0, 1.0, generator=gen)
    vel = torch.empty((3, 1, N, N), device=DEV).uniform_(-0.95, 0.95, generator=gen)
    out = torch.empty_like(phi)
    for scheme in ("CIR", "FEC", "BEC"):
        out.fill_(float("nan"))
        sl.advect(phi, vel, 1.0, [1.0, 1.0, 1.0], scheme, out=out)
        torch.cuda.synchronize()
        assert sl.sl_device_status() == 0
        assert bool(torch.isfinite(out).all())
        for r0, r1 in ((-12, 12), (N // 2 - 8, N // 2 + 8)):
            # a band is periodic in y for the oracle, which spoils three rows at its edges
            ref = O.step(band(phi, r0, r1), band(vel, r0, r1), O.SCHEMES[scheme], 0)
            got = band(out, r0, r1)
            assert_parity(got[:, 4:-4], np.asarray(ref)[:, 4:-4], "f32", f"{scheme} rows {r0}..{r1}")
