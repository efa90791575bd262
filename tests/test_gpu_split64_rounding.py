"""Rounding of the SL_F64 split CEC step on smooth fields: no further from the
exact step than the 1D scheme in its usual form (L_U[Phi] from the upwind
neighbour, delta = (Phi - L) - U (L_up - L)) evaluated in doubles with one
rounding per multiply-add."""
import numpy as np
import pytest
import torch

from paper_1606_06117_gb300 import _lib as sl
from paper_1606_06117_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"
LD = np.longdouble


def shifted(a, s, axis):
    """a at j - s_j along axis, s in {-1, 0, 1}, periodic."""
    return np.where(s > 0, np.roll(a, 1, axis), np.where(s < 0, np.roll(a, -1, axis), a))


def fma(a, b, c):
    return (a.astype(LD) * b.astype(LD) + c.astype(LD)).astype(np.float64)


def sweep_doubles(f, c, axis):
    s, U = np.sign(c).astype(int), np.abs(c)
    nb = shifted(f, s, axis)
    L = fma(1.0 - U, f - nb, nb)
    d = fma(-U, shifted(L, -s, axis) - L, f - L)
    w = fma(U, np.full_like(U, 1.0 / 6.0), np.full_like(U, 1.0 / 6.0))
    return fma(w, shifted(d, s, axis) - d, fma(np.full_like(d, 0.5), d, L))


def sweep_exact(f, c, axis):
    s, U = np.sign(c).astype(int), np.abs(c).astype(LD)
    L = f - U * (f - shifted(f, s, axis))
    d = (f - L) - U * (shifted(L, -s, axis) - L)
    return L + d / 2 + (1 + U) / 6 * (shifted(d, s, axis) - d)


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 2e-19, reason="needs a long double wider than a double")
@pytest.mark.parametrize("flow", ["rotation", "shear"])
@pytest.mark.parametrize("parity", [0, 1])
def test_a_double_step_rounds_no_worse_than_the_usual_form(flow, parity):
    shape = (128, 160)
    make = {"rotation": W.rotation_velocity, "shear": W.shear_patch_velocity}[flow]
    vel = make(shape, device="cpu", dtype=torch.float64)
    sp = [1.0 / n for n in shape[::-1]]
    dt = 0.8 / max(float(vel[d].abs().max()) / sp[d] for d in range(2))
    C = [(vel[d] * (dt / sp[d])).numpy() for d in range(2)]
    got, usual = [], []
    for seed in range(4):
        phi = W.random_modes(shape, W.draw_modes(2, 32, 8, seed=seed), length=1.0, dtype=torch.float64)
        out = sl.advect(phi.to(DEV), vel.to(DEV), dt, sp, "CEC", parity).cpu().numpy()
        f, x = phi.numpy(), phi.numpy().astype(LD)
        for axis in ((0, 1) if parity else (1, 0)):
            c = C[1 - axis]
            f, x = sweep_doubles(f, c, axis), sweep_exact(x, c, axis)
        scale = np.sqrt((x * x).sum())
        got.append(float(np.sqrt(((out - x) ** 2).sum()) / scale))
        usual.append(float(np.sqrt(((f - x) ** 2).sum()) / scale))
    # 4 x 20480 cells: the mean of either error is known to about 0.3 %
    assert np.mean(got) <= 1.01 * np.mean(usual), (got, usual)
