"""Every form of the Rayleigh-Benard step against the oracle: rows projected in
pairs or singly, operands staged in shared memory or not, the x solve by one
matrix per z mode or by two transforms, launches that overlap or not.

The oracle's dense pseudo-inverse is too large for these boxes; the same
zero-mean Neumann problem is solved here with a sparse factorisation of the
operator bordered by the zero-mean condition.  Bounds as in test_gpu_rb.py."""
import numpy as np
import pytest
import torch

import test_gpu_rb as T
from gpu_helpers import assert_parity
from oracle import oracle as O
from oracle import rb_oracle as R
from paper_1606_06117_gb300 import _lib as sl

pytestmark = pytest.mark.gpu
sparse = pytest.importorskip("scipy.sparse")
linalg = pytest.importorskip("scipy.sparse.linalg")


def second_difference(n, h):
    d = -2.0 * np.ones(n)
    d[0] = d[-1] = -1.0   # no flux through the walls
    return sparse.diags([np.ones(n - 1), d, np.ones(n - 1)], [-1, 0, 1]) / h ** 2


class Box(R.Box):
    def __init__(self, nx, nz, Ra, scheme):
        self.nx, self.nz, self.dx, self.dz = nx, nz, 2.0 / nx, 1.0 / nz
        self.Ra, self.Pr, self.scheme, self.n = Ra, 1.0, O.SCHEMES[scheme], 0
        A = sparse.kron(sparse.identity(nz), second_difference(nx, self.dx)) + \
            sparse.kron(second_difference(nz, self.dz), sparse.identity(nx))
        one = sparse.csr_matrix(np.ones((nx * nz, 1)))
        self.lu = linalg.splu(sparse.bmat([[A, one], [one.T, None]]).tocsc())

    def solve(self, rhs):
        return self.lu.solve(np.append(rhs.ravel(), 0.0))[:-1].reshape(rhs.shape)


FORMS = [
    (6, 155, "f64"), (6, 156, "f64"),         # pairs, staged; an odd and an even number of rows
    (100, 155, "f64"), (100, 156, "f64"),     # pairs, one matrix per mode from global memory
    (480, 160, "f64"),                        # pairs, two transforms
    (20, 100, "f64"), (120, 100, "f64"),      # single rows without overlap, staged and not
    (768, 64, "f64"),                         # single rows, two transforms, overlap
    (112, 60, "f64"),                         # single rows, one matrix per mode from global memory, overlap
    (100, 155, "f32"), (100, 156, "f32"),     # FP32: pairs, two transforms
]


@pytest.mark.parametrize("nx,nz,dtype", FORMS)
def test_a_form_matches_the_oracle(nx, nz, dtype):
    steps, dt, Ra = 2, 1e-6, 1e4
    t = torch.float64 if dtype == "f64" else torch.float32
    start = [np.asarray(torch.from_numpy(a).to(t).double()) for a in T.random_start(nx, nz, seed=nz, cmax=0.2, dt=dt)]
    box = Box(nx, nz, Ra, "CEC")
    box.u, box.w, box.theta = start
    g = sl.RayleighBenard(nx, nz, Ra=Ra, scheme="CEC", dtype=t)
    try:
        sl.sl_device_status()
        g.set_state(*(torch.from_numpy(np.ascontiguousarray(a)) for a in start))
        for _ in range(steps):
            box.step(dt)
        g.step(dt, steps)
        got = [a.cpu().double().numpy() for a in g.state()]
        assert sl.sl_device_status() == 0
    finally:
        g.close()
    for name, a, b in zip(("u", "w", "theta"), got, (box.u, box.w, box.theta)):
        assert_parity(a, b, dtype, f"{nx}x{nz} {name}", T.allowance(nx, nz, steps, f64=dtype == "f64"))


@pytest.mark.parametrize("nx,nz", [(1024, 32), (2800, 4), (48, 2048)])
def test_creating_a_box_costs_no_more_than_a_few_hundred_steps(nx, nz):
    """The tables of a box are a few passes over nx^2 nz (where it keeps them) and nz^2
    elements, below 0.3 GB: a millisecond or two on the device, no host loops over
    them (134 and 402 ms for the first two with host tables and a sum per element).  The
    bound is several times that, for the allocation and a busy host."""
    import time
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        h = sl.sl_rb_create(nx, nz, scheme="CEC", dtype=sl.F64)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
        sl.sl_rb_destroy(h)
    assert best < 0.02, best
