"""The autotuner keeps the launch that an untuned step makes: the shape it files for
that launch gives the same grid of CTAs when it is read back, for every kernel
family, and on grids whose cached planes per item batch plans take over it is no
smaller than the least the tuner tries."""
import ctypes
import math

import pytest
import torch

from paper_1606_06117_gb300 import _lib as sl
from paper_1606_06117_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


class KernelNode(ctypes.Structure):
    """CUDA_KERNEL_NODE_PARAMS"""
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def launches(fn):
    """(grid, block) of the kernels that fn launches, from a captured graph."""
    fn()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    cu = ctypes.CDLL("libcuda.so.1")
    graph, n = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        p, kind = KernelNode(), ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            out.append((tuple(p.grid), tuple(p.block)))
    return out


def inputs(shape, dtype):
    t = torch.float64 if dtype == sl.F64 else torch.float32
    phi = W.random_modes(shape, W.draw_modes(len(shape), 8, 3, seed=1), device=DEV, dtype=t)
    vel = W.abc_velocity(shape, device=DEV, dtype=t)
    sp = [2 * math.pi / n for n in shape[::-1]]
    return phi, vel, sp, 0.4 * min(sp)


@pytest.fixture(autouse=True)
def empty_cache():
    sl.sl_tuning_clear()
    yield
    sl.sl_tuning_clear()


# shape, scheme, dtype, and the filed form of the untuned launch: kernel, tile_y, tile_z, CTAs per SM
DEFAULTS = [((192, 192, 192), "CEC", sl.F32, (1, 32, 0, 2)), ((131, 150, 187), "CEC", sl.F32, (2, 32, 32, 0)),
            ((24, 36, 40), "CEC", sl.F32, (2, 32, 24, 0)), ((60, 52, 44), "CEC", sl.F64, (2, 16, 0, 0)),
            ((100, 160, 160), "CIR", sl.F32, (3, 16, 0, 0)), ((150, 160, 160), "FEC", sl.F32, (4, 16, 0, 0)),
            ((400, 160, 160), "BEC", sl.F32, (4, 16, 0, 0)), ((40, 50, 61), "BEC", sl.F32, (4, 16, 0, 0)),
            ((40, 50, 60), "FEC", sl.F64, (4, 8, 0, 0))]


@pytest.mark.parametrize("shape,scheme,dtype,filed", DEFAULTS)
def test_the_filed_default_is_the_untuned_launch(tmp_path, shape, scheme, dtype, filed):
    if not hasattr(torch.cuda.CUDAGraph, "raw_cuda_graph"):
        pytest.skip("needs access to the captured graph")
    phi, vel, sp, dt = inputs(shape, dtype)
    out = torch.empty_like(phi)
    for parity in ((0, 1) if scheme == "CEC" else (0,)):
        def step():
            sl.advect(phi, vel, dt, sp, scheme, parity, out=out)
        untuned = launches(step)
        kernel, ty, tz, ctas = filed
        dims = " ".join(str(n) for n in shape[::-1])
        (tmp_path / "t.txt").write_text(f"{dims} {sl.SCHEMES[scheme]} {dtype} {kernel} 32 {ty} {tz} {ctas} 1\n")
        sl.sl_tuning_load(str(tmp_path / "t.txt"))
        assert launches(step) == untuned
        sl.sl_tuning_clear()


def test_planes_filed_for_batch_plans_are_no_fewer_than_those_tried():
    shape = (24, 36, 40)
    phi, vel, sp, dt = inputs(shape, sl.F32)
    t = sl.sl_autotune_scheme(torch.empty_like(phi), phi, vel, 3, list(shape[::-1]), sp, dt, sl.CEC, sl.F32)
    assert t.kernel == 2 and t.tile_z in (8, 16, 24)


@pytest.mark.parametrize("shape,dtype,tile_y", [((20, 40, 50), sl.F32_D64, 16), ((20, 40, 50), sl.F64, 16),
                                                ((128, 128), sl.F64, 4), ((128, 128), sl.F32_D64, 4),
                                                ((600, 520), sl.F64, 16)])
def test_double_cec_files_the_tile_height_it_runs(tmp_path, shape, dtype, tile_y):
    t = torch.float64 if dtype == sl.F64 else torch.float32
    dims = (list(shape[::-1]) + [1])[:3]
    phi = torch.rand(shape, device=DEV, dtype=t)
    vel = torch.rand((len(shape),) + shape, device=DEV, dtype=t)
    args = (phi, vel, len(shape), dims, [1.0] * 3, 0.5)
    got = sl.sl_autotune_scheme(torch.empty_like(phi), *args, sl.CEC, dtype)
    assert (got.kernel, got.tile_y) == (2, tile_y)
    sl.sl_tuning_save(str(tmp_path / "t.txt"))
    sl.sl_tuning_clear()
    sl.sl_tuning_load(str(tmp_path / "t.txt"))
    assert sl.sl_tuning_get(dims, sl.CEC, dtype).tile_y == tile_y
