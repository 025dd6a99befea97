"""Default launches of boxes whose rows do not start on 16-byte boundaries, where two kernels are near
each other: the rule takes the one that was measured faster, on each side of its lines."""
import ctypes

import pytest
import torch

from paper_1803_01262_gb300 import cdi

pytestmark = pytest.mark.gpu
ROW, SCALAR = (7, 8), (1, 3)


@pytest.mark.parametrize("shape,tiles", [
    ((1, 129, 129), SCALAR), ((1, 513, 513), SCALAR), ((1, 2049, 2049), SCALAR), ((1, 1, 1000003), SCALAR),
    ((64, 64, 129), SCALAR), ((64, 64, 65), SCALAR), ((300, 7, 129), SCALAR), ((150, 32, 65), SCALAR),
    ((129, 129, 129), ROW), ((150, 129, 65), ROW), ((64, 42, 129), ROW), ((150, 28, 129), ROW)])
def test_fp64_euler(shape, tiles):
    g = cdi.Grid(*shape[::-1], 0.01, torch.float64)
    assert g.get_launch()["tile"] in tiles


@pytest.mark.parametrize("shape,tile", [((1, 2049, 2049), 7), ((255, 255, 255), 8), ((129, 129, 129), 7)])
def test_fp32_euler(shape, tile):
    assert cdi.Grid(*shape[::-1], 0.01, torch.float32).get_launch()["tile"] == tile


def stage_kernels(shape, dtype):
    """Names of the kernels that one RK2 step of a new grid launches."""
    cu = ctypes.CDLL("libcuda.so.1")
    g = cdi.Grid(*shape[::-1], 0.01, dtype)
    a = torch.rand(shape, device="cuda", dtype=dtype)
    b, c, d, u = (torch.empty_like(a) for _ in range(4))
    g.set_velocity(u.zero_(), u, u)
    prm = (1e-6, 0.01, 1.0)
    g.step_rk(a, b, c, d, *prm, scheme="rk2")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        g.step_rk(a, b, c, d, *prm, scheme="rk2")
    h, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(2)
    nodes = (ctypes.c_void_p * 2)()
    assert cu.cuGraphGetNodes(h, nodes, ctypes.byref(n)) == 0 and n.value == 2
    names = []
    for x in nodes:
        p = (ctypes.c_uint64 * 16)()        # CUDA_KERNEL_NODE_PARAMS_v2: func first, kern eighth
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(x), p) == 0
        s = ctypes.c_char_p()
        f = cu.cuFuncGetName if p[0] else cu.cuKernelGetName
        assert f(ctypes.byref(s), ctypes.c_void_p(p[0] or p[7])) == 0
        names.append(s.value.decode())
    return names


@pytest.mark.parametrize("dtype,shape,row", [
    (torch.float64, (1, 129, 129), True), (torch.float64, (1, 513, 513), True), (torch.float64, (1, 5, 1001), False),
    (torch.float64, (1, 1, 300001), False), (torch.float64, (64, 64, 129), False), (torch.float64, (300, 7, 129), False),
    (torch.float64, (150, 28, 129), True), (torch.float32, (1, 1, 300001), False),
    (torch.float32, (1, 1, 10001), True), (torch.float32, (9, 33, 67), True)])
def test_runge_kutta_stage(dtype, shape, row):
    for name in stage_kernels(shape, dtype):
        assert ("fwd_row_kernel" in name) == row, name


@pytest.mark.parametrize("dtype,shape,row", [
    (torch.float32, (1, 1, 1001), False), (torch.float32, (300, 2, 201), False), (torch.float32, (1, 4, 1000003), False),
    (torch.float32, (1, 5, 1000003), True), (torch.float32, (64, 64, 67), True), (torch.float64, (1, 1, 1001), False),
    (torch.float64, (64, 64, 16), False), (torch.float64, (64, 5, 129), False), (torch.float64, (1, 17, 17), False),
    (torch.float64, (16, 16, 16), True), (torch.float64, (1, 129, 129), True), (torch.float64, (64, 64, 33), True),
    (torch.float64, (150, 7, 129), True), (torch.float64, (129, 129, 129), True)])
def test_adjoint(dtype, shape, row):
    g = cdi.Grid(*shape[::-1], 0.01, dtype)
    t = g.get_launch(cdi.CDI_KERNEL_ADJOINT)["tile"]
    aligned = shape[2] % (4 if dtype == torch.float32 else 2) == 0
    assert t == ((3 if aligned else 4) if row else (1 if shape[2] >= 32 and shape[1] >= 16 else 2))
