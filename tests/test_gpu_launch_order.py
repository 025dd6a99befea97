"""The face velocities of a call may have been written by the caller's kernel directly before it.
Every launch may start while the one before it ends, so the first of a call waits for the caller's
work before it reads them, and only the later ones, behind a launch of the library's own, read them
at once: the kernels' argument ``chained``, read here from the captured graph."""
import ctypes

import pytest
import torch

from paper_1803_01262_gb300 import cdi

pytestmark = pytest.mark.gpu


class KernelNodeParams(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 6), ("smem", ctypes.c_uint),
                ("params", ctypes.POINTER(ctypes.c_void_p)), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def chained_flags(call):
    """The third argument (chained) of the kernels that ``call`` captures, after the first kernel,
    which is the caller's own."""
    cu = ctypes.CDLL("libcuda.so.1")
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        call()
    n = ctypes.c_size_t(0)
    h = ctypes.c_void_p(g.raw_cuda_graph())
    assert cu.cuGraphGetEdges_v2(h, None, None, None, ctypes.byref(n)) == 0
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (ctypes.c_uint64 * n.value)()
    assert cu.cuGraphGetEdges_v2(h, src, dst, data, ctypes.byref(n)) == 0
    nxt = dict(zip(src, dst))
    at = next(iter(set(src) - set(dst)))
    flags = []
    while at in nxt:
        at = nxt[at]
        p = KernelNodeParams()
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(at), ctypes.byref(p)) == 0
        flags.append(ctypes.cast(p.params[2], ctypes.POINTER(ctypes.c_int))[0])
    assert len(flags) == n.value   # one chain
    return flags


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nx", [64, 66, 67])
@pytest.mark.parametrize("kind", ["step", "planes", "run", "path", "rk4", "run_rk", "adjoint", "adjoint_path"])
def test_first_launch_waits_for_the_caller(kind, nx, dtype):
    shape = (20, 24, nx)
    g = cdi.Grid(nx, 24, 20, 1.0 / 64, dtype)
    a, u = torch.rand(shape, device="cuda", dtype=dtype), torch.rand(shape, device="cuda", dtype=dtype)
    b, c, d = (torch.empty_like(a) for _ in range(3))
    g.set_velocity(u, u, u)
    prm = (1e-3, 1.0 / 64, 1.0)
    calls = {
        "step": lambda: g.step(a, b, *prm),
        "planes": lambda: g.step_planes(a, b, 3, 11, *prm),
        "run": lambda: g.run(a, b, 3, *prm),
        "path": lambda: g.step_path([a, b, c], *prm, [1.0, 0.5]),
        "rk4": lambda: g.step_rk(a, b, c, d, *prm),
        "run_rk": lambda: g.run_rk(a, b, c, d, 2, *prm, scheme="rk2"),
        "adjoint": lambda: g.step_adjoint(a, b, c, *prm),
        "adjoint_path": lambda: g.adjoint_path([a, a], b, c, *prm, [1.0, 0.5]),
    }
    calls[kind]()   # sets up the launch configurations
    torch.cuda.synchronize()
    flags = chained_flags(lambda: (u.mul_(0.5), calls[kind]()))
    assert flags == [0] + [1] * (len(flags) - 1)   # the later launches still overlap


@pytest.mark.parametrize("nx", [64, 67])
def test_new_velocities_reach_every_call(nx):
    """Velocities overwritten by a kernel directly before a call give what they give after a wait."""
    shape = (40, 60, nx)
    g = cdi.Grid(nx, 60, 40, 1.0 / 64, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(nx)
    a, u, new = (torch.rand(shape, generator=gen, device="cuda") for _ in range(3))
    c, d = torch.empty_like(a), torch.empty_like(a)
    prm = (1e-3, 1.0 / 64, 1.0)
    for f in (lambda o: g.step(a, o, *prm), lambda o: g.step_rk(a, o, c, d, *prm),
              lambda o: g.step_adjoint(a, new, o, *prm)):
        out, ref = torch.empty_like(a), torch.empty_like(a)
        g.set_velocity(u, u, u)
        u.copy_(new)
        f(out)
        torch.cuda.synchronize()
        f(ref)
        assert torch.equal(out, ref)
        u.mul_(0.25)
