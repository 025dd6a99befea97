"""Runs of 2D grids held in shared memory (bands of rows, one per block, halo words between them):
the same buffers, extrema and counts as one launch per step on the one-cell-per-thread tile, bit
for bit (the sums to rounding), for one band (no neighbour), bands of two rows and of uneven
heights, odd rows, every buffer parity, runs of several launches and time-dependent velocities."""
import ctypes
import os
import subprocess
import sys
import time

import pytest
import torch

from paper_1803_01262_gb300 import cdi

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def setup(ny, nx, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.rand((1, ny, nx), generator=gen, device="cuda", dtype=dtype)
    phi, u, v = 1.1 * r() - 0.05, r() - 0.5, r() - 0.5     # values outside [0, 1]: the counts take part
    h = 1.0 / max(ny, nx, 2)
    g = cdi.Grid(nx, ny, 1, h, dtype)
    g.set_velocity(u, v, torch.zeros_like(u))
    return g, phi, (0.1 * h, h, 1.0)


def ran(g, phi, n, prm, tile):
    g.set_launch(cdi.CDI_KERNEL_FORWARD, tile, 0, 0)
    g.reset_run_stats()
    a, b = phi.clone(), torch.full_like(phi, 3.0)
    out = g.run(a, b, n, *prm, period=0.7, t0=0.05)
    return out.clone(), (b if out is a else a).clone(), g.stats()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("ny,nx", [(1, 1), (1, 37), (3, 5), (4, 300), (5, 301), (37, 1), (33, 129), (128, 128),
                                   (157, 260), (200, 63)])
def test_run_equals_one_launch_per_step(dtype, ny, nx):
    g, phi, prm = setup(ny, nx, dtype, 10 + nx)
    rel = 1e-12 if dtype == torch.float64 else 1e-6   # order of the sums alone
    for n in (2, 3, 4, 7):
        (o0, p0, s0), (o1, p1, s1) = ran(g, phi, n, prm, 0), ran(g, phi, n, prm, -1)
        assert torch.equal(o0, o1) and torch.equal(p0, p1), n
        for k in s0:
            if k in ("mass", "sum"):
                assert abs(s0[k] - s1[k]) <= rel * max(1.0, abs(s0[k])), (n, k)
            else:
                assert s0[k] == s1[k], (n, k)


@pytest.mark.parametrize("n", [513, 1030])
def test_runs_of_several_launches(n):
    g, phi, prm = setup(20, 70, torch.float32, 5)
    phi.clamp_(0, 1)
    (o0, p0, s0), (o1, p1, s1) = ran(g, phi, n, prm, 0), ran(g, phi, n, prm, -1)
    assert torch.equal(o0, o1) and torch.equal(p0, p1)
    assert all(s0[k] == s1[k] for k in s0 if k not in ("mass", "sum"))


def test_two_grids_on_two_streams_and_a_captured_run():
    """Halo words and tags belong to a grid: runs of two grids may overlap, and a captured run may
    be replayed (the tags move on from one replay to the next)."""
    ga, pa, prm = setup(64, 64, torch.float32, 1)
    gb, pb, prm_b = setup(96, 50, torch.float32, 2)
    pa.clamp_(0, 1), pb.clamp_(0, 1)
    ref_a, ref_b = ran(ga, pa, 30, prm, 0)[0], ran(gb, pb, 30, prm_b, 0)[0]
    ga.set_launch(cdi.CDI_KERNEL_FORWARD)
    gb.set_launch(cdi.CDI_KERNEL_FORWARD)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    a, a2, b, b2 = pa.clone(), torch.empty_like(pa), pb.clone(), torch.empty_like(pb)
    torch.cuda.synchronize()
    for _ in range(5):
        a.copy_(pa), b.copy_(pb)
        torch.cuda.synchronize()
        ga.run(a, a2, 30, *prm, period=0.7, t0=0.05, stream=s1)
        gb.run(b, b2, 30, *prm_b, period=0.7, t0=0.05, stream=s2)
        torch.cuda.synchronize()
        assert torch.equal(a, ref_a) and torch.equal(b, ref_b)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ga.run(a, a2, 30, *prm, period=0.7, t0=0.05)
    for _ in range(3):
        a.copy_(pa)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, ref_a)
    ga.stats(), gb.stats()      # would raise if a bounded wait had given up


def boxes(dtype, sizes, seed):
    out = []
    for i, (ny, nx) in enumerate(sizes):
        gen = torch.Generator(device="cuda").manual_seed(seed + i)
        r = lambda: torch.rand((1, ny, nx), generator=gen, device="cuda", dtype=dtype)
        h = 1.0 / max(ny, nx, 2)
        phi, u, v = 1.1 * r() - 0.05, r() - 0.5, r() - 0.5
        out.append(dict(dx=h, dt=0.1 * h, eps=h, gamma=1.0, u=u, v=v, w=torch.zeros_like(u), phi_a=phi,
                        phi_b=torch.full_like(phi, 3.0)))
    return out


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("sharpen", ["centre", "face"])
@pytest.mark.parametrize("nbox", [4, 5, 700])
def test_batch_run_equals_other_tiles(dtype, sharpen, nbox):
    """Batch tile 4's run (boxes held in shared memory; with more boxes than slots, in units of a
    few steps handed from block to block): both buffers, extrema and counts of tile 0's run bit
    for bit, for runs of 1..16 steps in sequence and a run after single steps."""
    sizes = [(7, 9), (33, 40), (1, 37), (3, 2), (16, 64)] if nbox == 5 else [(5 + i % 7, 4 + i % 11) for i in range(nbox)]
    b0 = boxes(dtype, sizes, 3)
    b4 = [dict(x, phi_a=x["phi_a"].clone(), phi_b=x["phi_b"].clone()) for x in b0]
    bt = [cdi.Batch(x) for x in (b0, b4)]
    for b, tile in zip(bt, (0, 4)):
        b.set_sharpening(sharpen)
        b.set_launch(tile, 0)
    for n in (2, 5, 1, 16, 3):
        for b in bt:
            b.step(1.0)
            b.run(n)
        for x, y in zip(b0, b4):
            assert torch.equal(x["phi_a"], y["phi_a"]) and torch.equal(x["phi_b"], y["phi_b"]), n
    rel = 1e-12 if dtype == torch.float64 else 1e-6
    for p, q in zip(bt[0].stats(), bt[1].stats()):
        for k in p:
            if k in ("mass", "sum"):
                assert abs(p[k] - q[k]) <= rel * max(1.0, abs(p[k])), k
            else:
                assert p[k] == q[k], k


def test_batch_autotune_leaves_state_and_records():
    """The autotuner's trial runs on chip read the current state and restore the records."""
    bx = boxes(torch.float64, [(20, 30), (50, 50), (12, 9)], 9)
    bt = cdi.Batch(bx)
    bt.step(1.0)
    ref, st = [bt.current(i).clone() for i in range(3)], bt.stats()
    bt.autotune(reps=2)
    assert all(torch.equal(bt.current(i), r) for i, r in enumerate(ref)) and bt.stats() == st


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nbox", [90, 700])
def test_units_wait_bounded_and_are_claimed_in_order(dtype, nbox):
    """A unit after its box's first waits for the one before it, which must have been claimed earlier:
    with the first units withheld every block's claim is a waiting one, no box is stepped, the wait
    runs out and is reported, and the next run is that of an untouched twin."""
    b0 = boxes(dtype, [(5 + i % 7, 4 + i % 11) for i in range(nbox)], 21)
    twin = [dict(x, phi_a=x["phi_a"].clone(), phi_b=x["phi_b"].clone()) for x in b0]
    bt = [cdi.Batch(x) for x in (b0, twin)]
    for b in bt:
        b.set_launch(4, 0)
        b.run(4)
    ref = [bt[0].current(i).clone() for i in range(nbox)]
    with pytest.raises(cdi.CDIError) as e:
        bt[0].probe_box_wait(0.02)
    assert e.value.code == cdi.CDI_ERR_TIMEOUT
    assert all(torch.equal(bt[0].current(i), ref[i]) for i in range(nbox))
    for b in bt:
        b.run(5)
    assert all(torch.equal(bt[0].current(i), bt[1].current(i)) for i in range(nbox))
    assert bt[0].stats() == bt[1].stats()


def test_run_beside_another_streams_kernels():
    """A chunked run whose blocks start late, because another stream's kernels hold the SMs."""
    b0 = boxes(torch.float32, [(20, 30)] * 700, 5)
    twin = [dict(x, phi_a=x["phi_a"].clone(), phi_b=x["phi_b"].clone()) for x in b0]
    bt = [cdi.Batch(x) for x in (b0, twin)]
    for b in bt:
        b.set_launch(4, 0)
    bt[1].run(64)
    m = torch.rand(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(8):
            m = (m @ m).clamp_(0, 1)
    bt[0].run(64)
    torch.cuda.synchronize()
    assert all(torch.equal(bt[0].current(i), bt[1].current(i)) for i in range(700))
    assert bt[0].stats() == bt[1].stats()


def test_violation_counts_of_a_long_run():
    """More than 2^32 violations of one box in one run: every cell of 118^2 is one in each of 310000
    steps (dt = 0 keeps the field)."""
    n, steps = 118, 310000
    z = torch.zeros((1, n, n), device="cuda")
    b = cdi.Batch([dict(dx=1.0, dt=0.0, eps=1.0, gamma=1.0, u=z, v=z, w=z, phi_a=torch.full_like(z, 2.0),
                        phi_b=torch.empty_like(z)) for _ in range(90)])
    b.set_launch(4, 0)
    b.run(steps)
    for s in b.stats():
        assert s["n_strict_run"] == s["n_tol_run"] == n * n * steps and s["steps_run"] == steps
        assert s["n_strict"] == s["n_tol"] == n * n and s["min_run"] == s["max_run"] == 2.0
    assert b.info()["parity"] == 0 and all(torch.equal(b.current(i), z + 2) for i in range(90))


def test_autotune_takes_the_run_on_chip_in_a_new_process():
    """256 boxes of 50^2 in FP32: a run on chip takes a third of any other tile's time, also where the
    autotuner's first trial of it loads its kernel."""
    code = """
import torch
from paper_1803_01262_gb300 import cdi
z = torch.rand((1, 50, 50), device="cuda")
b = cdi.Batch([dict(dx=0.02, dt=1e-4, eps=0.02, gamma=1.0, u=z, v=z, w=z, phi_a=z.clone(), phi_b=z.clone())
               for _ in range(256)])
b.autotune(reps=2)
print(b.get_launch()["tile"])
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=240, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split()[-1] == "4"


@pytest.mark.parametrize("dtype,nbox,n", [(torch.float32, 1000, 16), (torch.float64, 256, 16)])
def test_short_runs_of_many_boxes(dtype, nbox, n):
    """A run of eight steps takes no longer than eight single steps, also with more boxes than slots."""
    z = torch.rand((1, n, n), device="cuda", dtype=dtype)
    b = cdi.Batch([dict(dx=0.02, dt=1e-6, eps=0.02, gamma=1.0, u=z, v=z, w=z, phi_a=z.clone(), phi_b=z.clone())
                   for _ in range(nbox)])
    b.set_launch(4, 0)

    def timed(f):
        f()
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            f()
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    assert timed(lambda: b.run(8)) <= timed(lambda: [b.step(1.0) for _ in range(8)])


def nodes(call):
    """Number of nodes that ``call`` captures."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        call()
    n = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [64, 128, 300])
def test_autotune_times_the_run_on_chip(dtype, n):
    """The autotuner's choice for a run is the fastest it timed: one launch for all steps, at depth 1,
    its time per step that of the run."""
    g, phi, prm = setup(n, n, dtype, 3)
    phi.clamp_(0, 1)
    a, b = phi.clone(), torch.empty_like(phi)
    ms = g.autotune(a, b, *prm, reps=3)
    assert g.get_run_depth()["depth"] == 1
    assert nodes(lambda: g.run(a, b, 32, *prm)) == 1
    best = float("inf")
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        g.run(a, b, 33, *prm)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) / 33)
    assert 0.5 * best <= ms <= 1.5 * best


def test_setting_the_sharpening_restores_the_default_run():
    g, phi, prm = setup(64, 64, torch.float32, 4)
    a, b = phi.clone(), torch.empty_like(phi)
    run = lambda: g.run(a, b, 8, *prm)
    assert nodes(run) == 1
    g.set_launch(cdi.CDI_KERNEL_FORWARD, 0)
    assert nodes(run) == 8
    g.set_sharpening("face")
    assert nodes(run) == 8
    g.set_sharpening("centre")
    assert nodes(run) == 1


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_halo_wait_is_bounded_and_the_grid_stays_usable(dtype):
    """A wait for a halo that nobody writes ends at its limit and is reported; the next run waits for
    its own halos and equals tile 0's."""
    g, phi, prm = setup(96, 70, dtype, 6)
    ref = ran(g, phi, 12, prm, 0)
    ran(g, phi, 5, prm, -1)
    t0 = time.perf_counter()
    with pytest.raises(cdi.CDIError) as e:
        g.probe_bounded_wait(0.05)
    assert e.value.code == cdi.CDI_ERR_TIMEOUT and 0.1 <= time.perf_counter() - t0 < 5.0   # both waits
    out = ran(g, phi, 12, prm, -1)
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
    assert all(out[2][k] == ref[2][k] for k in ref[2] if k not in ("mass", "sum"))


@pytest.mark.parametrize("dtype,ny,nx,n,on_chip", [
    (torch.float32, 128, 128, 3, True), (torch.float32, 128, 128, 2, False), (torch.float32, 1024, 1024, 8, True),
    (torch.float32, 4, 3000, 32, False), (torch.float32, 2, 6000, 32, False), (torch.float32, 1, 13000, 32, False),
    (torch.float32, 1, 2000, 32, True), (torch.float64, 128, 128, 2, True), (torch.float64, 512, 512, 4, True),
    (torch.float64, 2, 3000, 32, False), (torch.float64, 64, 1000, 32, False), (torch.float64, 1, 5000, 32, False),
    (torch.float64, 301, 301, 8, True)])
def test_runs_are_held_on_chip_where_that_is_faster(dtype, ny, nx, n, on_chip):
    """Long rows give a block too many cells, short runs do not repay the launch and the first load."""
    g, phi, prm = setup(ny, nx, dtype, 8)
    a, b = phi.clone(), torch.empty_like(phi)
    assert nodes(lambda: g.run(a, b, n, *prm)) == (1 if on_chip else n)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("ny,nx", [(4, 300), (5, 301), (33, 700), (3, 1500)])
def test_long_rows_on_chip_by_the_autotuner_or_launched(dtype, ny, nx):
    """Where the autotuner decides, and whichever way, a run equals one launch per step."""
    g, phi, prm = setup(ny, nx, dtype, 12 + nx)
    ref = ran(g, phi, 40, prm, 0)
    a, b = phi.clone(), torch.empty_like(phi)
    g.autotune(a, b, *prm, reps=2)
    g.reset_run_stats()
    a.copy_(phi)
    out = g.run(a, b, 40, *prm, period=0.7, t0=0.05)
    st = g.stats()
    assert torch.equal(out, ref[0]) and all(st[k] == ref[2][k] for k in st if k not in ("mass", "sum"))
