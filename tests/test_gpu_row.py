"""The row kernel (forward tiles 4, 5, 7, 8; any row length) at the edges of its tiles: rows of one
vector, of a partial vector, one cell past or short of the tile's 16 vectors, tile heights of 14
and 6 rows with one row more or less, and unit depths around its four ring slots.  Reference: the
one-cell-per-thread tile 0, which computes the same expressions in the same order, so the fields
must be equal bit for bit (and the extrema and counts equal); NaN and infinity in phi reach the
same cells."""
import numpy as np
import pytest
import torch

import oracle
from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def grid(shape, dtype, seed):
    nz, ny, nx = shape
    h = 1.0 / max(shape)
    phi = torch.from_numpy(I.random_phi(shape, seed, smooth=True)).to("cuda", dtype)
    vel = [torch.from_numpy(x).to("cuda", dtype) for x in I.random_velocity(shape, h, 8, 3, seed + 1)]
    g = cdi.Grid(nx, ny, nz, h, dtype)
    g.set_velocity(*vel)
    eps, gamma = 1.1 * h, 1.0
    return g, phi, (0.1 * h * h / (gamma * eps), eps, gamma)


def stepped(g, phi, tile, split, prm, n=3):
    g.set_launch(cdi.CDI_KERNEL_FORWARD, tile, 0, split)
    a, b = phi.clone(), torch.empty_like(phi)
    out = g.run(a, b, n, *prm).clone()
    st = g.stats()
    return out, [st[k] for k in ("min", "max", "n_strict", "n_tol")], st["sum"]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", [(1, 1, 5), (2, 3, 1), (3, 13, 16), (4, 14, 17), (5, 15, 62), (6, 28, 63), (7, 29, 64),
                                   (8, 6, 65), (9, 7, 66), (10, 5, 67), (1, 43, 130), (2, 12, 31), (21, 20, 33)])
def test_tile_edges_bitwise(dtype, shape):
    g, phi, prm = grid(shape, dtype, 40 + shape[0])
    ref, ex, sm = stepped(g, phi, 0, 1, prm)
    aligned = shape[2] % (4 if dtype == torch.float32 else 2) == 0
    for tile in (7, 8) + ((4, 5) if aligned else ()):
        for split in (1, 2, 5, cdi.CDI_NCHUNKS_BALANCED, cdi.CDI_NCHUNKS_ROTATED, 0):
            if split > shape[0]:
                continue
            out, e2, s2 = stepped(g, phi, tile, split, prm)
            assert torch.equal(out, ref), (tile, split)
            assert e2 == ex, (tile, split)
            # the sum's order differs: FP32 pairs of ~48 bits over per-thread sums of ~2 ulp
            assert abs(s2 - sm) <= (1e-12 if dtype == torch.float64 else 1e-7) * abs(sm), (tile, split)


def test_non_finite_cells_reach_the_same_cells():
    g, phi, prm = grid((6, 17, 67), torch.float32, 3)
    phi[2, 3, 66] = float("nan")
    phi[4, 16, 0] = float("inf")
    ref = None
    for tile in (0, 7, 8):
        g.set_launch(cdi.CDI_KERNEL_FORWARD, tile, 0, 0)
        b = torch.empty_like(phi)
        g.step(phi, b, *prm)
        bad = ~torch.isfinite(b)
        if ref is None:
            ref, rbad = b, bad
        assert torch.equal(bad, rbad) and torch.equal(b[~bad], ref[~bad])


def test_default_tile_reaches_the_row_kernel():
    """The default of a box with odd rows is the row kernel in FP32; w of a 2D box is not read."""
    g, phi, prm = grid((9, 40, 67), torch.float32, 5)
    assert g.get_launch()["tile"] in (7, 8)
    g, phi, prm = grid((1, 33, 67), torch.float32, 6)
    u, v, w = (torch.rand_like(phi) for _ in range(3))
    outs = []
    for ww in (w, torch.full_like(w, float("nan"))):
        g.set_velocity(u, v, ww, umax=1.0)
        b = torch.empty_like(phi)
        g.step(phi, b, *prm)
        outs.append(b)
    assert torch.isfinite(outs[0]).all() and torch.equal(*outs)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("scheme", ["rk2", "rk3", "rk4"])
@pytest.mark.parametrize("shape", [(3, 15, 67), (9, 29, 64), (1, 33, 30)])
def test_rk_stages_bitwise(dtype, scheme, shape):
    """Stage operands staged a plane ahead: every combination of the schemes' stages against the
    one-cell-per-thread stage kernel."""
    g, phi, prm = grid(shape, dtype, 60 + shape[0])
    outs = []
    for tile in (0, 7) + ((4,) if shape[2] % 4 == 0 else ()):
        g.set_launch(cdi.CDI_KERNEL_FORWARD, tile, 0, 0)
        a, b, w1, w2 = phi.clone(), *(torch.empty_like(phi) for _ in range(3))
        outs.append(g.run_rk(a, b, w1, w2, 3, *prm, scheme=scheme).clone())
    assert all(torch.equal(o, outs[0]) for o in outs[1:])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape,zr", [((11, 17, 67), (4, 9)), ((11, 17, 64), (0, 3)), ((16, 15, 33), (15, 16))])
def test_plane_range_bitwise(dtype, shape, zr):
    g, phi, prm = grid(shape, dtype, 80 + shape[0])
    ref, out = torch.empty_like(phi), torch.full_like(phi, 7.0)
    g.set_launch(cdi.CDI_KERNEL_FORWARD, 0, 0, 0)
    g.step(phi, ref, *prm)
    g.step_planes(phi, out, zr[0], zr[1], *prm)
    assert torch.equal(out[zr[0]:zr[1]], ref[zr[0]:zr[1]])
    assert (out[:zr[0]] == 7.0).all() and (out[zr[1]:] == 7.0).all()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("shape,split", [((1, 1, 5), 0), ((3, 13, 16), 1), ((5, 15, 63), 2), ((9, 28, 65), 0),
                                         ((6, 29, 67), cdi.CDI_NCHUNKS_BALANCED), ((21, 16, 130), 3),
                                         ((4, 43, 33), cdi.CDI_NCHUNKS_ROTATED), ((2, 14, 128), 0)])
@pytest.mark.parametrize("with_vel", [False, True])
def test_adjoint_tile_edges(dtype, shape, split, with_vel):
    """The adjoint row kernel for any row length (tile 4) and for aligned rows (tile 3): the
    oracle's adjoint step, and velocity gradients added to what the arrays held."""
    t = np.float64 if dtype == torch.float64 else np.float32
    nz, ny, nx = shape
    h = 1.0 / max(shape)
    rng = np.random.default_rng(7 + nx)
    phi = np.asarray(I.random_phi(shape, 11 + nx, smooth=True), t).astype(np.float64)
    u, v, w = (np.asarray(x, t).astype(np.float64) for x in I.random_velocity(shape, h, 8, 3, 5))
    lam = np.asarray(rng.standard_normal(shape), t).astype(np.float64)
    dt, eps, gamma, vs = 0.15 * h * h / (1.3 * 1.1 * h), 1.1 * h, 1.3, 0.7
    ref = oracle.adjoint(phi, u, v, w, lam, h, dt, eps, gamma, vs, want_vel=True, tiny=oracle.adjoint_floor_of(t))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)
    g = cdi.Grid(nx, ny, nz, h, dtype)
    g.set_velocity(*[dev(x) for x in (u, v, w)])
    base = np.asarray(rng.standard_normal((3,) + shape), t).astype(np.float64)
    tol = 1e-12 if dtype == torch.float64 else 2e-6  # the bounds of the other adjoint kernels' tests
    for tile in (4,) + ((3,) if nx % (4 if dtype == torch.float32 else 2) == 0 else ()):
        g.set_launch(cdi.CDI_KERNEL_ADJOINT, tile, 0, split)
        out = torch.empty(shape, dtype=dtype, device="cuda")
        grads = [dev(x) for x in base] if with_vel else None
        g.step_adjoint(dev(phi), dev(lam), out, dt, eps, gamma, vs, grads=grads)
        assert np.abs(out.double().cpu().numpy() - ref[0]).max() <= tol * max(1.0, np.abs(ref[0]).max())
        for a, b, r in zip(grads or (), base, ref[1:]):
            assert np.abs(a.double().cpu().numpy() - (b + r)).max() <= 4 * tol * max(1.0, np.abs(r).max())
