"""Row kernels on rows that start on pairs of FP32 cells (nx even, not a multiple of four): copies,
stores and gradient reductions two cells at a time, at the tile's edges (16 vectors, rows of a
pair, groups of two at a row's end, heights of 6 and 14 rows).  Reference: tile 0's fields bit for
bit; for the adjoint the row kernel by elements does not run on these rows, so the one-cell-per-thread
tile, to the bounds of the other adjoint tests."""
import pytest
import torch

from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 2), (3, 13, 18), (5, 15, 62), (9, 7, 66), (6, 29, 126), (2, 12, 130), (7, 28, 34)]


def grid(shape):
    nz, ny, nx = shape
    h = 1.0 / max(shape)
    dev = lambda x: torch.from_numpy(x).to("cuda", torch.float32)
    g = cdi.Grid(nx, ny, nz, h, torch.float32)
    g.set_velocity(*[dev(x) for x in I.random_velocity(shape, h, 8, 3, 9)])
    eps, gamma = 1.1 * h, 1.0
    return g, dev(I.random_phi(shape, 30 + nx, smooth=True)), (0.1 * h * h / (gamma * eps), eps, gamma)


@pytest.mark.parametrize("shape", SHAPES)
def test_forward_rk_and_planes_bitwise(shape):
    g, phi, prm = grid(shape)
    runs, rks = [], []
    for tile in (0, 7, 8):
        g.set_launch(cdi.CDI_KERNEL_FORWARD, tile)
        a, b, w1, w2 = phi.clone(), *(torch.empty_like(phi) for _ in range(3))
        runs.append(g.run(a, b, 3, *prm).clone())
        a.copy_(phi)
        rks.append(g.step_rk(a, b, w1, w2, *prm, scheme="rk4").clone())
    assert all(torch.equal(x, runs[0]) for x in runs) and all(torch.equal(x, rks[0]) for x in rks)
    if shape[0] > 2:
        ref, out = torch.empty_like(phi), torch.full_like(phi, 7.0)
        g.step(phi, ref, *prm)
        g.step_planes(phi, out, 1, 3, *prm)
        assert torch.equal(out[1:3], ref[1:3]) and (out[0] == 7.0).all() and (out[3:] == 7.0).all()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("with_vel", [False, True])
def test_adjoint(shape, with_vel):
    g, phi, prm = grid(shape)
    lam = torch.randn_like(phi)
    res = []
    for tile in (1, 4):
        g.set_launch(cdi.CDI_KERNEL_ADJOINT, tile)
        gr = [torch.ones_like(phi) for _ in range(3)] if with_vel else None
        res.append([g.step_adjoint(phi, lam, torch.empty_like(lam), *prm, grads=gr)] + (gr or []))
    for a, b in zip(*res):
        assert (a - b).abs().max() <= 4e-6 * max(1.0, float(a.abs().max()))
