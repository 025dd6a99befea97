"""Scalar adjoint tiles with their default split on boxes whose default launch is the row kernel with
a rotated split (a split those tiles do not have): the launch is accepted and lam is the row
kernel's to rounding."""
import pytest
import torch

from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,shape", [(torch.float32, (72, 134, 198)), (torch.float64, (72, 88, 128)),
                                         (torch.float64, (62, 118, 143))])
def test_scalar_tiles_after_a_rotated_default(dtype, shape):
    nz, ny, nx = shape
    h = 1.0 / max(shape)
    dev = lambda x: torch.from_numpy(x).to("cuda", dtype)
    g = cdi.Grid(nx, ny, nz, h, dtype)
    g.set_velocity(*[dev(x) for x in I.random_velocity(shape, h, 8, 3, 2)])
    phi = dev(I.random_phi(shape, 1, smooth=True))
    lam = torch.randn_like(phi)
    eps, gamma = 1.1 * h, 1.0
    prm = (0.1 * h * h / (gamma * eps), eps, gamma)
    ref = g.step_adjoint(phi, lam, torch.empty_like(lam), *prm)
    # each cell's update is a sum of about 40 terms of at most |lam| in another order of rounding,
    # the normals' derivative floored at 8 machine epsilons: a few hundred units of rounding
    tol = 400 * torch.finfo(dtype).eps * float(lam.abs().max())
    for tile in (0, 1, 2):
        g.set_launch(cdi.CDI_KERNEL_ADJOINT, tile)
        out = g.step_adjoint(phi, lam, torch.empty_like(lam), *prm)
        assert g.get_launch(cdi.CDI_KERNEL_ADJOINT)["tile"] == tile
        assert (out - ref).abs().max() <= tol
