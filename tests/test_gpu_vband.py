"""Batch tile 6 (bands of whole rows of the batch's padded copies) at the edges of its layout: every
remainder of a row against its 16-byte vectors, rows of one vector and less, group counts that are
and are not multiples of eight (the staged pitch), bands that leave whole warps without cells, unit
depths around the four phi slots and three velocity slots, and the caller's arrays on and off
16-byte boundaries.  Reference: the one-cell-per-thread tile 0, which computes the same
expressions in the same order, so the fields must be equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(4, 9, 1), (5, 90, 2), (3, 6, 3), (6, 84, 4), (1, 12, 5), (7, 33, 6), (9, 30, 31), (5, 34, 32), (8, 17, 33),
          (4, 21, 34), (2, 22, 35), (3, 19, 60), (6, 11, 97), (5, 8, 131), (4, 3, 199)]


def placed(x, dtype, o):
    buf = torch.zeros(x.size + o, dtype=dtype, device="cuda")
    y = buf[o:].view(x.shape)
    y.copy_(torch.from_numpy(np.ascontiguousarray(x)))
    return y


def boxes(dtype, o):
    out = []
    for i, s in enumerate(SHAPES):
        h = 1.0 / max(s)
        vel = [placed(v, dtype, o) for v in I.random_velocity(s, h, 8, 3, 70 + i)]
        eps, gamma = 1.1 * h, 1.0
        phi = placed(I.random_phi(s, 20 + i, smooth=True), dtype, o)
        out.append(dict(dx=h, dt=0.1 * h * h / (gamma * eps), eps=eps, gamma=gamma, u=vel[0], v=vel[1], w=vel[2],
                        phi_a=phi, phi_b=placed(np.zeros(s), dtype, o)))
    return out


@pytest.mark.parametrize("dtype,o", [(torch.float32, 0), (torch.float32, 1), (torch.float64, 0), (torch.float64, 1)])
@pytest.mark.parametrize("zdepth", [0, 2, 4])
def test_layout_edges_bitwise(dtype, o, zdepth):
    ours, ref = cdi.Batch(boxes(dtype, o)), cdi.Batch(boxes(dtype, o))
    ours.set_launch(6, zdepth)
    ref.set_launch(0, zdepth)
    assert ours.get_launch()["tile"] == 6
    for b in (ours, ref):
        b.step(0.7)
        b.run(5)
    for i, s in enumerate(SHAPES):
        assert torch.equal(ours.current(i), ref.current(i)), s
    for a, b in zip(ours.stats(), ref.stats()):
        assert all(a[k] == b[k] for k in ("min", "max", "n_strict", "n_tol"))
