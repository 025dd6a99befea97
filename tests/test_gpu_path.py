"""A checkpoint segment in one native call (step_path, adjoint_path) against the same steps called
one by one: the same kernels, so the states and lam are equal bit for bit (the velocity gradients to
the rounding of their order of addition), for no, one and several steps, with a scale per step; and
a Grid whose step is overridden is still called per step by rollout."""
import pytest
import torch

from paper_1803_01262_gb300 import autograd as AG
from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def setup(shape, dtype, cls=cdi.Grid):
    nz, ny, nx = shape
    h = 1.0 / max(shape)
    dev = lambda x: torch.from_numpy(x).to("cuda", dtype)
    g = cls(nx, ny, nz, h, dtype)
    vel = [dev(x) for x in I.random_velocity(shape, h, 8, 3, 5)]
    g.set_velocity(*vel)
    return g, dev(I.random_phi(shape, 4, smooth=True)), vel, (0.1 * h, 1.1 * h, 1.0)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", [(9, 21, 33), (6, 16, 64), (1, 20, 24)])
@pytest.mark.parametrize("n", [0, 1, 4, 5])
def test_paths_equal_single_steps(dtype, shape, n):
    g, phi, vel, prm = setup(shape, dtype)
    scales = [0.9 - 0.1 * i for i in range(n)]
    states = [phi] + [torch.empty_like(phi) for _ in range(n)]
    assert g.step_path(states, *prm, scales) is states[-1]
    ref, p = [phi], phi
    for vs in scales:
        p = g.step(p, torch.empty_like(phi), *prm, vs)
        ref.append(p)
    assert all(torch.equal(a, b) for a, b in zip(states, ref))
    lam = torch.randn_like(phi)
    gr, gs = [torch.zeros_like(phi) for _ in range(3)], [torch.zeros_like(phi) for _ in range(3)]
    la, other = g.adjoint_path(states[:n], lam.clone(), torch.empty_like(lam), *prm, scales, grads=gr)
    a, b = lam.clone(), torch.empty_like(lam)
    for p, vs in zip(reversed(ref[:n]), reversed(scales)):
        g.step_adjoint(p, a, b, *prm, vs, grads=gs)
        a, b = b, a
    assert la is not other and torch.equal(la, a)
    # n additions of terms rounded alike, in any order
    eps = torch.finfo(dtype).eps
    for x, y in zip(gr, gs):
        assert (x - y).abs().max() <= 4 * max(n, 1) * eps * y.abs().max() + 1e-300


def test_paths_refuse_mismatched_lists():
    g, phi, vel, prm = setup((4, 8, 8), torch.float32)
    with pytest.raises(ValueError):
        g.step_path([phi], *prm, [1.0])
    with pytest.raises(ValueError):
        g.adjoint_path([phi, phi.clone()], phi.clone(), phi.clone(), *prm, [1.0])
    with pytest.raises(cdi.CDIError):
        g.step_path([phi, phi], *prm, [1.0])  # in place


def test_overridden_step_is_called():
    class Counting(cdi.Grid):
        n = 0

        def step(self, *a, **k):
            Counting.n += 1
            return super().step(*a, **k)

    g, phi, vel, prm = setup((5, 9, 16), torch.float32, Counting)
    out = AG.rollout(phi, *vel, g, 3, *prm)
    g2, _, _, _ = setup((5, 9, 16), torch.float32)
    assert Counting.n == 3 and torch.equal(out, AG.rollout(phi, *vel, g2, 3, *prm))


@pytest.mark.parametrize("bad", ["in place", "scale"])
def test_a_refused_path_enqueues_nothing(bad):
    """A path refused for a later step leaves the states and the run statistics as they were."""
    g, phi, vel, prm = setup((6, 16, 64), torch.float32)
    g.step(phi, torch.empty_like(phi), *prm)
    st = g.stats()
    out = torch.full_like(phi, 7.0)
    states, scales = ([phi, out, out], [1.0, 1.0]) if bad == "in place" else (
        [phi, out, phi.clone()], [1.0, float("inf")])
    with pytest.raises(cdi.CDIError) as e:
        g.step_path(states, *prm, scales)
    assert e.value.code == cdi.CDI_ERR_ARG
    assert (out == 7.0).all() and g.stats() == st
    with pytest.raises(cdi.CDIError):       # no grid, no steps
        cdi._ck(cdi.lib().cdi_step_path(None, None, 0, *prm, None, None))
