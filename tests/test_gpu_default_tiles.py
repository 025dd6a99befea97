"""Default launches of boxes whose rows do not start on 16-byte boundaries, where two kernels are near
each other: the rule takes the one that was measured faster, on each side of its lines."""
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
