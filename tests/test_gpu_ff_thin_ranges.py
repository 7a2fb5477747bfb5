"""Layer ranges that end inside a half tile run by quarters of four layers: every range of a two-tile grid around the
quarters' edges writes the whole grid's bits and nothing else."""
import pytest
import torch

from test_gpu_ff_tiles import build, case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("probe", ["quad", "image_cut"])
def test_ranges_around_quarter_edges(probe):
    c = case(70, (35, 20, 27), 0.1, probe, periodic=31.3 if probe == "image_cut" else None)
    whole, _ = build(c)
    plane = c["grid"]["nx"] * c["grid"]["ny"] * 4
    edges = (0, 3, 4, 5, 8, 11, 12, 15, 16, 17, 20, 24, 25, 27)
    for k0 in edges:
        for k1 in edges:
            if k1 > k0:
                part, _ = build(c, layers=(k0, k1))
                assert torch.equal(part[k0 * plane:k1 * plane], whole[k0 * plane:k1 * plane]), (k0, k1)
                assert torch.isnan(part[:k0 * plane]).all() and torch.isnan(part[k1 * plane:]).all(), (k0, k1)
