"""The FFT path's half-spectrum kernels at the edges of their ranges: one column past a tile of columns (every
half spectrum is), lengths of one radix, with and without a remainder stage, along each axis, the longest
axis beside the shortest, powers and accumulation, and the scratch: the values outside what
pp_fft_workspace() asks for stay untouched.

Bar: that of the other FFT tests, 2e-5 of each component's largest magnitude; a component that vanishes
identically (an axis of length 2 has only its Nyquist mode) shares a complex transform with another and holds its
rounding, so it is measured against the field's largest.  Added to a grid, one FP32 rounding of the sum more."""
import numpy as np
import pytest
import torch

from paper_2401_14564_gb300 import pp
from test_gpu_fft import TOL, fields, grid, run

pytestmark = pytest.mark.gpu


def check(got, ref, before=0.0):
    got, rounding = got - before, 2.0 ** -23 * np.abs(ref + before).max() if np.any(before) else 0.0
    largest = np.abs(ref).max()
    for c in range(4):
        scale = np.abs(ref[..., c]).max()
        err = np.abs(got[..., c] - ref[..., c]).max()
        assert err <= TOL * (scale if scale > 1e-6 * largest else largest) + rounding, (c, err, scale)


@pytest.mark.parametrize("shape", [(2, 8, 16), (4, 2, 8), (8, 4, 2), (16, 2, 32), (64, 4, 8), (128, 2, 4), (2, 32, 64),
                                   (32, 64, 2)])
@pytest.mark.parametrize("power,accumulate", [(1.0, False), (1.2, True)])
def test_small_grids_match_the_oracle(orc, shape, power, accumulate):
    g = grid(*shape)
    f, tip = fields(g, sum(shape))
    if power == 1.0:
        f = f - f.mean()
    n = f.size
    base = torch.randn(4 * n, device="cuda") if accumulate else None
    before = base.cpu().numpy().astype(np.float64).reshape(*f.shape, 4) if accumulate else 0.0
    got = run(f, tip, g, scale=0.6, power=power, ff=base, accumulate=accumulate)
    check(got, orc.correlate(f, tip, g, scale=0.6, power=power), before)


@pytest.mark.parametrize("shape", [(256, 4, 512), (512, 512, 2), (2, 256, 1024), (1024, 2, 2)])
def test_long_axes_against_the_direct_sum(orc, shape):
    g = grid(*shape, d=(0.05, 0.07, 0.06))
    f, tip = fields(g, sum(shape))
    got = run(f, tip, g, scale=1.3, power=1.05)
    nodes = np.random.default_rng(7).choice(f.size, 16, replace=False)
    E = orc.correlate_nodes(f, tip, g, nodes, scale=1.3, power=1.05)
    assert np.abs(got[..., 3].reshape(-1)[nodes] - E).max() <= TOL * np.abs(got[..., 3]).max()
    assert np.isfinite(got).all()


@pytest.mark.parametrize("shape", [(2, 2, 2), (32, 16, 8), (64, 32, 16)])
def test_scratch_stays_inside_its_size(shape):
    gr = pp.make_grid(grid(*shape), 0)
    n = shape[0] * shape[1] * shape[2]
    words = pp.pp_fft_workspace(gr) // 4
    ws = torch.full((words + 256,), 7.0, device="cuda")
    f, t = torch.rand(n, device="cuda"), torch.rand(n, device="cuda")
    ff = torch.empty(4 * n, device="cuda")
    pp.pp_fft_correlate(f, t, gr, 1.0, 1.0, ff, ws[:words])
    torch.cuda.synchronize()
    assert (ws[words:] == 7.0).all() and torch.isfinite(ff).all()
