"""The scan's pixels per warp: every tile shape, asked for or chosen by the library, writes the same bits.

Sizes: one pixel, a single row and column, one pixel past each tile's width and height, and a scan large
enough for full warps."""
import pytest
import torch

from helpers import case32
from paper_2401_14564_gb300 import afm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("px,py", [(1, 1), (1, 37), (33, 1), (9, 5), (17, 13), (160, 129)])
@pytest.mark.parametrize("variant", ["plain", "polish", "tricubic"])
def test_every_tile_shape_writes_the_same_bits(px, py, variant):
    c = case32(synth.small_case(seed=31, n_atoms=11, nxy=40, nz=44, scan_px=17, nz_scan=12))
    c["scan"] = dict(c["scan"], nx=px, ny=py, px=4.0 / px, py=4.0 / py)
    c["grid"] = dict(c["grid"], interp=int(variant == "tricubic"))
    fire = synth.default_fire(polish=4 if variant == "polish" else 0)
    sim = afm.Simulator(case32(c), fire=fire, plan_frac=0.0)
    atoms = afm.atoms_to_device(c["atoms"])
    want = None
    for lanes in (32, 0, 16, 8, 4, 2, 1, 31):
        sim.scan_lanes = lanes
        for t in (sim.df, sim.fz, sim.pos):
            t.fill_(float("nan"))
        sim.iters.fill_(-1)
        sim.run(atoms)
        got = [t.clone() for t in (sim.df, sim.fz, sim.pos, sim.iters)]
        assert all(torch.isfinite(t).all() for t in got[:3]) and (got[3] >= 0).all()
        if want is None:
            want = got
        assert all(torch.equal(a, b) for a, b in zip(got, want)), lanes
