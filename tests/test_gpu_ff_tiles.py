"""K1 by tiles (16 atoms and more): far atoms of a 16x16x16-node tile summed at its 8x8x8 Chebyshev points
and interpolated, near atoms at the nodes.

Bars against the FP64 oracle: the per-node bar of the direct kernel (1e-4 with a 1e-3 eV/A floor), and over
the grid a relative 2-norm of 4e-6: a pair's r^-8 from an rsqrt of 2 ulp is good to 8 x 2 x 2^-24 = 1e-6, the
r^-14 of a repulsive pair to 1.7e-6, and the interpolation adds at most 1.5e-7 of a pair's force; doubled.
"""
import numpy as np
import pytest
import torch

from helpers import case32, ff_rel_err, linear_ff
from paper_2401_14564_gb300 import afm, pp, synth

pytestmark = pytest.mark.gpu

PROBES = {"plain": dict(), "quad": dict(Qzz=-0.05), "image_cut": dict(coul_rc=8.0, min_image=1),
          "cut_quad": dict(coul_rc=6.5, Qzz=-0.05)}


def case(n, shape, d, probe, periodic=None):
    atoms = synth.random_molecule(n, n)
    nx, ny, nz = shape
    dx, dy = (d, d) if periodic is None else (periodic / nx, periodic / ny)
    c = {"atoms": atoms, "probe": synth.default_probe(**PROBES[probe]),
         "grid": {"nx": nx, "ny": ny, "nz": nz, "x0": -0.5 * nx * dx, "y0": -0.5 * ny * dy,
                  "z0": float(atoms["z"].max()) + 1.7, "dx": dx, "dy": dy, "dz": d, "periodic_xy": 1}}
    return case32(c)


def build(c, layout=0, zpt=0, forces=0, layers=None):
    grid = pp.make_grid(c["grid"], layout)
    ff = torch.full((pp.pp_ff_floats(grid),), float("nan"), device="cuda")
    args = (pp.make_atoms(afm.atoms_to_device(c["atoms"])), pp.make_probe(c["probe"]), grid, ff)
    if layers:
        pp.pp_make_ff_layers(*args, *layers, pp.Tuning(zpt, forces))
    elif c["grid"].get("interp"):
        pp.pp_make_ff(*args)
    else:
        pp.pp_make_ff_tuned(*args, pp.Tuning(zpt, forces))
    return ff, grid


# one tile exactly, one node past it each way, a tile of one node, and several ragged tiles; 15 atoms (direct),
# 16 and 24 (some tiles with too few far atoms), 300 (two classification passes); spacings that make
# most atoms far, some, and none
@pytest.mark.parametrize("probe", sorted(PROBES))
@pytest.mark.parametrize("n,shape,d", [(15, (17, 16, 33), 0.1), (16, (16, 16, 16), 0.1), (24, (17, 33, 18), 0.1),
                                       (60, (49, 35, 41), 0.1), (60, (33, 18, 17), 0.25), (300, (33, 17, 50), 0.08),
                                       (300, (2, 3, 2), 0.1)])
def test_tiles_match_the_oracle(orc, n, shape, d, probe):
    c = case(n, shape, d, probe, periodic=31.3 if probe == "image_cut" else None)
    ff, _ = build(c)
    F = linear_ff(ff.cpu().numpy(), c["grid"])
    ref, core = orc.make_ff(c["atoms"], c["probe"], c["grid"])
    assert np.isfinite(F).all()
    assert ff_rel_err(F, ref)[~core].max() <= 1e-4
    eerr = np.abs(F[..., 3] - ref[..., 3]) / np.maximum(np.abs(ref[..., 3]), 1e-2)
    assert eerr[~core].max() <= 1e-4
    a, b = F[..., :3][~core], ref[..., :3][~core]
    assert np.linalg.norm(a - b) <= 4e-6 * np.linalg.norm(b)
    c["grid"]["interp"] = 1
    E, _ = build(c)
    E = E.cpu().numpy().astype(np.float64).reshape(ref.shape[:3])
    err = np.abs(E - ref[..., 3]) / np.maximum(np.abs(ref[..., 3]), 1e-2)
    assert err[~core].max() <= 1e-4


@pytest.mark.parametrize("probe", ["plain", "image_cut"])
def test_layer_ranges_shapes_and_layouts_write_the_same_bits(probe):
    c = case(70, (35, 20, 43), 0.1, probe, periodic=31.3 if probe == "image_cut" else None)
    whole, _ = build(c)
    plane = c["grid"]["nx"] * c["grid"]["ny"] * 4
    for zpt in (4, 16):
        assert torch.equal(build(c, zpt=zpt)[0], whole)
    forces, _ = build(c, forces=1)
    assert torch.equal(forces.view(-1, 4)[:, :3], whole.view(-1, 4)[:, :3])
    assert torch.count_nonzero(forces.view(-1, 4)[:, 3]).item() == 0
    for k0, k1 in ((0, 1), (3, 26), (8, 16), (15, 17), (24, 43), (42, 43)):
        part, _ = build(c, layers=(k0, k1))
        assert torch.equal(part[k0 * plane:k1 * plane], whole[k0 * plane:k1 * plane]), (k0, k1)
        assert torch.isnan(part[:k0 * plane]).all() and torch.isnan(part[k1 * plane:]).all(), (k0, k1)
    brick, gb = build(c, layout=1)
    lin = torch.empty_like(whole)
    pp.pp_ff_convert(brick, gb, lin, pp.make_grid(c["grid"], 0))
    assert torch.equal(lin, whole)


@pytest.mark.parametrize("key,value", [("q", float("inf")), ("q", float("nan")), ("eps", float("inf")), ("x", float("nan"))])
def test_non_finite_atoms_spoil_every_node_as_a_direct_sum_does(key, value):
    c = case(40, (33, 17, 20), 0.1, "plain")
    c["atoms"][key] = np.array(c["atoms"][key])
    c["atoms"][key][7] = value
    ff, _ = build(c)
    # (a NaN coordinate reaches its own force component alone: the core floor takes the place of its r^2)
    assert not torch.isfinite(ff.view(-1, 4)).all(dim=1).any()
