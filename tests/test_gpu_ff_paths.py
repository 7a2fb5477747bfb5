"""The ways K1 assembles a grid (direct sums, direct sums about each tile's centre, tiles) on either side of each line:
every launch shape, layer range, layout and the batch write the same bits, and the grid matches the oracle.

Bars against the FP64 oracle: those of test_gpu_ff_tiles.py, over the grid 4e-6 and, for molecules, 1e-4 per node
(a sheet's nodes above its plane hold sums of terms a thousand times larger)."""
import numpy as np
import pytest
import torch

from helpers import case32, ff_rel_err, linear_ff
from paper_2401_14564_gb300 import batch, pp, synth
from test_gpu_ff_tiles import build

pytestmark = pytest.mark.gpu


def sheet(cells, shape, **probe):
    """A periodic sheet of cells[0] x cells[1] four-atom cells on one period."""
    atoms = synth.graphene_sheet(*cells, z=0.0)
    rng = np.random.default_rng(cells[0])
    for k in ("x", "y", "z"):
        atoms[k] = atoms[k] + rng.uniform(-0.05, 0.05, len(atoms[k]))
    nx, ny, nz = shape
    g = {"nx": nx, "ny": ny, "nz": nz, "x0": 0.0, "y0": 0.0, "z0": 1.6, "dx": cells[0] * 2.46 / nx,
         "dy": cells[1] * 2.46 * 3 ** 0.5 / ny, "dz": 0.1, "periodic_xy": 1}
    return {"atoms": atoms, "probe": synth.default_probe(coul_rc=8.0, min_image=1, **probe), "grid": g}


def molecule(n, shape, d, interp=0):
    atoms = synth.random_molecule(n, n)
    nx, ny, nz = shape
    g = {"nx": nx, "ny": ny, "nz": nz, "x0": -0.5 * nx * d, "y0": -0.5 * ny * d, "z0": float(atoms["z"].max()) + 1.7,
         "dx": d, "dy": d, "dz": d, "periodic_xy": 1, "interp": interp}
    return {"atoms": atoms, "probe": synth.default_probe(Qzz=-0.05 if n % 2 else 0.0), "grid": g}


# the line from either side: periodic cells, energies alone, 35 atoms (and 36, always by tiles; 15, always directly);
# ragged in every direction, with a last block of 4 layers or fewer (20, 28 and 60 layers; the last launched apart) and more
CASES = {"sheet_near": sheet((7, 5), (71, 93, 28)), "sheet_near_quad": sheet((7, 5), (71, 93, 23), Qzz=-0.05),
         "sheet_far": sheet((9, 6), (190, 201, 20)), "sheet_tail": sheet((14, 8), (142, 142, 60)),
         "energies_near": molecule(40, (55, 66, 60), 0.2, 1),
         "energies_far": molecule(40, (180, 151, 37), 0.1, 1), "atoms_35": molecule(35, (71, 66, 43), 0.1), "atoms_35_far": molecule(35, (190, 171, 43), 0.1),
        
         "atoms_36": molecule(36, (71, 66, 43), 0.1), "atoms_15": molecule(15, (71, 66, 43), 0.1)}
CASES = {k: case32(c) for k, c in CASES.items()}


@pytest.mark.parametrize("name", sorted(CASES))
def test_every_path_matches_the_oracle(orc, name):
    c = CASES[name]
    ff, _ = build(c)
    ref, core = orc.make_ff(c["atoms"], c["probe"], dict(c["grid"], interp=0))
    if c["grid"].get("interp"):
        E = ff.cpu().numpy().astype(np.float64).reshape(ref.shape[:3])
        assert (np.abs(E - ref[..., 3]) / np.maximum(np.abs(ref[..., 3]), 1e-2))[~core].max() <= 1e-4
        return
    F = linear_ff(ff.cpu().numpy(), c["grid"])
    if not name.startswith("sheet"):
        assert ff_rel_err(F, ref)[~core].max() <= 1e-4
    a, b = F[..., :3][~core], ref[..., :3][~core]
    assert np.linalg.norm(a - b) <= 4e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("name", sorted(CASES))
def test_ranges_shapes_and_layouts_write_the_same_bits(name):
    c = CASES[name]
    g = c["grid"]
    per = 1 if g.get("interp") else 4
    whole, _ = build(c)
    plane = g["nx"] * g["ny"] * per
    nz = g["nz"]
    for k0, k1 in ((0, 1), (3, nz - 2), (8, 16), (12, 16), (15, 17), (4, 13), (nz - 1, nz), (0, nz)):
        part, _ = build(c, layers=(k0, k1))
        assert torch.equal(part[k0 * plane:k1 * plane], whole[k0 * plane:k1 * plane]), (k0, k1)
        assert torch.isnan(part[:k0 * plane]).all() and torch.isnan(part[k1 * plane:]).all(), (k0, k1)
    if per == 1:
        return
    for zpt in (4, 16):
        assert torch.equal(build(c, zpt=zpt)[0], whole)
    forces, _ = build(c, forces=1)
    assert torch.equal(forces.view(-1, 4)[:, :3], whole.view(-1, 4)[:, :3])
    assert torch.count_nonzero(forces.view(-1, 4)[:, 3]).item() == 0
    brick, gb = build(c, layout=1)
    lin = torch.empty_like(whole)
    pp.pp_ff_convert(brick, gb, lin, pp.make_grid(g, 0))
    assert torch.equal(lin, whole)


@pytest.mark.parametrize("group", [("sheet_near", "sheet_far"), ("sheet_near_quad",), ("atoms_36", "atoms_15"), ("atoms_35", "atoms_35_far")])
def test_the_batch_writes_the_bits_of_k1(group):
    extra = {"tip": synth.default_tip(), "fire": synth.default_fire(max_iter=2), "df": synth.default_df()}
    cs = []
    for name in group:
        c = dict(CASES[name], **extra)
        if name.startswith("atoms"):
            c["probe"] = CASES["atoms_36"]["probe"] if len(group) > 1 else c["probe"]
        c["scan"] = {"nx": 4, "ny": 4, "nz": 11, "x0": 0.0, "y0": 0.0, "px": 0.3, "py": 0.3,
                     "z_top": c["grid"]["z0"] + 1.9 + 4.0, "dz": 0.1}
        cs.append(case32(c))
    b = batch.Batch(cs)
    b.run()
    assert b.status() == (0, 0)
    for n, c in enumerate(cs):
        assert torch.equal(b.molecule(n)["ff"].reshape(-1), build(c)[0]), group[n]


@pytest.mark.parametrize("value", [1e30, -2.5e38, float("inf")])
@pytest.mark.parametrize("key", ["x", "z"])
def test_an_atom_out_of_all_reach_adds_nothing_to_the_energies(key, value):
    c = CASES["energies_near"]
    want, _ = build(c)
    atoms = {k: np.append(v, v[:1]) for k, v in c["atoms"].items()}
    atoms[key][-1] = value
    got, _ = build(dict(c, atoms=atoms))
    assert torch.equal(got, want)
