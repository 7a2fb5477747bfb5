"""K5 by tiles: the node adjoints carried to a tile's points for far atoms, contracted with the nodes for near ones.

What K5 forms (the atoms' gradients and dL/dQ) at given positions against the FP64 oracle (relative L2 <=
1e-4 per vector, the bar of the adjoint's other tests) at the edges of its ranges: 16 atoms, lists that fill a slot count exactly and just
exceed it, more than one classification pass, grids of one tile, one node past it and ragged, image switches
and cutoff crossings, and too few far atoms for the points."""
import numpy as np
import pytest

from helpers import case32
from paper_2401_14564_gb300 import synth
from test_gpu_backward import KEYS, gpu_backward, rel, weights

pytestmark = pytest.mark.gpu

PROBES = {"plain": dict(), "quad": dict(Qzz=-0.05), "image_cut": dict(coul_rc=7.0, min_image=1),
          "cut_quad": dict(coul_rc=6.0, Qzz=-0.05)}


@pytest.mark.parametrize("probe", sorted(PROBES))
@pytest.mark.parametrize("n,nx,ny,nz,d", [(16, 16, 17, 48, 0.12), (17, 33, 16, 49, 0.12), (65, 40, 35, 45, 0.1),
                                          (260, 35, 34, 44, 0.1)])
def test_tiled_adjoint_matches_the_oracle(orc, n, nx, ny, nz, d, probe):
    atoms = synth.random_molecule(n, n)
    top = float(atoms["z"].max())
    if probe == "image_cut":
        nx, ny = nx + 65, ny + 65  # a period of 26.1 A in x at up to 0.33 A a node
    dx, dy = (d, d) if probe != "image_cut" else (26.1 / nx, 26.1 / ny)
    c = {"atoms": atoms, "probe": synth.default_probe(**PROBES[probe]), "tip": synth.default_tip(kx=3.0, ky=2.5),
         "fire": synth.default_fire(), "df": synth.default_df(),
         "grid": {"nx": nx, "ny": ny, "nz": nz, "x0": -0.5 * nx * dx, "y0": -0.5 * ny * dy, "z0": top + 2.2,
                  "dx": dx, "dy": dy, "dz": d, "periodic_xy": 1},
         "scan": {"nx": 9, "ny": 7, "nz": 14, "x0": -0.3 * nx * dx, "y0": -0.3 * ny * dy, "px": 0.6 * nx * dx / 9,
                  "py": 0.6 * ny * dy / 7, "z_top": top + 3.6 + 1.3 + 4.0, "dz": 0.1}}
    c = case32(c)
    s = c["scan"]
    ff, _ = orc.make_ff(c["atoms"], c["probe"], c["grid"])
    # positions: the rest position displaced by a fixed smooth field (the adjoint takes any)
    k, j, i = np.meshgrid(np.arange(s["nz"]), np.arange(s["ny"]), np.arange(s["nx"]), indexing="ij")
    pos = np.stack([s["x0"] + i * s["px"] + 0.13 * np.sin(1.7 * i + 0.4 * k), s["y0"] + j * s["py"] + 0.11 * np.cos(1.3 * j),
                    s["z_top"] - k * s["dz"] - c["tip"]["R0"] + 0.03 * np.sin(i + j + 0.7 * k)], -1)
    pos = pos.astype(np.float32).astype(np.float64)
    w = weights(c, 3).astype(np.float32).astype(np.float64)
    ref = orc.backward(ff, c["grid"], c["atoms"], c["probe"], s, c["tip"], c["df"], pos, w)
    got = gpu_backward(c, pos, w, ff_host=ff)
    bad = {q: rel(got[q], ref[q]) for q in KEYS + ("Q",) if not rel(got[q], ref[q]) <= 1e-4}
    assert not bad, bad
