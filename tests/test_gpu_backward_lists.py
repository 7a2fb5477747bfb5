"""K5 by tiles: atom lists at the edges where they are split over a CTA's threads (a little above a power of two, three
quarters of one, full), on grids with nearly all atoms near (near parts of two layers) and with many far (four).

At given positions and grid the atoms' gradients are sums over the grid's adjoint, whoever else is in the sample: against
calls of 15 atoms each, which are contracted directly, relative L2 <= 1e-4 per vector (the bar of the adjoint's other
tests)."""
import numpy as np
import pytest

from helpers import case32
from paper_2401_14564_gb300 import synth
from test_gpu_backward import KEYS, gpu_backward, rel, weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [24, 25, 33, 48, 49, 97, 128, 129, 193, 256, 257])
@pytest.mark.parametrize("nx,ny,d", [(40, 37, 0.15), (130, 121, 0.1)])
def test_atom_lists_of_every_length_match_the_oracle(orc, n, nx, ny, d):
    atoms = synth.random_molecule(n, n)
    top = float(atoms["z"].max())
    nz = 40 if d == 0.15 else 45
    c = {"atoms": atoms, "probe": synth.default_probe(Qzz=-0.05 if n % 2 else 0.0), "tip": synth.default_tip(kx=3.0, ky=2.5),
         "fire": synth.default_fire(), "df": synth.default_df(),
         "grid": {"nx": nx, "ny": ny, "nz": nz, "x0": -0.5 * nx * d, "y0": -0.5 * ny * d, "z0": top + 2.2,
                  "dx": d, "dy": d, "dz": d, "periodic_xy": 1},
         "scan": {"nx": 9, "ny": 7, "nz": 14, "x0": -0.3 * nx * d, "y0": -0.3 * ny * d, "px": 0.6 * nx * d / 9,
                  "py": 0.6 * ny * d / 7, "z_top": top + 3.6 + 1.3 + 4.0, "dz": 0.1}}
    c = case32(c)
    s = c["scan"]
    ff, _ = orc.make_ff(c["atoms"], c["probe"], c["grid"])
    k, j, i = np.meshgrid(np.arange(s["nz"]), np.arange(s["ny"]), np.arange(s["nx"]), indexing="ij")
    pos = np.stack([s["x0"] + i * s["px"] + 0.13 * np.sin(1.7 * i + 0.4 * k), s["y0"] + j * s["py"] + 0.11 * np.cos(1.3 * j),
                    s["z_top"] - k * s["dz"] - c["tip"]["R0"] + 0.03 * np.sin(i + j + 0.7 * k)], -1)
    pos = pos.astype(np.float32).astype(np.float64)
    w = weights(c, 3).astype(np.float32).astype(np.float64)
    got = gpu_backward(c, pos, w, ff_host=ff)
    parts = [gpu_backward(dict(c, atoms={q: np.asarray(v)[a:a + 15] for q, v in c["atoms"].items()}), pos, w, ff_host=ff)
             for a in range(0, n, 15)]
    ref = {q: np.concatenate([p[q] for p in parts]) for q in KEYS}
    ref["Q"] = sum(p["Q"] for p in parts)
    bad = {q: rel(got[q], ref[q]) for q in KEYS + ("Q",) if not rel(got[q], ref[q]) <= 1e-4}
    assert not bad, bad
