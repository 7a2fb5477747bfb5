"""The adjoint on a workspace full of garbage: grids large enough (64 MB of adjoint) to be cleared in the scan's
band alone give the gradients of a workspace of zeros, also for scans across the grid's top and bottom layers
(which positions outside it read), and for atom counts that fill the final sums' blocks and exceed them."""
import numpy as np
import pytest
import torch

from helpers import case32
from paper_2401_14564_gb300 import afm, pp, synth

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "z", "q", "R", "eps")


@pytest.mark.parametrize("n,lift", [(40, 0.0), (128, 0.0), (129, 0.0), (40, 9.9), (40, -3.9)])
def test_garbage_in_the_workspace_does_not_reach_the_gradients(n, lift):
    atoms = synth.random_molecule(n, n)
    top = float(atoms["z"].max())
    c = case32({"atoms": atoms, "probe": synth.default_probe(), "tip": synth.default_tip(kx=3.0, ky=3.0),
                "fire": synth.default_fire(), "df": synth.default_df(),
                "grid": {"nx": 180, "ny": 170, "nz": 144, "x0": -9.0, "y0": -8.5, "z0": top + 2.0, "dx": 0.1, "dy": 0.1,
                         "dz": 0.1, "periodic_xy": 1},
                "scan": {"nx": 40, "ny": 30, "nz": 13, "x0": -6.0, "y0": -6.0, "px": 0.3, "py": 0.4,
                         "z_top": top + 7.0 + 4.0 + lift, "dz": 0.1}})
    s = c["scan"]
    sim = afm.Simulator(c)
    dev = afm.atoms_to_device(c["atoms"])
    sim.make_ff(dev)
    k, j, i = np.meshgrid(np.arange(s["nz"]), np.arange(s["ny"]), np.arange(s["nx"]), indexing="ij")
    pos = torch.as_tensor(np.stack([s["x0"] + i * s["px"], s["y0"] + j * s["py"],
                                    s["z_top"] - k * s["dz"] - c["tip"]["R0"] + 0.02 * np.sin(i + j)], -1),
                          dtype=torch.float32, device="cuda").contiguous()
    w = torch.randn(sim.df.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    words = pp.pp_backward_workspace(sim.grid) // 4
    assert words * 4 >= 64 << 20
    out = []
    for fill in (0.0, 3.0):
        ws = torch.full((words,), fill, device="cuda")
        g = {q: torch.full((n,), float("nan"), device="cuda") for q in KEYS}
        g["tip"] = torch.full((5,), float("nan"), device="cuda")
        pp.pp_backward(pp.make_atoms(dev), sim.probe, sim.grid, sim.ff, sim.scan, sim.tip, sim.dfp, pos, w, pp.make_grads(g), ws)
        torch.cuda.synchronize()
        out.append(g)
    for q in (*KEYS, "tip"):
        a, b = (o[q].double() for o in out)
        assert torch.isfinite(a).all() and torch.isfinite(b).all(), q
        # (only the order of FP32 additions differs: the bar of the adjoint's other two-run test)
        assert float((a - b).norm()) <= 1e-4 * float(a.norm()), q
