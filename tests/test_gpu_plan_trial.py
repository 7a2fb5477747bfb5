"""Scans of one to eight pixel tiles per SM: auto_plan looks at a plan's figures and plans from then on or not at all."""
import pytest
import torch

from helpers import case32
from paper_2401_14564_gb300 import afm, pp, synth

pytestmark = pytest.mark.gpu


def simulator(px, **kw):
    c = case32(synth.small_case(seed=31, n_atoms=11, nxy=40, nz=44, scan_px=17, nz_scan=12))
    c["scan"] = dict(c["scan"], nx=px, ny=px, px=4.0 / px, py=4.0 / px)
    return afm.Simulator(case32(c), **kw), afm.atoms_to_device(c["atoms"])


def test_the_plans_header_holds_the_costliest_columns():
    sim, _ = simulator(100, auto_plan=False, plan_frac=0.02)
    nz = sim.scan.nz
    gen = torch.Generator(device="cuda").manual_seed(2)
    iters = torch.randint(0, 40, (nz, 100, 100), device="cuda", generator=gen, dtype=torch.int32)
    iters[:, 7, 9] = 300
    sim.plan_from(iters)
    cost = iters.sum(0).flatten()
    npix = cost.numel()
    mask = sim._plan[-((npix + 31) // 32):]
    listed = ((mask[torch.arange(npix, device="cuda") // 32] >> (torch.arange(npix, device="cuda") % 32)) & 1).bool()
    assert int(listed.sum()) == sim._plan_k == 200
    assert int(sim._plan[5]) == int(cost.max()) == 300 * nz and int(sim._plan[6]) == int(cost[~listed].max())


@pytest.mark.parametrize("gain", [0, 10 ** 6])
def test_every_scan_plans_or_none_does_once_the_figures_are_here(gain, monkeypatch):
    sim, atoms = simulator(100)  # 325 tiles
    plain, _ = simulator(100, plan_frac=0.0)
    plain.run(atoms)
    looks = []

    def pays(g, tiles):
        looks.append((g, tiles))
        return gain > 0

    monkeypatch.setattr(sim, "plan_pays", pays)
    held = []
    for _ in range(2 * sim._PLAN_EVERY):
        sim.run(atoms)
        torch.cuda.synchronize()
        held.append(sim._plan_ready)
        assert torch.equal(sim.df, plain.df) and torch.equal(sim.pos, plain.pos)
    # the second call looks, the third knows
    assert held[:2] == [False, False] and all(h == (gain > 0) for h in held[2:])
    assert len(looks) == 2 and all(t == 325 and g >= 0 for g, t in looks)


def test_scans_under_capture_take_the_last_answer():
    sim, atoms = simulator(100)
    sim.run(atoms)
    torch.cuda.synchronize()
    want = sim.df.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sim.run(atoms)
        sim.run(atoms)
    sim.df.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(sim.df, want)
