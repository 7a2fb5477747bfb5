"""K1 by tiles on atoms that no sample has but the entry points take: R_i + R_PP below zero, whose core floor and
pair terms reach as far as those of its magnitude, and an infinite coordinate, which adds nothing to the energies."""
import numpy as np
import pytest
import torch

from helpers import ff_rel_err, linear_ff
from test_gpu_ff_tiles import build, case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [-12.0, 8.0])
def test_a_wide_core_of_either_sign_matches_direct_sums(R):
    # against the sum of grids of ten atoms each, which are assembled directly (the per-node bar of test_gpu_ff_tiles.py)
    c = case(40, (49, 35, 41), 0.1, "plain")
    c["probe"]["core_frac"] = 0.9
    c["atoms"]["R"] = np.array(c["atoms"]["R"])
    c["atoms"]["R"][5] = R
    ff, _ = build(c)
    ref = 0.0
    for a in range(0, 40, 10):
        part, _ = build(dict(c, atoms={k: np.asarray(v)[a:a + 10] for k, v in c["atoms"].items()}))
        ref = ref + linear_ff(part.cpu().numpy(), c["grid"])
    assert ff_rel_err(linear_ff(ff.cpu().numpy(), c["grid"]), ref).max() <= 1e-4


@pytest.mark.parametrize("key", ["x", "z"])
def test_an_infinite_coordinate_adds_nothing_to_the_energies(key):
    c = case(40, (33, 17, 20), 0.1, "plain")
    c["grid"]["interp"] = 1
    want, _ = build(c)
    c["atoms"] = {k: np.append(v, v[:1]) for k, v in c["atoms"].items()}
    c["atoms"][key][-1] = np.inf
    got, _ = build(c)
    assert torch.isfinite(got).all() and torch.equal(got, want)
