"""The autotuner times z-nodes per thread only where they can change the launch."""
import numpy as np
import pytest

from paper_2401_14564_gb300 import tune


@pytest.mark.parametrize("n,d,interp,min_image,matters", [
    (15, 0.1, 0, 0, True), (35, 0.1, 0, 0, True), (36, 0.1, 0, 0, False), (15, 0.2, 0, 1, True), (16, 0.2, 0, 1, False),
    (500, 0.36, 0, 0, True), (500, 0.36, 0, 1, True), (15, 0.1, 1, 0, False), (500, 0.4, 1, 0, False)])
def test_where_z_nodes_per_thread_matter(n, d, interp, min_image, matters):
    case = {"atoms": {"x": np.zeros(n)}, "grid": {"dx": 0.1, "dy": d, "dz": 0.1, "interp": interp},
            "probe": {"min_image": min_image}}
    assert tune._zpt_matters(case) == matters


def test_the_batch_sweeps_no_knob_without_effect():
    assert [name for name, _ in tune.BATCH_SHAPES] == ["relax_tile_w"]
