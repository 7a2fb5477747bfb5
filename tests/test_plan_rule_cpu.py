"""When a pixel-to-warp plan pays: more spread is asked of larger scans."""
import pytest

from paper_2401_14564_gb300 import afm


@pytest.mark.parametrize("tiles", [152, 528, 1215])
def test_the_line_grows_with_the_scan(tiles):
    line = 100 + tiles / 26
    assert afm.Simulator.plan_pays(line, tiles) and not afm.Simulator.plan_pays(line - 1, tiles)
    assert not afm.Simulator.plan_pays(line, tiles + 26)
