"""Layout of the FFT path's scratch for every accepted size, 2 to 1024 per axis, on the host alone.

The header that the launcher uses is compiled with the host compiler: every array starts and ends inside the
workspace, arrays that live at the same time do not overlap, and offsets inside an array fit 32 bits."""
import itertools
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2401_14564_gb300", "csrc")
SIZES = [2 ** k for k in range(1, 11)]
PROGRAM = """
#include <cstdio>
#include "fft_layout.cuh"
int main() {
    for (int nx = 2; nx <= 1024; nx *= 2) for (int ny = 2; ny <= 1024; ny *= 2) for (int nz = 2; nz <= 1024; nz *= 2) {
        const pp::FftLayout L = pp::fft_layout(nx, ny, nz);
        const long long v[] = {nx, ny, nz, L.px, L.pz, L.hx, L.hz, L.zlen, L.hlen, L.a, L.b, L.c, L.d, L.e, L.size};
        for (long long x : v) printf("%lld ", x);
        printf("\\n");
    }
}
"""


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    d = tmp_path_factory.mktemp("fft_layout")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)
    rows = subprocess.run([str(d / "p")], check=True, capture_output=True, text=True).stdout.split("\n")
    return {tuple(v[:3]): v[3:] for v in (list(map(int, r.split())) for r in rows if r)}


def test_every_array_lies_inside_the_workspace_and_apart_from_the_live_ones(layouts):
    assert sorted(layouts) == sorted(itertools.product(SIZES, repeat=3))
    for (nx, ny, nz), (px, pz, hx, hz, zlen, hlen, a, b, c, d, e, size) in layouts.items():
        shape = (nx, ny, nz)
        # rows, planes and arrays hold what they are indexed with
        assert px >= nx and pz >= px * (ny - 1) + nx and zlen >= pz * (nz - 1) + px * (ny - 1) + nx, shape
        assert hx >= nx // 2 + 1 and hz >= hx * ny and hlen >= hz * nz, shape
        assert zlen <= np.iinfo(np.int32).max and hlen <= np.iinfo(np.int32).max, shape
        assert size == 3 * (((nx + 16) * ny + 16) * nz), shape
        for first in (a, b, c, d, e):
            assert 0 <= first <= size - hlen, (shape, first)
        # z with a and b (z kernel); a and b with c, d and e (y kernel)
        assert zlen <= a and a + hlen <= b, shape
        assert c + hlen <= d and d + hlen <= e and e + hlen <= a, shape
