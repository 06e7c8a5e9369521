"""The axis the circles are sorted on is exact (no GPU).

The function is compiled for the host: the coordinate axis nearest to the lane's direction, whatever the
coordinates.
"""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "mppi_iter.cuh"
int main() {
    double ref[4];
    while (scanf("%lf %lf %lf %lf", ref, ref + 1, ref + 2, ref + 3) == 4) {
        const float2 d = mppi::circle_axis(ref, 2);
        printf("%a %a\n", d.x, d.y);
    }
}
"""


@pytest.fixture(scope="module")
def axes(tmp_path_factory):
    from paper_2308_01654_gb300 import _build
    d = tmp_path_factory.mktemp("circle_axis")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O1", "-std=c++17", "-I", CSRC, "-I", _build.INCLUDE, "-o",
                    str(d / "t"), str(d / "t.cu")], check=True, capture_output=True)

    def run(rows):
        text = "\n".join(" ".join(repr(float(v)) for v in r) for r in rows) + "\n"
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return np.array([float.fromhex(v) for v in out]).reshape(-1, 2)
    return run


def test_the_nearest_axis(axes):
    rng = np.random.default_rng(7)
    at = rng.uniform(-1e4, 1e4, (500, 2))
    e = np.exp(rng.uniform(-5.0, 9.0, (500, 1))) * rng.normal(size=(500, 2))
    rows = np.concatenate([at, at + e], 1)
    d = np.abs(rows[:, 2:] - rows[:, :2])
    np.testing.assert_array_equal(axes(rows), np.where((d[:, 0] >= d[:, 1])[:, None], [1.0, 0.0], [0.0, 1.0]))


def test_ties_and_extremes(axes):
    rows = [[1, 2, 4, 5], [3, 4, 3, 4], [0, 0, 0, -2], [0, 0, -1e-300, 0], [-1e308, 0, 1e308, 5], [0, -1e308, 3, 1e308]]
    np.testing.assert_array_equal(axes(rows), [[1, 0], [1, 0], [0, 1], [1, 0], [1, 0], [0, 1]])
