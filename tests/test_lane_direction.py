"""The axis the circles are sorted on is formed in binary64 and rounded once (no GPU).

The function is compiled for the host and compared with the direction in exact decimal arithmetic: each
component within half a unit in the last place of binary32, plus what binary64 can add before the
rounding (a few 2^-53 relative).
"""
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "mppi_iter.cuh"
int main() {
    double ref[4];
    while (scanf("%lf %lf %lf %lf", ref, ref + 1, ref + 2, ref + 3) == 4) {
        const float2 d = mppi::lane_direction(ref, 2);
        printf("%a %a\n", (double)d.x, (double)d.y);
    }
}
"""


@pytest.fixture(scope="module")
def directions(tmp_path_factory):
    from paper_2308_01654_gb300 import _build
    d = tmp_path_factory.mktemp("lane_direction")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O1", "-std=c++17", "-I", CSRC, "-I", _build.INCLUDE, "-o",
                    str(d / "t"), str(d / "t.cu")], check=True, capture_output=True)

    def run(rows):
        text = "\n".join(" ".join(repr(float(v)) for v in r) for r in rows) + "\n"
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return np.array([float.fromhex(v) for v in out]).reshape(-1, 2)
    return run


def test_rounded_once(directions):
    rng = np.random.default_rng(7)
    n = 2000
    at = rng.uniform(-1e4, 1e4, (n, 2))
    ang, length = rng.uniform(-np.pi, np.pi, n), np.exp(rng.uniform(np.log(1e-2), np.log(1e4), n))
    rows = np.concatenate([at, at + length[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1)], 1)
    got = directions(rows)
    getcontext().prec = 40
    for r, g in zip(rows, got):
        ex, ey = Decimal(float(r[2] - r[0])), Decimal(float(r[3] - r[1]))      # as binary64 forms them
        m = (ex * ex + ey * ey).sqrt()
        for e, v in ((ex / m, g[0]), (ey / m, g[1])):
            ulp = np.spacing(np.float32(abs(float(e))))
            assert abs(Decimal(float(v)) - e) <= Decimal(float(ulp)) / 2 + abs(e) * Decimal(2.0 ** -50)


def test_no_direction(directions):
    got = directions([[3.0, 4.0, 3.0, 4.0], [0.0, 0.0, 0.0, -2.0], [0.0, 0.0, 1e-30, 0.0]])
    np.testing.assert_array_equal(got, [[1.0, 0.0], [0.0, -1.0], [1.0, 0.0]])
