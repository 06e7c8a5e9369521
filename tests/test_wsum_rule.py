"""Steps per tile of the weighted sum: the rule counts the blocks an SM really holds (no GPU).

The rule is compiled for the host. Its count must be the one the kernel's launch bounds ask for, its
choice the length with the fewest rounds x (steps + 1), and the sizes of the GPU test must reach every length.
"""
import itertools
import os
import re
import shutil
import subprocess

import pytest

from test_gpu_wsum_tiles import CTG, PLAIN, STAGED

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300", "csrc")
LENGTHS = (1, 2, 3, 4, 6, 8)

PROGRAM = r"""
#include <stdio.h>
#include "mppi_internal.h"
int main() {
    for (int tt : {1, 2, 3, 4, 6, 8}) printf("%d %d\n", mppi::wsum_blocks_per_sm(tt, false), mppi::wsum_blocks_per_sm(tt, true));
    int K, T, n_sm, bf16, ctg;
    while (scanf("%d %d %d %d %d", &K, &T, &n_sm, &bf16, &ctg) == 5)
        printf("%d\n", mppi::wsum_tile_steps(K, T, (K + mppi::WSUM_KT - 1) / mppi::WSUM_KT, n_sm, bf16, ctg));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    from paper_2308_01654_gb300 import _build
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    d = tmp_path_factory.mktemp("wsum")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", include, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def run(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows) + "\n"
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return [int(v) for v in out[:12]], [int(v) for v in out[12:]]
    return run


def blocks(tt, bf16, ctg, K):
    """256 threads: 65,536 registers at 40 or 32 a thread; the staged form 32 registers and its tile."""
    if bf16 and not ctg and K % 4 == 0:
        return min(8, (224 * 1024) // (tt * 2048 * 4 + 2048))
    return 65536 // (256 * (40 if ctg or tt == 1 else 32))


def rounds(K, T, n_sm, bf16, ctg, tt):
    tiles, slots = -(-K // 2048) * -(-T // tt), n_sm * blocks(tt, bf16, ctg, K)
    return -(-tiles // slots)


def test_the_count_is_the_launch_bounds(rule):
    src = open(os.path.join(CSRC, "mppi_kernels.cu")).read()
    assert re.search(r"__launch_bounds__\(256, wsum_blocks_per_sm\(TT, CTG\)\) wsum_kernel", src)
    got, _ = rule([])
    assert got == [b for tt in LENGTHS for b in (blocks(tt, 0, 0, 2048), blocks(tt, 0, 1, 2048))]


def test_the_fewest_rounds(rule):
    rows = [(K, T, n_sm, bf16, ctg) for K, T, n_sm, bf16, ctg in itertools.product(
        (1, 2048, 2049, 16384, 43366, 65536, 65538, 131072, 200611, 262144), (1, 2, 12, 50, 77, 100, 200, 256, 1024),
        (148, 152, 160), (0, 1), (0, 1))]
    _, got = rule(rows)
    for (K, T, n_sm, bf16, ctg), tt in zip(rows, got):
        cost = {t: rounds(K, T, n_sm, bf16, ctg, t) * (t + 1) for t in LENGTHS}
        assert tt == max(t for t in LENGTHS if cost[t] == min(cost.values()))


def test_the_gpu_cases_reach_every_length(rule):
    for cases, bf16, ctg, want in ((PLAIN, 0, 0, LENGTHS), ([(K + 2, T) for K, T in PLAIN], 1, 0, LENGTHS),
                                   (STAGED, 1, 0, (1, 2, 3, 4)), (CTG, 0, 1, (4, 6, 8))):
        _, got = rule([(K, T, 152, bf16, ctg) for K, T in cases])
        assert set(want) <= set(got), (bf16, ctg, got)


def test_the_staged_form_has_no_longer_tile(rule):
    """Tiles of 6 and 8 steps hold no more steps an SM than tiles of 3 and cost more: never chosen."""
    rows = [(K, T, n_sm, 1, 0) for K in list(range(4, 40000, 1020)) + list(range(40000, 700000, 8188))
            for T in range(1, 1025, 7) for n_sm in (148, 152, 160)]
    _, got = rule(rows)
    assert max(got) <= 4
