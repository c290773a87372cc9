"""Which batch entries share a tensor-core tile (csrc/merge.h), compiled with the host compiler: a batched launch is
merged where that leaves every SM work and takes items away, and is left to the plan's tile variant otherwise."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_05540_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "merge.h"
int main(int argc, char** argv) {
    int first[heff::MERGE_CLASSES + 1] = {0};            // tasks of each class
    for (int c = 0; c < heff::MERGE_CLASSES; ++c) first[c + 1] = first[c] + std::atoi(argv[3 + c]);
    const int nb = std::atoi(argv[1]), cap = heff::merge_cap(first, nb, std::atoi(argv[2]));
    std::printf("%d %ld\n", cap, heff::merge_items(first, nb, cap).item0[heff::MERGE_CLASSES]);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("merge")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return lambda nb, sms, *classes: tuple(map(int, subprocess.run(
        [str(exe), str(nb), str(sms), *map(str, classes)], capture_output=True, text=True, check=True).stdout.split()))


@pytest.mark.parametrize("nb", [2, 16, 64])
def test_blocks_too_wide_to_share_a_tile_are_not_merged(rule, nb):
    assert rule(nb, 152, 1000, 0, 0, 0, 0, 0) == (0, 1000 * nb)
    assert rule(nb, 152, 1000, 20, 0, 0, 0, 0)[0] == 0            # a few that are not: no tenth of the items


def test_small_blocks_are_merged_as_far_as_every_sm_has_two_items(rule):
    assert rule(16, 152, 0, 0, 0, 400, 0, 0) == (3, 800)          # eight to a tile
    assert rule(16, 152, 0, 0, 0, 80, 0, 0) == (2, 320)           # four: two items an SM
    assert rule(16, 152, 0, 0, 0, 30, 0, 0)[0] == 0               # 480 items at best unmerged
    assert rule(1, 152, 0, 0, 0, 400, 0, 0)[0] == 0


def test_the_rest_of_a_batch_takes_an_item(rule):
    assert rule(9, 152, 0, 0, 0, 400, 0, 0) == (3, 800)
    assert rule(7, 152, 100, 300, 0, 0, 200, 0) == (3, 100 * 7 + 300 * 4 + 200 * 4)
