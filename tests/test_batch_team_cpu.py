"""The team size of a batch (heom_team.h), compiled for the host: sizes whose teams cannot be resident are not picked,
and the packing counts the teams that the GPU really holds."""
import os
import subprocess

import pytest

from paper_1012_4382_gb300 import build as heom_build

MAIN = """
#include <cstdio>
#include <cstdlib>
#include "heom_team.h"
int main(int argc, char** argv) {
  int resident[5];
  for (int i = 0; i < 5; ++i) resident[i] = atoi(argv[2 + i]);
  std::vector<int64_t> blocks;
  for (int i = 7; i < argc; ++i) blocks.push_back(atoi(argv[i]));
  printf("%d", heom::pick_team(blocks, atof(argv[1]), resident));
}
"""
GPU = [152, 76, 36, 15, 7]  # 152 SMs
IDEAL = [152, 76, 38, 19, 9]


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    d = tmp_path_factory.mktemp("team")
    (d / "team.cpp").write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + heom_build.CSRC, str(d / "team.cpp"), "-o", str(d / "team")],
                   check=True)

    def run(m, resident, blocks):
        return int(subprocess.run([str(d / "team"), str(m)] + [str(x) for x in resident + blocks],
                                  capture_output=True, text=True, check=True).stdout)

    return run


def test_sizes_that_cannot_be_resident_are_not_picked(pick):
    few = [100] * 4  # so large teams are best
    assert pick(8.1, GPU, few) == 16
    assert pick(8.1, [152, 76, 36, 15, 0], few) == 8
    assert pick(8.1, [152, 76, 0, 0, 0], few) == 2
    assert pick(8.1, [0, 0, 36, 0, 0], few) == 4
    assert pick(8.1, [1, 0, 0, 0, 0], few) == 1
    assert pick(8.1, [0, 0, 0, 0, 0], few) == 1


def test_packing_counts_the_teams_that_exist(pick):
    # FP64, seven sites, depths 3 to 6 (4, 11, 25 and 54 blocks), six of each: 240 us a step with 8 CTAs, 305 with 16
    blocks = [4, 11, 25, 54] * 6
    assert pick(8.1, GPU, blocks) == 8
    assert pick(8.1, IDEAL, blocks) == 16


def test_small_hierarchies_stay_in_one_cta(pick):
    # mixed precision; m as for three, four and seven sites (us per step with one CTA and the best cluster)
    assert pick(0.0625, GPU, [2] * 5) == 1  # 4.4, 6.9
    assert pick(0.0625, GPU, [2] * 64) == 1  # 4.6, 7.5
    assert pick(0.128, GPU, [3] * 24) == 1  # 5.1, 7.3
    assert pick(0.128, GPU, [7] * 24) == 4  # 8.3, 7.4
    assert pick(0.52, GPU, [4] * 5) in (2, 4)


def test_every_batch_picks_a_size_that_exists(pick):
    for n in (1, 3, 17, 300):
        for b in (1, 2, 7, 60, 400):
            for m in (0.02, 0.52, 12.0):
                assert pick(m, [152, 76, 36, 15, 0], [b] * n) in (1, 2, 4, 8)
