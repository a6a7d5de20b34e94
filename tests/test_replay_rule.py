"""The line between the CUDA-core replays and the block replay for codes of few bits (csrc/replay_rule.h) against measured calls of more
units than the 148 SMs: prompts 2.5 times the budget, us on CUDA cores and of the block kernel on clustered, drifting and independent
keys. A shape goes to the kernel that is ahead over the three kinds of keys together."""
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16187_b200", "csrc")
# (bits, group, slots, units): CUDA cores, (block kernel on clustered, drifting, independent keys)
MEASURED = {
    (16, 1, 512, 160): (284, (357, 215, 195)), (16, 1, 512, 320): (362, (518, 333, 305)), (16, 1, 512, 592): (486, (826, 492, 443)),
    (16, 1, 1024, 160): (503, (682, 368, 339)), (16, 1, 1024, 296): (550, (830, 436, 395)), (16, 1, 1024, 320): (632, (976, 571, 524)),
    (16, 1, 1024, 448): (771, (1208, 738, 682)), (16, 1, 1536, 320): (1281, (1849, 731, 614)), (16, 1, 2044, 320): (1595, (2379, 940, 791)),
    (12, 1, 1024, 224): (549, (959, 486, 384)), (12, 1, 1024, 296): (551, (1045, 497, 413)), (12, 1, 1024, 320): (632, (1279, 656, 544)),
    (12, 1, 1536, 160): (1011, (1677, 670, 433)), (12, 1, 1536, 320): (1280, (2545, 957, 677)),
    (8, 1, 1024, 160): (505, (1154, 690, 440)), (8, 1, 1024, 320): (632, (1769, 1023, 676)), (8, 1, 3072, 320): (2953, (7115, 3966, 2067)),
    (8, 4, 3072, 320): (4530, (8945, 6513, 6823)), (8, 2, 1536, 160): (3116, (4153, 3440, 3733)), (8, 2, 2048, 320): (6060, (8539, 6927, 7522)),
    (8, 2, 3072, 320): (12632, (12810, 10539, 11364)), (5, 3, 2048, 320): (6130, (10146, 8149, 6094)),
    (5, 3, 3072, 320): (12764, (16320, 12292, 9276)), (4, 4, 1024, 320): (792, (2731, 2826, 2606)),
}
PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "replay_rule.h"
int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3)
    std::printf("%d ", he::block_replay_min_budget(1, std::atoi(argv[i + 1]), std::atoi(argv[i]), std::atoi(argv[i + 2]), 148));
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", d / "t", d / "t.cpp"], check=True)
    out = subprocess.run([d / "t"] + [str(x) for k in MEASURED for x in (k[0], k[1], k[3])], capture_output=True, text=True, check=True).stdout.split()
    return dict(zip(MEASURED, map(int, out)))


@pytest.mark.parametrize("shape", list(MEASURED))
def test_few_bit_shapes_go_to_the_kernel_that_is_ahead(shape, lines):
    cores, block = MEASURED[shape]
    assert (shape[2] >= lines[shape]) == (math.prod(block) < cores ** 3)
