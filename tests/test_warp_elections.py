"""Elections of a lane (tc_elect: elect.sync over all 32) stand where the whole warp arrives: a flag that other warps raise
meanwhile is voted on first, never read by each lane for itself in the same condition."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16187_b200", "csrc")


def test_no_election_behind_a_flag_read_lane_by_lane():
    elections = 0
    for path in glob.glob(os.path.join(CSRC, "*.cuh")):
        for number, line in enumerate(open(path), 1):
            code = line.split("//")[0]
            if "tc_elect()" not in code or "bool tc_elect" in code:
                continue
            elections += 1
            assert not re.search(r"\babort_flag\b", code), f"{os.path.basename(path)}:{number}: {code.strip()}"
    assert elections > 0
