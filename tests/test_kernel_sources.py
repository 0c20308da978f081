"""Rules that every kernel source keeps, checked on the text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2508_06012_gb300", "csrc")


def test_warp_votes_name_their_lanes():
    """A vote or exchange among a warp's lanes is over a mask that the program knows (all
    lanes, or those of the turn): the lanes that __activemask() names after a divergent
    loop are whichever happen to run together."""
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    for f in files:
        with open(f) as fh:
            assert not re.search(r"__activemask\s*\(", fh.read()), os.path.basename(f)


def test_turn_mask_names_the_lanes_that_run_it():
    """The mask of a turn, from the last unit and the lane's own, against the lanes whose
    unit is below the end, in every warp of a strided loop."""
    for first, end, nt in ((0, 1, 32), (0, 31, 32), (0, 33, 64), (5, 300, 128), (96, 1000, 1024),
                           (17, 17, 32), (0, 4099, 1024)):
        for base in range(first, end + nt, 32):
            running = [lane for lane in range(32) if base + lane < end]
            for lane in running:
                s = base + lane
                left = end - (s - lane)
                mask = 0xffffffff if left >= 32 else (1 << left) - 1
                assert mask == sum(1 << q for q in running), (first, end, base, lane)
