"""The cluster barriers take whole warps: wherever the instruction stands, __syncwarp() stands in front of it (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23815_b200", "csrc")


def test_every_aligned_cluster_barrier_follows_a_warp_barrier():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        lines = [re.sub(r"//.*", "", x).strip() for x in open(os.path.join(CSRC, name))]
        lines = [x for x in lines if x]
        for before, line in zip(lines, lines[1:]):
            if re.search(r"barrier\.cluster\.(arrive|wait)\S*\.aligned", line):
                seen += 1
                assert before == "__syncwarp();", f"{name}: {line}"
    assert seen == 2                            # the two helpers that every kernel goes through
