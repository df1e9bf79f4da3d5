"""Barriers over a cluster of thread blocks take whole warps (`.aligned`): the sources reach them through one function, which first
brings together the lanes that a test or a loop of their own sent different ways (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_04179_b200", "csrc")


def test_lanes_are_brought_together_before_a_cluster_barrier():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            found += [(name, text[:m.start()]) for m in re.finditer(r"asm volatile\(\"barrier\.cluster", text)]
    assert len(found) == 1, [name for name, _ in found]
    assert re.search(r"void gram_cluster_sync\(\) \{\s*__syncwarp\(\);\s*$", found[0][1])
