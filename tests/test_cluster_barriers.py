"""The aligned cluster barriers want whole warps.  What the compiler does with
lanes that leave a loop at different steps shows on no output, so this reads
the source: the barrier's two halves exist once, in wrappers whose first
statement brings the warp together, and nothing else issues them."""

import glob
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1209_0960_gb300", "csrc")


def test_every_cluster_barrier_meets_its_warp_first():
    found = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"asm volatile\(\"barrier\.cluster\.(\w+)", text):
            before = text[text.rindex("{", 0, m.start()) + 1:m.start()]
            assert before.strip() == "__syncwarp();", f
            found.append((os.path.basename(f), m.group(1)))
    assert found == [("device_util.cuh", "arrive"), ("device_util.cuh", "wait")]
