"""The launch-shape syntax for levels in the cluster launch of the small levels:
reported with the suffix t and read back as AMG_SHAPE_CLUSTER."""

import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_1209_0960_gb300 import amg


def test_levels_in_the_cluster_round_trip():
    def level(lanes, threads, sweep, carveout, cluster):
        return {"lanes_per_row": lanes, "threads_per_block": threads, "sweep": sweep,
                "carveout": carveout, "cluster": cluster}
    levels = [level(0, 256, 0, -1, 0), level(2, 128, 0, -1, 0), level(8, 128, 0, -1, 1),
              level(0, 256, 0, 58, 1), level(0, 0, 0, -1, 0)]
    text = bench.shape_string(levels)
    assert text == "0,2h,8ht,0tc58"
    assert bench.parse_lanes(text) == [(0, 0, None), (2, 128, None),
                                       (8 | amg.AMG_SHAPE_CLUSTER, 128, None),
                                       (amg.AMG_SHAPE_CLUSTER, 0, 58)]
