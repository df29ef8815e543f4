"""The tuner's cache and the cluster launch of the small levels: a choice timed
with the coarsest solve inside the launch is not replayed, untimed, on a
hierarchy where it is outside; on the same hierarchy it is."""

import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_the_cache_tells_levels_apart_by_the_cluster():
    # the same level 1 of 6,300 rows, above two more levels and a coarsest one of
    # at most 256 rows, and right above a coarsest one of 900
    p = P.lognormal3d((38, 41, 29), variance=6.0, seed=5)
    ms, n = [], []
    for target in (60, 60, 900):
        s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, autotune=1)
        summary, levels = s.info()
        ms.append(summary["autotune_ms"])
        n.append([l["n"] for l in levels])
        s.close()
    assert n[0][:2] == n[2][:2] and n[0][-1] <= 256 < n[2][-1] and len(n[2]) == 3
    assert ms[1] == 0.0 and ms[2] > 0.0
