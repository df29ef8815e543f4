"""The tuner's cache and the cluster launch of the small levels: a choice timed
with the coarsest solve inside the launch is not replayed, untimed, on a
hierarchy where it is outside; on the same hierarchy it is.  In a child process,
whose cache is empty at first."""

import json
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHILD = r"""
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_1209_0960_gb300 import amg, problems as P
# the same level 1 of 6,300 rows, above two more levels and a coarsest one of
# at most 256 rows, and right above a coarsest one of 900
p = P.lognormal3d((38, 41, 29), variance=6.0, seed=5)
out = []
for target in (60, 60, 900):
    s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, autotune=1)
    summary, levels = s.info()
    out.append([summary["autotune_ms"], [l["n"] for l in levels]])
    s.close()
print("RESULT " + json.dumps(out))
"""


def test_the_cache_tells_levels_apart_by_the_cluster():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    line = [l for l in r.stdout.splitlines() if l.startswith("RESULT ")][-1]
    ms, n = zip(*json.loads(line[len("RESULT "):]))
    assert n[0][:2] == n[2][:2] and n[0][-1] <= 256 < n[2][-1] and len(n[2]) == 3
    assert ms[0] > 0.0 and ms[1] == 0.0 and ms[2] > 0.0
