"""The kernels that run as thread-block clusters (the small levels, the CG work of
small systems) on a device that holds no such cluster, or only smaller ones: the
same calls run as ordinary launches.  The checked build answers for such a
device when it is told to; in a child process, as test_gpu_checked_build.py."""

import json
import os
import subprocess
import sys

import pytest

from conftest import ROOT
from paper_1209_0960_gb300 import amg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHILD = r"""
import json, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
from paper_1209_0960_gb300 import amg, problems as P
assert amg.lib().amg_device_checks() == 1
out = []
# a first coarse level of 1,265 rows (8 blocks) and one of 6,338 (16 blocks)
for shape, target in (((21, 19, 23), 40), ((38, 41, 29), 60)):
    p = P.lognormal3d(shape, variance=6.0, seed=5)
    b = torch.from_numpy(p.b).cuda()
    for limit in (16, 8, 0):
        assert amg.lib().amg_debug_cluster_limit(limit) == amg.AMG_OK
        for tune in (0, 1):
            for prec in (amg.AMG_FP64, amg.AMG_FP32_IN_FP64):
                s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, precision=prec,
                            autotune=tune)
                x, rc, info = s.solve(b, tol=1e-8, maxit=100)
                s.profile(1)
                s.solve(b, tol=0.0, maxit=1)
                n = {d["name"]: d["launches"] for d in s.profile_read()}
                s.profile(0)
                out.append([p.n, limit, tune, rc, info["iterations"], n.get("gs_coarse", 0),
                            "cg_update_dot" in n, x.cpu().numpy().tolist()[:3]])
                s.close()
assert amg.lib().amg_debug_cluster_limit(17) == amg.AMG_EINVAL
print("RESULT " + json.dumps(out))
"""


def test_without_clusters_the_calls_run_as_launches():
    from paper_1209_0960_gb300 import build as B
    B.build(checked=True)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True,
                       env=dict(os.environ, AMG_LIB="checked"), timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    line = [l for l in r.stdout.splitlines() if l.startswith("RESULT ")][-1]
    its = {}
    for n, limit, tune, rc, iters, coarse, five_launches, x in json.loads(line[len("RESULT "):]):
        assert rc == amg.AMG_OK
        its.setdefault(n, set()).add(iters)
        # the CG work is a cluster of 16 blocks up to 24,576 rows
        assert five_launches == (limit < 16 or n > 24576)
        if limit == 0:
            assert coarse > 20   # every colour pass of every coarse level a launch
        elif limit == 16 and not tune:
            assert coarse == 0   # all of them in the cluster
    for v in its.values():
        assert max(v) - min(v) <= 1


def test_the_regular_build_refuses_the_limit():
    assert amg.lib().amg_debug_cluster_limit(8) == amg.AMG_EINVAL
