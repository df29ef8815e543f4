"""The checked build on levels that run in the cluster launch, whose columns are
packed with 16 bits: an index outside its level is reported by every solve that
meets it, also where its low 16 bits lie inside the level, in both precisions.
In a child process, as test_gpu_checked_build.py."""

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
import torch
sys.path.insert(0, sys.argv[1])
from paper_1209_0960_gb300 import amg, problems as P
assert amg.lib().amg_device_checks() == 1
out = {}
p = P.lognormal3d((21, 19, 23), variance=6.0, seed=5)
b = torch.from_numpy(p.b).cuda()
for prec in (amg.AMG_FP64, amg.AMG_FP32_IN_FP64):
    s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=40, precision=prec)
    res = [s.solve(b, tol=1e-8, maxit=50)[1]]
    s.profile(1)
    s.solve(b, tol=0.0, maxit=1)
    names = [d["name"] for d in s.profile_read()]
    s.profile(0)
    n1 = s.info()[1][1]["n"]
    for col in (65536 + 7, n1 + 65536, 2**30 + 5):
        assert amg.lib().amg_debug_set_column(s.ctx, 1, 5, 0, col) == amg.AMG_OK
        for _ in range(2):
            res.append(s.solve(b, tol=1e-8, maxit=50)[1])
    out[prec] = [names, res]
    s.close()
print("RESULT " + json.dumps(out))
"""


def test_an_index_past_16_bits_is_reported():
    from paper_1209_0960_gb300 import build as B
    B.build(checked=True)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True,
                       env=dict(os.environ, AMG_LIB="checked"), timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    line = [l for l in r.stdout.splitlines() if l.startswith("RESULT ")][-1]
    for names, res in json.loads(line[len("RESULT "):]).values():
        assert "gs_coarse" not in names   # every coarse level is in the launch
        assert res == [amg.AMG_OK] + 6 * [amg.AMG_ERANGE]
