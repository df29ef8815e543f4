"""amg_vcycle launches its kernels one by one on a context's first call and
replays them as one graph afterwards (V-cycles of 40 launches and more): the
same bits on every call and for every input, in both precisions, after a change
of shapes, and inside a stream capture of the caller's, where it launches
directly."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def problem():
    return P.lognormal3d((60, 58, 55), seed=5)


def _inputs(n):
    rng = np.random.default_rng(2)
    return [torch.from_numpy(rng.standard_normal(n)).cuda() for _ in range(2)]


@pytest.mark.parametrize("precision", [amg.AMG_FP64, amg.AMG_FP32_IN_FP64])
def test_graph_replays_give_the_direct_launches_bits(problem, precision):
    p = problem
    rs = _inputs(p.n)
    solver = amg.AMG(p.row_ptr, p.col, p.val, dim=3, precision=precision)
    try:
        for shape in (None, 4):
            if shape is not None:
                solver.set_level_shape(1, shape)   # drops the graph: direct again
            # 4 colours' worth of launches per level and more: the graph is used
            assert sum(4 * l["ncolours"] + 1 for l in solver.info()[1][:2]) >= 40
            direct = solver.vcycle(rs[0]).clone()
            for _ in range(3):
                # back to back, other inputs and outputs in between, no waits
                other = solver.vcycle(rs[1])
                again = solver.vcycle(rs[0])
            torch.cuda.synchronize()
            assert torch.equal(again, direct)
            assert not torch.equal(other, direct)
    finally:
        solver.close()


def test_vcycle_inside_a_capture(problem):
    p = problem
    rs = _inputs(p.n)
    s = torch.cuda.Stream()
    solver = amg.AMG(p.row_ptr, p.col, p.val, dim=3, stream=s)
    try:
        with torch.cuda.stream(s):
            r = rs[0].clone()
            want = [solver.vcycle(x).clone() for x in (rs[0], rs[1], rs[0])]
            z = torch.empty_like(r)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            solver.vcycle(r, z)
        for k in (1, 0):
            r.copy_(rs[k])
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(z, want[k])
    finally:
        solver.close()
