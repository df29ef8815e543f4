"""Launch shapes round-trip: the shapes a context reports, set on another one,
select the same kernels, with the small levels in the cluster or out of it, by
the rules and by the tuner."""

import numpy as np
import pytest

import bench
from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _launches(solver, b):
    solver.profile(1)
    solver.solve(b, tol=0.0, maxit=1)
    n = {d["name"]: d["launches"] for d in solver.profile_read()}
    solver.profile(0)
    return n


def _shapes(solver):
    return [[l[k] for k in ("lanes_per_row", "threads_per_block", "sweep", "carveout", "cluster")]
            for l in solver.info()[1]]


@pytest.mark.parametrize("precision", [amg.AMG_FP64, amg.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("autotune", [0, 1])
@pytest.mark.parametrize("shape,target", [((21, 19, 23), 40), ((37, 40, 35), 1000)],
                         ids=["solve_inside", "solve_outside"])
def test_reported_shapes_select_the_same_kernels(shape, target, autotune, precision):
    p = P.lognormal3d(shape, variance=6.0, seed=5)
    r = torch.from_numpy(np.random.default_rng(2).standard_normal(p.n)).cuda()
    a = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, precision=precision,
                autotune=autotune)
    b = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, precision=precision)
    try:
        lev = a.info()[1]
        if not autotune:
            assert [l["cluster"] for l in lev] == [0] + [1] * (len(lev) - 2) + [0]
        for l in range(len(lev) - 1):   # out of the cluster first
            b.set_level_shape(l, 4 if lev[l]["ncolours"] >= 3 else 0)
        assert not any(l["cluster"] for l in b.info()[1])
        for l, (lanes, threads, carve) in enumerate(bench.parse_lanes(bench.shape_string(lev))):
            b.set_level_shape(l, lanes, threads)
            if carve is not None:
                b.set_level_carveout(l, carve)
        assert _shapes(a) == _shapes(b)
        assert torch.equal(a.vcycle(r), b.vcycle(r))
        assert _launches(a, r) == _launches(b, r)
    finally:
        a.close()
        b.close()


def test_a_level_leaves_and_joins_the_cluster():
    p = P.lognormal3d((38, 41, 29), variance=6.0, seed=5)
    s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=60)
    try:
        n = len(s.info()[1])
        cl = lambda: [l["cluster"] for l in s.info()[1]]
        assert cl() == [0] + [1] * (n - 2) + [0]
        s.set_level_shape(2, 8)   # the level and those above it
        assert cl() == [0, 0, 0] + [1] * (n - 4) + [0]
        s.set_level_shape(1, 8 | amg.AMG_SHAPE_CLUSTER, 128)   # not while one below is out
        assert cl() == [0, 0, 0] + [1] * (n - 4) + [0]
        s.set_level_shape(2, 8 | amg.AMG_SHAPE_CLUSTER, 128)
        assert cl() == [0] + [1] * (n - 2) + [0]
        for bad in (8 | amg.AMG_SHAPE_CLUSTER | amg.AMG_SHAPE_SWEEP, 3 | amg.AMG_SHAPE_CLUSTER):
            with pytest.raises(amg.AmgError):
                s.set_level_shape(1, bad)
        with pytest.raises(amg.AmgError):   # level 0 has two colours
            s.set_level_shape(0, 4 | amg.AMG_SHAPE_CLUSTER)
    finally:
        s.close()

