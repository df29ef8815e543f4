"""The cluster launch of the small levels: every block holds the same values.

The blocks keep copies of the rows they read, so a value that differs between
copies shows up as a V-cycle that differs from run to run, or from one launch
per colour pass.  Hierarchies in which a block's rows do not fill its warps (the
last warp's lanes leave the loops over own rows at different steps), with one, 8
and 16 blocks, the coarsest solve inside the launch and outside, in both
precisions; many V-cycles on each, bit for bit."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# grid, coarsening target
CASES = {
    "one_block": ((9, 11, 7), 12),
    "eight_blocks": ((21, 19, 23), 40),
    "sixteen_blocks": ((38, 41, 29), 60),
    "solve_outside": ((37, 40, 35), 1000),
}


@pytest.mark.parametrize("precision", [amg.AMG_FP64, amg.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("case", list(CASES))
def test_every_cycle_is_the_same(case, precision):
    shape, target = CASES[case]
    p = P.lognormal3d(shape, variance=6.0, seed=5)
    solver = amg.AMG(p.row_ptr, p.col, p.val, dim=3, coarsen_target=target, precision=precision)
    try:
        _, levels = solver.info()
        assert len(levels) >= 3 and all(l["ncolours"] >= 3 for l in levels[1:-1])
        r = torch.from_numpy(np.random.default_rng(8).standard_normal(p.n)).cuda()
        z0 = solver.vcycle(r).clone()
        for _ in range(200):
            assert torch.equal(solver.vcycle(r), z0)
        for l in range(1, len(levels) - 1):
            solver.set_level_shape(l, 4)   # a launch per colour pass
        z = solver.vcycle(r)
        # 1e-12 in float64 is about 1e4 unit roundoffs; the same factor in float32
        tol = 1e-12 if precision == amg.AMG_FP64 else 1e4 * 6e-8
        assert (z - z0).abs().max() <= tol * z.abs().max()
    finally:
        solver.close()
