"""The small levels of the V-cycle as one cluster launch (two around a larger
coarsest solve) against one launch per colour pass on the same hierarchy:
levels from a few rows per block to the shared-memory limit, with one, 8 and 16
blocks, one level and several, the coarsest solve inside and outside, both
precisions.  An explicit launch shape takes a level out of the cluster."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# grid, coarsening target, dimension
CASES = {
    "one_block": ((14, 13), 12, 2),          # a first level of about 45 rows
    "eight_blocks": ((64, 61), 60, 2),       # about 950 rows, three levels
    "sixteen_blocks": ((40, 37, 33), 100, 3),   # about 6,200 rows, coarsest inside
    "solve_outside": ((36, 41, 33), 1000, 3),   # coarsest of more than 256 rows
    "chunks_of_one": ((9, 8, 7), 4, 3),      # fewer rows of a colour than blocks
}


def _gs_launches(solver, b):
    solver.profile(1)
    solver.solve(b, tol=0.0, maxit=1)
    n = sum(d["launches"] for d in solver.profile_read() if d["name"] == "gs_coarse")
    solver.profile(0)
    return n


@pytest.mark.parametrize("precision", [amg.AMG_FP64, amg.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("case", list(CASES))
def test_tail_matches_a_launch_per_pass(case, precision):
    shape, target, dim = CASES[case]
    p = P.lognormal3d(shape, seed=3) if dim == 3 else None
    if p is None:
        K = np.exp(np.random.default_rng(4).standard_normal(shape))
        rp, ci, va, b = P.assemble_fv(K, bc=[(1.0, 0.0), (None, None)])
    else:
        rp, ci, va, b = p.row_ptr, p.col, p.val, p.b
    solver = amg.AMG(rp, ci, va, dim=dim, coarsen_target=target, precision=precision)
    try:
        _, levels = solver.info()
        split = [l for l in range(1, len(levels) - 1) if levels[l]["ncolours"] >= 3]
        if not split or split[-1] != len(levels) - 2:
            pytest.skip("no tail on this hierarchy")
        r = torch.from_numpy(np.random.default_rng(6).standard_normal(len(b))).cuda()
        bd = torch.from_numpy(b).cuda()
        z_tail = [solver.vcycle(r).cpu().numpy() for _ in range(3)]
        assert np.array_equal(z_tail[0], z_tail[1]) and np.array_equal(z_tail[0], z_tail[2])
        x, rc, info = solver.solve(bd, tol=1e-8)
        assert rc == amg.AMG_OK and info["true_rel_residual"] <= 1.05e-8
        with_tail = _gs_launches(solver, bd)
        for l in split:
            solver.set_level_shape(l, 4)
        assert _gs_launches(solver, bd) > with_tail
        z = solver.vcycle(r).cpu().numpy()
        # the V-cycle bar of 1e-12 in float64 is about 1e4 unit roundoffs; the
        # same factor in float32
        tol = 1e-12 if precision == amg.AMG_FP64 else 1e4 * 6e-8
        assert np.abs(z_tail[0] - z).max() <= tol * np.abs(z).max()
        x2, rc, info2 = solver.solve(bd, tol=1e-8)
        assert rc == amg.AMG_OK and abs(info2["iterations"] - info["iterations"]) <= 1
    finally:
        solver.close()
