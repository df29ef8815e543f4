"""The dissected coarsest solve among overlapping launches: V-cycles with and
without launch overlap are the same, bit for bit, whether the level above the
solve runs as launches or in the cluster, in two-level hierarchies too, and in
one launch stream of many cycles."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [amg.AMG_FP64, amg.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("shape", [(27, 26, 25), (50, 50, 50), (61, 47, 70)],
                         ids=["two_levels", "cluster_above_in_float32", "larger_coarsest"])
def test_overlap_changes_nothing(shape, precision):
    p = P.lognormal3d(shape, seed=4)
    rng = np.random.default_rng(1)
    r = [torch.from_numpy(rng.standard_normal(p.n)).cuda() for _ in range(6)]
    out = []
    for overlap in (0, 1):
        s = amg.AMG(p.row_ptr, p.col, p.val, dim=3, precision=precision, launch_overlap=overlap)
        try:
            assert s.info()[1][-1]["n"] >= 2000
            out.append([s.vcycle(v).clone() for v in r + r])
        finally:
            s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    for a, b in zip(out[1][:6], out[1][6:]):
        assert torch.equal(a, b)
