"""Lanes per row of split coarse levels: eight where the rows are long or few,
fewer as the level grows, by the rule's two lines; and the V-cycle on a 27-point
stencil, whose coarse rows are about twice as long as a 7-point one's, against
the oracle's."""

import itertools

import numpy as np
import pytest

from conftest import coo_to_csr
from oracle import oracle as O
from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _stencil27(m, seed):
    """Weighted graph Laplacian of an m^3 grid with all 26 neighbours, SPD by a
    shift on one face."""
    rng = np.random.default_rng(seed)
    idx = np.arange(m ** 3).reshape(m, m, m)
    pairs = []
    for off in itertools.product((-1, 0, 1), repeat=3):
        if off > (0, 0, 0):
            lo = tuple(slice(max(0, -o), m - max(0, o)) for o in off)
            hi = tuple(slice(max(0, o), m - max(0, -o)) for o in off)
            pairs.append((idx[lo].ravel(), idx[hi].ravel()))
    i, j = (np.concatenate(v) for v in zip(*pairs))
    w = np.exp(rng.standard_normal(len(i)))
    d = np.zeros(m ** 3)
    np.add.at(d, i, w)
    np.add.at(d, j, w)
    d[idx[0].ravel()] += 1.0
    k = np.arange(m ** 3)
    return coo_to_csr(m ** 3, np.concatenate([i, j, k]), np.concatenate([j, i, k]),
                      np.concatenate([-w, -w, d]))


@pytest.mark.parametrize("kind", ["seven", "twentyseven"])
def test_lanes_of_a_level_of_some_25000_rows(kind):
    if kind == "seven":
        p = P.lognormal3d((58, 58, 58), seed=2)
        A = (p.row_ptr, p.col, p.val)
    else:
        A = _stencil27(57, seed=2)
    solver = amg.AMG(*A, dim=3)
    try:
        lev = solver.info()[1]
        mean = lev[1]["nnz"] / lev[1]["n"] - 1
        assert 20_000 < lev[1]["n"] < 30_000 and (mean > 16) == (kind == "twentyseven")
        assert (lev[1]["lanes_per_row"], lev[1]["threads_per_block"]) == (8, 128)
        r = np.random.default_rng(3).standard_normal(solver.n)
        z = solver.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        ref = O.Hierarchy(*A, O.default_params(3)).vcycle(r)
        assert np.abs(z - ref).max() <= 1e-12 * np.abs(ref).max()
    finally:
        solver.close()
