"""Which levels run in the cluster launch without tuning: up to 7,000 rows, and in
float32 larger ones of long rows; the V-cycle either way against the oracle's."""

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


@pytest.mark.parametrize("kind,m,rows,cluster", [
    ("seven", 36, 6_000, (1, 1)), ("seven", 45, 11_800, (0, 0)), ("twentyseven", 40, 8_800, (0, 1))])
def test_levels_by_rows_and_their_length(kind, m, rows, cluster):
    if kind == "seven":
        p = P.lognormal3d((m, m, m), seed=0)
        A = (p.row_ptr, p.col, p.val)
    else:
        A = _stencil27(m, seed=0)
    r = np.random.default_rng(3).standard_normal(m ** 3)
    ref = O.Hierarchy(*A, O.default_params(3)).vcycle(r)
    solver = amg.AMG(*A, dim=3, coarsen_target=5000)
    try:
        for prec in (amg.AMG_FP64, amg.AMG_FP32_IN_FP64):
            solver.set_precision(prec)
            lev = solver.info()[1]
            assert len(lev) == 3 and abs(lev[1]["n"] - rows) < 0.05 * rows
            assert lev[1]["cluster"] == cluster[prec]
            z = solver.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
            # the V-cycle bar of 1e-12 in float64 is about 1e4 unit roundoffs; the
            # same factor in float32
            tol = 1e-12 if prec == amg.AMG_FP64 else 1e4 * 6e-8
            assert np.abs(z - ref).max() <= tol * np.abs(ref).max()
    finally:
        solver.close()
