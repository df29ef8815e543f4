"""The dissected coarsest solve (levels solved directly that have 2,000 rows or
more) against a dense solve: grids whose parts and separators have odd sizes, a
long thin graph with separators of one row, two components, a graph with no
small separator (which keeps the dense inverse), and the limit of 2,000 rows."""

import numpy as np
import pytest
import scipy.sparse as sp

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _spd(pattern, rng):
    """Random weights on a symmetric pattern, diagonally dominant."""
    U = sp.triu(pattern, 1).tocoo()
    w = -(0.5 + rng.random(U.nnz))
    A = sp.coo_matrix((w, (U.row, U.col)), shape=pattern.shape)
    A = (A + A.T).tocsr()
    return (A + sp.diags(-np.asarray(A.sum(axis=1)).ravel() + 0.05 + rng.random(A.shape[0]))).tocsr()


def _grid(shape):
    rp, ci, va = P.grid_laplacian(shape)
    return sp.csr_matrix((np.abs(va), ci, rp))


def _random_graph(n, degree, rng):
    i = np.repeat(np.arange(n), degree)
    j = rng.integers(0, n, size=i.size)
    A = sp.coo_matrix((np.ones(i.size), (i, j)), shape=(n, n))
    return (A + A.T + sp.eye(n)).tocsr()


CASES = {
    "grid3d_2028": lambda rng: _grid((12, 13, 13)),
    "grid3d_2000": lambda rng: _grid((10, 10, 20)),
    "grid2d_2809": lambda rng: _grid((53, 53)),
    "chain_2100": lambda rng: _grid((2100,)),
    "two_components": lambda rng: sp.block_diag([_grid((11, 11, 11)), _grid((31, 33))]).tocsr(),
    "random_2200": lambda rng: _random_graph(2200, 6, rng),
    "below_1999": lambda rng: _grid((1999,)),
}


@pytest.mark.parametrize("case", list(CASES))
def test_dissected_solve_matches_dense(case):
    rng = np.random.default_rng(8)
    A = _spd(CASES[case](rng), rng)
    A.sort_indices()
    n = A.shape[0]
    solver = amg.AMG(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, dim=3)
    try:
        s, levels = solver.info()
        assert s["num_levels"] == 1
        dense = 8.0 * n * n + 16.0 * n
        if case in ("random_2200", "below_1999"):
            assert levels[0]["vcycle_bytes_fp64"] == dense
        else:
            assert levels[0]["vcycle_bytes_fp64"] < 0.51 * dense
        M = A.toarray()
        b = rng.standard_normal(n)
        ref = np.linalg.solve(M, b)
        cond = np.linalg.cond(M)
        bd = torch.from_numpy(b).cuda()
        z = solver.vcycle(bd).cpu().numpy()
        # the bar of the blocked dense inverse at production size
        assert np.abs(z - ref).max() <= 1e-13 * cond * np.abs(ref).max()
        solver.set_precision(amg.AMG_FP32_IN_FP64)
        z = solver.vcycle(bd).cpu().numpy()
        # float64 products between float32 vectors: rounding of b and x
        assert np.abs(z - ref).max() <= 4 * 6e-8 * cond * np.abs(ref).max()
        x, rc, info = solver.solve(bd, tol=1e-10)
        assert rc == amg.AMG_OK and np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * cond * np.linalg.norm(ref)
    finally:
        solver.close()
