"""The CG work outside the V-cycle as one cluster launch (systems of up to
kCgClusterRows rows): iterates against a CG in numpy float64 that applies the
same V-cycle, at the edges of the cluster's rows (8,192 at once), for slice
widths with and without a constant in the kernel, and on both sides of the
limit; and the scalars' stops."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(3,), (33,), (1021,), (128, 64), (2731, 3), (20, 20, 20), (16, 16, 32), (125, 131),
          (4, 6144), (3511, 7)]   # 24,576 rows, the most, and one more


def _cg(A, b, B, iters, flexible):
    rp, ci, va = A
    x, r = np.zeros_like(b), b.copy()
    z = B(r)
    p, rho = z.copy(), r @ z
    for _ in range(iters):
        q = O.spmv(rp, ci, va, p)
        alpha = rho / (p @ q)
        x += alpha * p
        r -= alpha * q
        zn = B(r)
        beta = (r @ (zn - z) if flexible else r @ zn) / rho
        rho, z = r @ zn, zn
        p = z + beta * p
    return x


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("flexible", [0, 1])
def test_iterates_match_numpy(shape, flexible):
    A = P.grid_laplacian(shape, dirichlet_shift=0.05)
    n = len(A[0]) - 1
    b = np.random.default_rng(n).uniform(-1.0, 1.0, n)
    solver = amg.AMG(*A, dim=max(2, len(shape)), coarsen_target=200, flexible_cg=flexible)
    try:
        bd = torch.from_numpy(b).cuda()
        B = lambda r: solver.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        iters = 1 if n < 200 else 4   # a directly solved system ends after one
        x, rc, info = solver.solve(bd, tol=0.0 if n >= 200 else 1e-8, maxit=iters)
        assert info["iterations"] == iters
        ref = _cg(A, b, B, iters, flexible)
        # sums of n < 25,000 terms differ by at most n 2^-53 = 3e-12 of the sum
        # of their magnitudes, in four iterations of a well-conditioned system
        # (shift 0.05 of a diagonal of at most 6)
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
    finally:
        solver.close()


def test_no_iteration_leaves_the_guess():
    A = P.grid_laplacian((40, 30), dirichlet_shift=0.05)
    for loop in (0, 1):
        solver = amg.AMG(*A, dim=2, coarsen_target=200, device_loop=loop)
        x0 = np.random.default_rng(1).uniform(size=1200)
        x = x0.copy()
        rc, info = solver.solve_host(np.ones(1200), x, tol=1e-8, maxit=0)
        assert rc == amg.AMG_ENOTCONV and info["iterations"] == 0
        assert np.array_equal(x, x0)
        solver.close()
