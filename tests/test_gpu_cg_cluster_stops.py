"""The CG work as one cluster launch: which systems run it, read off the launches
themselves on both sides of the limit, and its stops inside the loop (a
direction of negative curvature, a dot product that overflows, the tolerance),
with the loop on the device and on the host, against a CG in numpy that applies
the same V-cycle."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_1209_0960_gb300 import amg
from paper_1209_0960_gb300 import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _kinds(solver, b):
    solver.profile(1)
    solver.solve(b, tol=0.0, maxit=2)
    kinds = {d["name"] for d in solver.profile_read()}
    solver.profile(0)
    return kinds


@pytest.mark.parametrize("shape,cluster", [((64, 64), True), ((4, 6144), True), ((3511, 7), False)],
                         ids=["4096", "24576", "24577"])
@pytest.mark.parametrize("flexible", [0, 1])
def test_which_systems_run_it(shape, cluster, flexible):
    A = P.grid_laplacian(shape, dirichlet_shift=0.05)
    solver = amg.AMG(*A, dim=2, coarsen_target=200, flexible_cg=flexible)
    try:
        b = torch.from_numpy(np.random.default_rng(0).uniform(-1.0, 1.0, solver.n)).cuda()
        own = {"cg_update_dot", "cg_dot", "cg_p_update"}   # launches that the cluster replaces
        kinds = _kinds(solver, b)
        assert "cg_spmv_dot" in kinds
        assert kinds & own == (set() if cluster else own)
    finally:
        solver.close()


def _cg(A, b, B, tol, maxit):
    """Iterate, iterations begun, and whether p.Ap > 0 held throughout."""
    x, r = np.zeros_like(b), b.copy()
    z = B(r)
    p, rho = z.copy(), r @ z
    for it in range(1, maxit + 1):
        q = O.spmv(*A, p)
        pq = p @ q
        if not pq > 0.0:
            return x, it, False
        x += rho / pq * p
        r -= rho / pq * q
        if np.linalg.norm(r) <= tol * np.linalg.norm(b):
            break
        z = B(r)
        rho, old = r @ z, rho
        p = z + rho / old * p
    return x, it, True


@pytest.mark.parametrize("diag", [3.99, 4.05])
def test_stops_at_negative_curvature_and_at_the_tolerance(diag):
    # 3.99 on the diagonal of the 5-point stencil leaves the smoothest mode of
    # 60 x 50 cells at -0.0036; the piecewise constant coarse levels do not see it
    rp, ci, va = P.grid_laplacian((60, 50))
    n = len(rp) - 1
    va = np.where(np.repeat(np.arange(n), np.diff(rp)) == ci, diag, va)
    b = np.random.default_rng(n).uniform(-1.0, 1.0, n)
    bd = torch.from_numpy(b).cuda()
    got = []
    for loop in (0, 1):
        solver = amg.AMG(rp, ci, va, dim=2, coarsen_target=100, device_loop=loop)
        B = lambda r: solver.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        ref, iters, definite = _cg((rp, ci, va), b, B, 1e-8, 60)
        x, rc, info = solver.solve(bd, tol=1e-8, maxit=60)
        assert "cg_update_dot" not in _kinds(solver, bd)
        solver.close()
        assert definite == (diag > 4.0)
        assert rc == (amg.AMG_OK if definite else amg.AMG_ENOTSPD)
        assert abs(info["iterations"] - iters) <= (1 if definite else 0)
        # a stop at the tolerance leaves both within it of the solution; the
        # iterates before the breakdown agree to the rounding of a few steps
        bar = 1e-6 if definite else 1e-10
        assert np.linalg.norm(x.cpu().numpy() - ref) <= bar * np.linalg.norm(ref)
        got.append((x, info["iterations"]))
    assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]


def test_an_overflowing_dot_product_stops_the_loop():
    # r.r is about 1e293, z = B r about 1e165, so r.z overflows in the loop's
    # first step; the guess is left as it was
    rp, ci, va = P.grid_laplacian((40, 30), dirichlet_shift=0.05)
    b = 1e145 * np.random.default_rng(2).uniform(-1.0, 1.0, 1200)
    for loop in (0, 1):
        solver = amg.AMG(rp, ci, va * 1e-20, dim=2, coarsen_target=100, device_loop=loop)
        x, rc, info = solver.solve(torch.from_numpy(b).cuda(), tol=1e-8, maxit=50)
        assert rc == amg.AMG_ENONFINITE and info["iterations"] <= 1
        assert not x.any()
        x, rc, info = solver.solve(torch.from_numpy(b * 1e-145).cuda(), tol=1e-8, maxit=50)
        assert rc == amg.AMG_OK   # the context stays usable
        solver.close()
