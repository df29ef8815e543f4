"""The calls a user of this library makes, as measurable cases.

A case is one call through the Python binding on a seeded cell-centred
finite-volume system -div(K grad u) = f: one V-cycle (a user's own Krylov
method calls it as its preconditioner), a preconditioned solve from device or
host buffers, a residual check, or a whole request (setup and solve of a new
coefficient field, the unit of work of the serving stream).  `prepare` makes
the system on the GPU from the seed and sets up the hierarchy a program keeps
between calls; `run` is the call itself.

Fields of a case:
  call       vcycle | pcg | pcg_host | bicgstab | residual | request
  field      laplace2d (K = 1, u = 0 on the boundary, f ~ U[-1, 1]),
             lognormal (K = exp(Z)), layered (lognormal with slabs of factor
             1e-6), anisotropic (K = exp(Z) diag(1, 1, 1e-3)); the last three
             with u = 1 at x = 0, u = 0 at x = 1 and no flux elsewhere
  nx, ny, nz cells per axis (nz = 1: two dimensions)
  variance, corr_len   of Z
  mixed      the float32 V-cycle inside float64 CG (else float64 throughout)
  target     coarsening target (rows of the directly solved level)
  tile       rows per tile of the decoupled aggregation (0: sequential)
  autotune   launch shapes timed at setup
  tol        relative residual of a solve
"""

import math

import numpy as np
import torch

from paper_1209_0960_gb300 import amg

MODES = 1000   # cosine modes of the Gaussian field


def _case(name, call, field, shape, *, variance=4.0, corr_len=0.05, mixed=False, target=5000,
          tile=0, autotune=False, tol=1e-8):
    c = dict(call=call, field=field, nx=shape[0], ny=shape[1], nz=shape[2], variance=variance,
             corr_len=corr_len, mixed=mixed, target=target, tile=tile, autotune=autotune, tol=tol)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest hierarchy: the 64 x 64 Poisson problem coarsened to 200
        # rows; every kernel is shorter than its launch
        _case("vcycle_2d_64", "vcycle", "laplace2d", (64, 64, 1), target=200),
        # the same system solved, as a small 2D program does it
        _case("pcg_2d_64", "pcg", "laplace2d", (64, 64, 1), target=200),
        # one request of the serving stream (a ragged box with its own field):
        # setup in tiles on the host cores, solve in mixed precision, all from
        # host buffers
        _case("request_37x52x29", "request", "lognormal", (37, 52, 29), variance=3.0, corr_len=0.1,
              mixed=True, target=1000, tile=4096),
        # the solve of such a request when its hierarchy is kept
        _case("pcg_host_mixed_61x47x70", "pcg_host", "lognormal", (61, 47, 70), variance=2.0,
              corr_len=0.1, mixed=True, target=1000, tile=4096),
        # the library's defaults on a middle size, float64, odd sides
        _case("pcg_81x64x77", "pcg", "lognormal", (81, 64, 77)),
        # the Krylov method of the paper's experiments, tighter tolerance
        _case("bicgstab_72x96x64", "bicgstab", "lognormal", (72, 96, 64), tol=1e-10),
        # the V-cycle alone on the standard 128^3 workload, tuned shapes
        _case("vcycle_128", "vcycle", "lognormal", (128, 128, 128), tile=32768, autotune=True),
        # the standard 128^3 workload solved in float64 and in mixed precision
        _case("pcg_128", "pcg", "lognormal", (128, 128, 128), tile=32768, autotune=True),
        _case("pcg_mixed_128", "pcg", "lognormal", (128, 128, 128), mixed=True, tile=32768,
              autotune=True),
        # high contrast in layers, a box of unequal sides, float64 (the float32
        # V-cycle leaves the slabs' values to about 1e-8 there)
        _case("pcg_layered_192x160x145", "pcg", "layered", (192, 160, 145), tile=131072,
              autotune=True),
        # the anisotropic workload at the largest size that is set up quickly:
        # 12 million unknowns, every large level beyond the caches, in mixed
        # precision; solved far enough that the solution is determined (at 1e-8
        # two orders of the same sums give solutions 1e-7 apart, at 1e-12 1e-11)
        _case("pcg_mixed_anisotropic_256x224x209", "pcg", "anisotropic", (256, 224, 209),
              variance=6.0, corr_len=0.02, mixed=True, tile=262144, autotune=True, tol=1e-12),
        # the residual check of a caller that keeps its own matrix
        _case("residual_160x144x131", "residual", "lognormal", (160, 144, 131)),
    ]


def _sides(rng, lo, hi, most):
    while True:
        s = tuple(int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(3))
        if s[0] * s[1] * s[2] <= most:
            return s


def draw(rng):
    """One more case of the listed kinds: sides spread over their logarithm."""
    kind = rng.choice(["vcycle_2d", "pcg_2d", "request", "pcg_host", "pcg", "bicgstab", "vcycle",
                       "pcg_large", "layered", "anisotropic", "residual"])
    variance = round(rng.uniform(1.0, 4.0), 2)
    if kind in ("vcycle_2d", "pcg_2d"):
        s = tuple(int(round(math.exp(rng.uniform(math.log(48), math.log(200))))) for _ in range(2))
        return _case(None, kind[:-3], "laplace2d", s + (1,), target=rng.choice([200, 1000]))
    if kind == "request":
        return _case(None, "request", "lognormal", _sides(rng, 16, 72, 120000), variance=variance,
                     corr_len=0.1, mixed=True, target=1000, tile=4096)
    if kind == "pcg_host":
        return _case(None, "pcg_host", "lognormal", _sides(rng, 24, 96, 500000), variance=variance,
                     corr_len=0.1, mixed=rng.random() < 0.7, target=1000, tile=4096)
    if kind in ("pcg", "bicgstab"):
        return _case(None, kind, "lognormal", _sides(rng, 24, 96, 450000), variance=variance,
                     tol=1e-8 if kind == "pcg" else 1e-10)
    if kind == "vcycle":
        return _case(None, "vcycle", "lognormal", _sides(rng, 32, 144, 2500000), variance=variance,
                     tile=32768, autotune=rng.random() < 0.5)
    if kind == "pcg_large":
        return _case(None, "pcg", "lognormal", _sides(rng, 72, 144, 2500000), variance=variance,
                     mixed=rng.random() < 0.5, tile=32768, autotune=rng.random() < 0.5)
    if kind == "layered":
        return _case(None, "pcg", "layered", _sides(rng, 80, 200, 4400000), variance=variance,
                     tile=131072, autotune=True)
    if kind == "anisotropic":
        call = rng.choice(["vcycle", "pcg"])
        return _case(None, call, "anisotropic", _sides(rng, 96, 256, 11000000), variance=6.0,
                     corr_len=0.02, mixed=call == "pcg" and rng.random() < 0.5, tile=262144,
                     autotune=True, tol=1e-12)
    return _case(None, "residual", "lognormal", _sides(rng, 32, 200, 6000000), variance=variance)


# ---------------------------------------------------------------------------
# the systems
# ---------------------------------------------------------------------------

def _field(shape, variance, corr_len, seed):
    """Gaussian field Z on the cell centres, [nz, ny, nx]: a sum of cosines
    with wave vectors N(0, 1 / corr_len^2) in its separable form."""
    g = np.random.default_rng(seed)
    k = torch.from_numpy(g.normal(0.0, 1.0 / corr_len, size=(MODES, 3))).cuda()
    phi = torch.from_numpy(g.uniform(0.0, 2.0 * np.pi, size=MODES)).cuda()
    e = []
    for a, m in enumerate(shape):
        x = (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m
        t = torch.outer(x, k[:, a])
        e.append(torch.complex(torch.cos(t), torch.sin(t)))
    ex = e[0] * torch.complex(torch.cos(phi), torch.sin(phi))
    nx, ny, nz = shape
    out = torch.empty((nz, ny, nx), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // (nx * MODES))
    for y in range(0, ny, step):
        w = (e[1][y:y + step, None, :] * ex[None, :, :]).reshape(-1, MODES)
        z = e[2].real @ w.real.T - e[2].imag @ w.imag.T
        out[:, y:y + step, :] = z.reshape(nz, -1, nx)
    return out * math.sqrt(2.0 * variance / MODES)


def _system(case, seed):
    """(diag, [(axis, T)], b): the diagonal, the transmissibility of every face
    between a cell and its next one along the array axes z, y, x, and f, all
    float64 on the GPU."""
    shape = (case["nx"], case["ny"], case["nz"])
    nx, ny, nz = shape
    two_d = nz == 1
    g = np.random.default_rng(seed + 1)
    if case["field"] == "laplace2d":
        K = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
        b = torch.from_numpy(g.uniform(-1.0, 1.0, size=(nz, ny, nx))).cuda()
    else:
        K = torch.exp(_field(shape, case["variance"], case["corr_len"], seed))
        b = torch.zeros_like(K)
    if case["field"] == "layered":
        zc = (torch.arange(nz, dtype=torch.float64, device="cuda") + 0.5) / nz
        for _ in range(8):
            c, t = g.uniform(0.0, 1.0), g.uniform(2.0 / nz, max(2.0 / nz, 0.05))
            K[(zc - c).abs() <= 0.5 * t] *= 1e-6
    aniso = (1e-3 if case["field"] == "anisotropic" else 1.0, 1.0, 1.0)   # array axes z, y, x
    diag = torch.zeros_like(K)
    faces = []
    for ax in range(3):
        m = K.shape[ax]
        if two_d and ax == 0:
            continue
        fac = aniso[ax] * m * m
        lo, hi = K.narrow(ax, 0, m - 1), K.narrow(ax, 1, m - 1)
        T = fac * 2.0 * lo * hi / (lo + hi)
        diag.narrow(ax, 0, m - 1).add_(T)
        diag.narrow(ax, 1, m - 1).add_(T)
        faces.append((ax, T))
        if case["field"] == "laplace2d" or ax == 2:
            for at, u in ((0, 0.0 if case["field"] == "laplace2d" else 1.0), (m - 1, 0.0)):
                w = 2.0 * fac * K.narrow(ax, at, 1)
                diag.narrow(ax, at, 1).add_(w)
                b.narrow(ax, at, 1).add_(w * u)
    return diag, faces, b


def _apply(diag, faces, x):
    """A x on arrays [nz, ny, nx]."""
    y = diag * x
    for ax, T in faces:
        m = x.shape[ax]
        y.narrow(ax, 0, m - 1).sub_(T * x.narrow(ax, 1, m - 1))
        y.narrow(ax, 1, m - 1).sub_(T * x.narrow(ax, 0, m - 1))
    return y


def _csr(diag, faces):
    """CSR of the system on the GPU: row_ptr, col (int32), val (float64)."""
    nz, ny, nx = diag.shape
    n = diag.numel()
    stride = {0: nx * ny, 1: nx, 2: 1}
    vals = torch.zeros((n, 7), dtype=torch.float64, device="cuda")
    has = torch.zeros((n, 7), dtype=torch.bool, device="cuda")
    off = torch.zeros(7, dtype=torch.int32, device="cuda")
    vals[:, 3] = diag.reshape(-1)
    has[:, 3] = True
    for ax, T in faces:
        m = diag.shape[ax]
        for slot, start in ((ax, 1), (6 - ax, 0)):      # the lower, the upper neighbour
            off[slot] = -stride[ax] if start else stride[ax]
            vals[:, slot].view(diag.shape).narrow(ax, start, m - 1).copy_(-T)
            has[:, slot].view(diag.shape).narrow(ax, start, m - 1).fill_(True)
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.cumsum(has.sum(1), 0)
    col = torch.arange(n, dtype=torch.int32, device="cuda")[:, None] + off[None, :]
    return row_ptr, col[has], vals[has]


def _guess(case, seed):
    """A rough field: the error a solve or a V-cycle meets, U[0, 1] per cell."""
    g = np.random.default_rng(seed + 2)
    return torch.from_numpy(g.uniform(0.0, 1.0, size=(case["nz"], case["ny"], case["nx"]))).cuda()


def _solver(case, row_ptr, col, val):
    return amg.AMG(row_ptr, col, val, dim=2 if case["nz"] == 1 else 3,
                   precision=amg.AMG_FP32_IN_FP64 if case["mixed"] else amg.AMG_FP64,
                   coarsen_target=case["target"], aggregation_tile=case["tile"],
                   autotune=int(case["autotune"]))


def prepare(case, seed):
    diag, faces, b = _system(case, seed)
    row_ptr, col, val = _csr(diag, faces)
    state = {"case": case}
    call = case["call"]
    if call == "request":
        state["matrix"] = tuple(t.cpu().numpy() for t in (row_ptr, col, val))
        state["b"] = b.reshape(-1).cpu().numpy()
        return state
    if call == "residual":
        state["matrix"] = (row_ptr, col, val)
        state["b"], state["x"] = b.reshape(-1), _guess(case, seed).reshape(-1)
        state["norm"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return state
    torch.cuda.synchronize()
    state["solver"] = _solver(case, row_ptr, col, val)
    if call == "vcycle":
        # the residual of a rough guess
        state["r"] = (b - _apply(diag, faces, _guess(case, seed))).reshape(-1)
        state["z"] = torch.empty_like(state["r"])
    elif call == "pcg_host":
        state["b"] = b.reshape(-1).cpu().pin_memory()
        state["x"] = torch.empty_like(state["b"]).pin_memory()
    else:
        state["b"] = b.reshape(-1)
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "vcycle":
        return state["solver"].vcycle(state["r"], state["z"])
    if call == "pcg":
        return state["solver"].solve(state["b"], tol=case["tol"])[0]
    if call == "bicgstab":
        return state["solver"].solve_bicgstab(state["b"], tol=case["tol"])[0]
    if call == "pcg_host":
        state["solver"].solve_host(state["b"].numpy(), state["x"].numpy(), tol=case["tol"], zero_guess=True)
        return state["x"]
    if call == "residual":
        amg.amg_residual_norm_noalloc(*state["matrix"], state["b"], state["x"], state["norm"])
        return state["norm"]
    solver = _solver(case, *state["matrix"])
    x = np.empty_like(state["b"])
    solver.solve_host(state["b"], x, tol=case["tol"], zero_guess=True)
    solver.close()
    return x


def work(case):
    """One pass reads the system (or its hierarchy's finest level) and its
    vectors once and does two operations per entry; a solve does so in every
    iteration, a number that depends on the field and is not counted here."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    faces = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    nnz = n + 2 * faces
    return {"bytes": 12.0 * nnz + 4.0 * (n + 1) + 16.0 * n, "flops": 2.0 * nnz}


def exact(case, seed):
    """The solution of A x = b by conjugate gradients with the diagonal as
    preconditioner, run to rounding; the norm of the residual.  Nothing for a
    V-cycle, whose value is the hierarchy's own, nor for the largest systems."""
    if case["call"] == "vcycle" or case["nx"] * case["ny"] * case["nz"] > 5000000 and case["call"] != "residual":
        return None
    diag, faces, b = _system(case, seed)
    if case["call"] == "residual":
        return torch.linalg.vector_norm(b - _apply(diag, faces, _guess(case, seed))).reshape(1)
    x = torch.zeros_like(b)
    inv = 1.0 / diag
    for restart in range(3):   # each restart recomputes the true residual
        r = b - _apply(diag, faces, x)
        z = inv * r
        p = z.clone()
        rz = (r * z).sum()
        for it in range(20000):
            q = _apply(diag, faces, p)
            alpha = rz / (p * q).sum()
            x.add_(alpha * p)
            r.sub_(alpha * q)
            z = inv * r
            new = (r * z).sum()
            p.mul_(new / rz).add_(z)
            rz = new
            if it % 50 == 49 and float(r.norm()) <= 1e-14 * float(b.norm()):
                break
    return x.reshape(-1)
