"""The allocation-free residual norm on rows of any length: groups of 32 rows
with no entry, one, a full tile of 224, one more (the limit between its two
kernels), and several thousand, in matrices whose last group is short, against
numpy."""

import numpy as np
import pytest

from paper_1209_0960_gb300 import amg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-12   # relative, as the other float64 norm checks of the suite


def _lengths(kind, n, rng):
    if kind == "empty":
        return np.zeros(n, dtype=np.int64)
    if kind == "mixed":   # some rows empty, some of thousands of entries
        return rng.choice([0, 1, 7, 27, 300, 5000], size=n, p=[0.2, 0.2, 0.3, 0.2, 0.08, 0.02])
    if kind == "few long":   # short on the mean: several tiles in some groups
        out = rng.integers(0, 4, size=n)
        out[rng.integers(0, n, size=1 + n // 4000)] += 3000
        return out
    out = np.zeros(n, dtype=np.int64)   # groups of `kind` entries, spread over their rows
    for g in range(0, n, 32):
        m = min(32, n - g)
        np.add.at(out, g + rng.integers(0, m, size=kind), 1)
    return out


@pytest.mark.parametrize("n", [1, 31, 33, 8191, 60_013])
@pytest.mark.parametrize("kind", ["empty", 1, 224, 225, 449, 864, "mixed", "few long"])
def test_rows_of_any_length(kind, n):
    rng = np.random.default_rng(n)
    lens = _lengths(kind, n, rng)
    rp = np.zeros(n + 1, dtype=np.int32)
    rp[1:] = np.cumsum(lens)
    nnz = int(rp[-1])
    ci = rng.integers(0, n, size=max(1, nnz)).astype(np.int32)
    va = rng.standard_normal(max(1, nnz))
    b, x = rng.standard_normal(n), rng.standard_normal(n)
    r = b.copy()
    np.subtract.at(r, np.repeat(np.arange(n), lens), va[:nnz] * x[ci[:nnz]])
    ref = float(np.linalg.norm(r))
    dev = [torch.from_numpy(a).cuda() for a in (rp, ci, va, b, x)]
    out = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    for _ in range(2):
        amg.amg_residual_norm_noalloc(*dev, out)
        torch.cuda.synchronize()
        assert abs(float(out.item()) - ref) <= TOL * ref
