"""Sparse lines through the fixed-point stages of large primes: one cell's source, or 36 of them, on a line between two walls,
against the tridiagonal system solved in extended precision.  The bar is what FP64 transforms in Bluestein form leave: each
errs by up to 6.5e-16 of its input (L2), the forward one's error e in any mode m, |e| / sqrt(n), twice that in an unlucky one,
comes out as e / lambda_m; two roundings of the division by the eigenvalues add 4.4e-16 of p."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


def walls(f):
    """p of (p[i-1] - 2 p[i] + p[i+1]) n^2 = f with p = 0 on both walls (half a cell out), long double."""
    n = len(f)
    d = np.full(n, -2.0, dtype=np.longdouble)
    d[0] = d[-1] = -3.0
    r = f.astype(np.longdouble) / np.longdouble(n) ** 2
    for i in range(1, n):
        d[i] -= 1 / d[i - 1]
        r[i] -= r[i - 1] / d[i - 1]
    p = np.zeros(n, dtype=np.longdouble)
    p[-1] = r[-1] / d[-1]
    for i in range(n - 2, -1, -1):
        p[i] = (r[i] - p[i + 1]) / d[i]
    return p


@pytest.mark.parametrize("kind", ["one", "36"])
@pytest.mark.parametrize("n", [61, 127, 151, 197, 199])
def test_sparse_line(n, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    plan = vp.Plan((n, 1, 1), 1.0 / n, 1.0, 1.0, ("DD", "NN", "NN"))
    r = synth.rng(n)
    lam = (2 * n * np.sin(np.pi * np.arange(1, n + 1) / (2 * n))) ** 2
    for _ in range(8):
        f = np.zeros(n)
        at = r.integers(0, n, 1 if kind == "one" else 36)
        f[at] = r.uniform(0.5, 1.0, len(at))
        want = walls(f)
        p = plan.poisson_solve(torch.tensor(f.reshape(1, 1, n), dtype=torch.float64, device="cuda")).cpu().numpy().ravel()
        low = np.linalg.norm(f) / np.sqrt(n) * np.sqrt((1 / lam ** 2).sum())
        assert np.linalg.norm(p - want) <= 2 * 6.5e-16 * low + (6.5e-16 + 4.4e-16) * np.linalg.norm(want), at
    plan.close()
