"""Lengths with many short odd stages, whose fixed-point transforms would end with few bits: dense lines keep the accuracy of FP64
butterflies.  A thin slab between walls (z eigenvalue -4e8) divides every mode by about the same number, so that the error
is that of the two transforms, 4e-16 each, and of the division, against the tridiagonal system in extended precision."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1029, 1323, 1701, 1715, 1764, 1911])
def test_dense_line(n, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("VOFP_FX", "1")  # (a single line is a small grid)
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    dz = 2.0 ** -13
    plan = vp.Plan((n, 1, 1), 1.0 / n, 1.0, dz, ("DD", "NN", "DD"))
    ld = np.longdouble
    for seed in range(4):
        f = synth.rng(seed).standard_normal(n)
        d = np.full(n, -2 - 4 / ld(dz) ** 2 / ld(n) ** 2, dtype=ld)
        d[0] -= 1
        d[-1] -= 1
        r = f.astype(ld) / ld(n) ** 2
        for i in range(1, n):
            d[i] -= 1 / d[i - 1]
            r[i] -= r[i - 1] / d[i - 1]
        r[-1] /= d[-1]
        for i in range(n - 2, -1, -1):
            r[i] = (r[i] - r[i + 1]) / d[i]
        p = plan.poisson_solve(torch.tensor(f.reshape(1, 1, n), dtype=torch.float64, device="cuda")).cpu().numpy().ravel()
        assert np.linalg.norm(p - r) <= (2 ** 0.5 * 4e-16 + 4.4e-16) * np.linalg.norm(r)
    plan.close()
