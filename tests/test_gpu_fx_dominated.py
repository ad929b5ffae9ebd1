"""Long lines with one dominating value through the fixed-point transforms: a source in one cell, alone or 1000 times the rest,
on a line between two walls, against the tridiagonal system solved in extended precision.  The bar is what FP64 transforms
leave (see test_gpu_fx_sparse.py): 3.5e-16 of a transform's input for butterflies, 6.5e-16 in Bluestein form (398)."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth
from test_gpu_fx_sparse import walls

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise", [0.0, 1e-3])
@pytest.mark.parametrize("n", [398, 512, 1024, 2048])
def test_dominated_line(n, noise, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("VOFP_FX", "1")  # (a single line is a small grid)
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    plan = vp.Plan((n, 1, 1), 1.0 / n, 1.0, 1.0, ("DD", "NN", "NN"))
    eps = 6.5e-16 if n == 398 else 3.5e-16
    r = synth.rng(n)
    lam = (2 * n * np.sin(np.pi * np.arange(1, n + 1) / (2 * n))) ** 2
    for _ in range(16):
        f = noise * r.standard_normal(n)
        f[r.integers(0, n)] = r.uniform(0.5, 1.0)
        want = walls(f)
        p = plan.poisson_solve(torch.tensor(f.reshape(1, 1, n), dtype=torch.float64, device="cuda")).cpu().numpy().ravel()
        low = np.linalg.norm(f) / np.sqrt(n) * np.sqrt((1 / lam ** 2).sum())
        assert np.linalg.norm(p - want) <= 2 * eps * low + (eps + 4.4e-16) * np.linalg.norm(want)
    plan.close()
