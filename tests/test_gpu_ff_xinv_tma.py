"""FP32-pair plans of 128, 256 and 512 samples on grids below the fixed-point passes' lines: the inverse x pass on TMA-staged tiles
(full, ragged and single tiles), written and added to the potential, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refine", [0, 2])
@pytest.mark.parametrize("bc", [("P", "NN", "NN"), ("DD", "P", "DN"), ("ND", "NN", "P")])
@pytest.mark.parametrize("n", [(128, 16, 16), (128, 7, 5), (256, 32, 11), (256, 5, 3), (512, 9, 13), (512, 1, 1)])
def test_small_ff_grids(n, bc, refine):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    f = synth.rng(n[0] + n[1]).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.FF, max_refine=refine)
    got = plan.poisson_solve(torch.tensor(f, dtype=torch.float64, device="cuda")).cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
    plan.close()
