"""Refinement of a right-hand side whose squares leave the FP32 range (the norms the corrections are judged by add up FP32
terms): the corrections still run, and the solution is as accurate as that of the right-hand side scaled to 1."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "ff"])
@pytest.mark.parametrize("e", [0, 20, 25])
def test_corrections_run_past_the_fp32_range(prec, e):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    n, bc = (40, 36, 24), ("NN", "P", "DN")
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    f = synth.rng(21).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.MIXED if prec == "mixed" else vp.FF,
                   max_refine=3)
    p = plan.poisson_solve(torch.tensor(f * 10.0 ** e, dtype=torch.float64, device="cuda")).cpu().numpy() / 10.0 ** e
    assert np.linalg.norm(p - want) <= 1e-10 * np.linalg.norm(want)
    plan.close()
