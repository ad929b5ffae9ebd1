"""Lengths with a prime factor above 13 on the GPU: rolled fixed-point stages up to 199 (FP64) and 53 (FP32 pairs), the
Bluestein form beyond, on both sides of each limit, alone and beside other stages, even and odd lines, every kind of
boundary, against the CPU oracle at the parity bars (1e-12, 1e-10)."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("bc", [("P", "NN", "NN"), ("NN", "P", "DD"), ("ND", "DN", "ND"), ("DD", "DD", "NN")])
@pytest.mark.parametrize("n", [(17, 34, 3), (53, 59, 3), (106, 199, 2), (211, 61, 2), (398, 16, 2), (13, 1007, 1),
                               (17 * 19, 5 * 37, 1), (1990, 7, 1)])
def test_primes_vs_oracle(n, bc, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    f = synth.rng(n[0] + 5 * n[1]).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.FP64 if prec == "fp64" else vp.FF,
                   max_refine=0)
    got = plan.poisson_solve(torch.tensor(f, dtype=torch.float64, device="cuda")).cpu().numpy()
    assert np.linalg.norm(got - want) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(want)
    plan.close()
