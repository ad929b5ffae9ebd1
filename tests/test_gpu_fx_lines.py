"""Both sides of the lines at which a plan takes its x and y transforms in fixed point: grids of one-warp tiles of 32 samples, three
short stages, FP32 pairs of powers of two and of other lengths; and grids of prime lengths whose tiles take an eighth of
their values in threads, or more, against the CPU oracle at the parity bars."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp64", (32, 32, 37)), ("fp64", (32, 32, 38)), ("fp64", (32, 40, 374)), ("fp64", (32, 40, 376)),
                                    ("fp64", (30, 25, 399)), ("fp64", (30, 25, 401)), ("fp64", (97, 89, 28)),
                                    ("fp64", (97, 89, 29)), ("fp64", (127, 60, 65)), ("fp64", (127, 60, 66)),
                                    ("fp64", (151, 9, 7)), ("ff", (53, 36, 261)), ("ff", (53, 36, 263)), ("ff", (53, 12, 9)),
                                    ("ff", (128, 36, 151)), ("ff", (128, 36, 152)), ("ff", (40, 50, 1199)),
                                    ("ff", (40, 50, 1201)), ("ff", (90, 100, 311)), ("ff", (90, 100, 312))])
def test_both_sides(prec, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    bc = ("P", "NN", "DN")
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    f = synth.rng(n[2]).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.FP64 if prec == "fp64" else vp.FF,
                   max_refine=0)
    got = plan.poisson_solve(torch.tensor(f, dtype=torch.float64, device="cuda")).cpu().numpy()
    assert np.linalg.norm(got - want) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(want)
    plan.close()
