"""Fixed-point transforms on grids too small for the plan to choose them: the files of the compiled-in, run-time and prime
lengths once more with VOFP_FX=1 (tile remainders, zero lines, scaling, non-finite values are tested on small grids there),
and the sizes on both sides of the lines the choice is made at, in FP64 and FP32 pairs, against the CPU oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("name", ["test_gpu_fixed_point.py", "test_gpu_fx_primes.py"])
def test_small_grids_forced(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(HERE, name), "-x", "-q", "-m", "gpu"],
                       cwd=os.path.dirname(HERE), env=dict(os.environ, VOFP_FX="1"), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("n", [(32, 32, 46), (32, 32, 47), (40, 50, 99), (40, 50, 100), (32, 24, 624), (32, 24, 625),
                               (24, 256, 3), (24, 320, 3)])
def test_both_sides_of_the_lines(n, prec):
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
