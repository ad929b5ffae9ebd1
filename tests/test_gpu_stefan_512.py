"""The projection with the phase-change source, on x lines of 512 samples in tiles of eight pairs (2,432 lines or more), whose
right-hand side only the run-time fixed-point kernel forms, in FP64 and FP32 pairs, against the CPU oracle; fewer
lines as well."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("n", [(512, 40, 64), (512, 38, 64), (512, 24, 43)])
def test_project_stefan_long_lines(n, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    bc = ("P", "P", "NN")
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    C, centre = synth.droplet(n, bc, 3)
    mdot = np.ones(C.shape)
    u0 = synth.swirl_velocity(n, bc, centre, 4)
    want = oracle.project(g, *u0, src=oracle.stefan_source(g, C, mdot, 100.0, 1.0), dt_over_rho0=0.02)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.FP64 if prec == "fp64" else vp.FF,
                   max_refine=0)
    u = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in u0]
    p = plan.project_stefan(*u, *(torch.tensor(a, dtype=torch.float64, device="cuda") for a in (C, mdot)), 100.0, 1.0,
                            dt_over_rho0=0.02)
    for a, b in zip((*u, p), want):
        assert np.linalg.norm(a.cpu().numpy() - b) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(b)
    plan.close()
