"""Launch shapes of the interface geometry and the face kernels on small and thin grids: both sides of the lines at which the
geometry marches one plane or four, a block takes one axis or three and the velocity correction takes tiles or flat rows,
in planes of no whole warp, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,bc", [((33, 20, 240), ("P", "P", "NN")), ((33, 20, 244), ("NN", "P", "DN")),
                                  ((64, 64, 36), ("P", "P", "NN")), ((64, 64, 37), ("P", "P", "NN")),
                                  ((64, 64, 74), ("P", "P", "NN")), ((64, 64, 76), ("P", "P", "NN")),
                                  ((65, 63, 80), ("NN", "NN", "DD")), ((3, 2, 1), ("NN", "DD", "P")), ((1, 5, 2), ("P", "NN", "ND"))])
def test_extension_and_projections(n, bc, mode):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp

    def dev(a):
        return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")

    def close(got, want):
        for a, b in zip(got, want):
            assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-12 * max(np.linalg.norm(b), 1e-30)

    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    C = synth.rng(1).uniform(0.0, 1.0, g.shape)
    C[:, :, : n[0] // 2] = 0.0  # a phase beside a mixture
    mdot = 1.0 + 0.1 * synth.rng(2).standard_normal(g.shape)
    u0 = synth.random_velocity(n, bc, 3)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, grad_mode=mode)
    close(plan.extend(*[dev(a) for a in u0], dev(C), dev(mdot), 100.0, 1.0),
          oracle.extend_liquid_velocity(g, *u0, C, mdot, 100.0, 1.0, mode=mode))
    u = [dev(a) for a in u0]
    p = plan.project(*u, dt_over_rho0=0.5)
    close((*u, p), oracle.project(g, *u0, dt_over_rho0=0.5))
    pn = synth.rng(4).standard_normal(g.shape)
    u = [dev(a) for a in u0]
    p = plan.project_vd(*u, dev(C), dev(pn), dev(0.9 * pn), 1e-3, 2e-3, 100.0, 1.0)
    close((*u, p), oracle.project_variable_density(g, *u0, C, pn, 0.9 * pn, 1e-3, 2e-3, 100.0, 1.0))
    plan.close()
