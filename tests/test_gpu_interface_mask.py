"""Interface geometry and extension where most of the domain has no interface (the kernels skip flat cells and read the
normals through a mask): C zero or one up to the walls with an interface in a corner, rows of 31 to 65 cells, all
precisions and gradient stencils, against the CPU oracle; and what a non-finite C or mdot away from the interface does."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp
    return vofp


def dev(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def step_c(n, at):
    """Liquid (1) in the corner cells below `at`, a one-cell ramp around it, gas (exactly 0) elsewhere."""
    C = np.zeros((n[2], n[1], n[0]))
    C[:at[2], :at[1], :at[0]] = 1.0
    C[at[2], :at[1], :at[0]] = 0.3
    C[:at[2], at[1], :at[0]] = 0.6
    C[:at[2], :at[1], at[0]] = 1e-9  # below the clip
    return C


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,at,bc", [((31, 9, 7), (4, 3, 2), ("P", "NN", "P")), ((33, 6, 8), (31, 4, 3), ("NN", "P", "DD")),
                                     ((64, 5, 6), (32, 2, 4), ("P", "P", "NN")), ((65, 7, 5), (63, 5, 1), ("DN", "NN", "ND"))])
def test_extension_with_flat_cells(vp, n, at, bc, mode, prec):
    dz = synth.uniform_dz(n[2])
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    C = step_c(n, at)
    mdot = 1.0 + 0.1 * synth.rng(3).standard_normal(C.shape)
    u = synth.random_velocity(n, bc, 4)
    want = oracle.extend_liquid_velocity(g, *u, C, mdot, 100.0, 1.0, mode=mode)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc, prec=vp.FP64 if prec == "fp64" else vp.FF, max_refine=0,
                   grad_mode=mode)
    got = plan.extend(*[dev(a) for a in u], dev(C), dev(mdot), 100.0, 1.0)
    tol = 1e-12 if prec == "fp64" else 1e-10
    for a, b in zip(got, want):
        assert np.linalg.norm(a.cpu().numpy() - b) <= tol * np.linalg.norm(b)
    s = plan.stefan_source(dev(C), dev(mdot), 100.0, 1.0).cpu().numpy()
    ref = oracle.stefan_source(g, C, mdot, 100.0, 1.0, mode=mode)
    assert np.abs(s - ref).max() <= 1e-13 * np.abs(ref).max()
    assert not s[ref == 0.0].any()
    plan.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_nonfinite_inputs_away_from_the_interface(vp, mode):
    n, bc = (40, 8, 6), ("P", "NN", "NN")
    plan = vp.Plan(n, 1.0 / 40, 1.0 / 8, synth.uniform_dz(6), bc, grad_mode=mode)
    C = step_c(n, (5, 3, 2))
    one = np.ones(C.shape)
    for bad in (np.nan, np.inf):
        m = one.copy()
        m[4, 6, 30] = bad
        assert np.isnan(plan.stefan_source(dev(C), dev(m), 100.0, 1.0).cpu().numpy()[4, 6, 30])  # 0 times it
        everywhere = np.full(C.shape, bad)
        assert np.isnan(plan.stefan_source(dev(everywhere), dev(one), 100.0, 1.0).cpu().numpy()).all()
    plan.close()
