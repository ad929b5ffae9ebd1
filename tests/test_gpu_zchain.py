"""Bounded z axes at the lengths where the staged chains' look-ahead (16 rows) and the low-mode systems' rows per lane
change, against the CPU oracle; and the variable-density pass where most faces lie inside a phase."""
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


@pytest.mark.parametrize("prec", ["fp64", "mixed", "ff"])
@pytest.mark.parametrize("bc", [("P", "P", "NN"), ("NN", "P", "DN")])
@pytest.mark.parametrize("nz", [1, 2, 15, 16, 17, 18, 33, 48, 128, 129, 130, 256, 257, 400])
def test_row_counts(vp, nz, bc, prec):
    n = (35, 6, nz)
    dz = synth.uniform_dz(nz)
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    f = synth.rng(nz).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc, prec={"fp64": vp.FP64, "mixed": vp.MIXED, "ff": vp.FF}[prec])
    got = plan.poisson_solve(dev(f)).cpu().numpy()
    tol = 1e-12 if prec == "fp64" else 1e-10
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
    plan.close()


@pytest.mark.parametrize("rho", [(100.0, 1.0), (1.0, 100.0), (5.0, 5.0)])
@pytest.mark.parametrize("hist", [True, False])
def test_variable_density_inside_the_phases(vp, rho, hist):
    n, bc = (33, 18, 9), ("P", "DD", "ND")
    dz = synth.uniform_dz(n[2])
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    r = synth.rng(21)
    C = np.zeros((n[2], n[1], n[0]))
    C[:5, 4:, 7:20] = 1.0
    C[5, 4:, 7:20] = r.random((14, 13))
    pn = r.standard_normal(C.shape)
    pm = 0.9 * pn if hist else None
    u = synth.random_velocity(n, bc, 6)
    want = oracle.project_variable_density(g, *u, C, pn, pm, 0.01, 0.02, *rho)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    d = [dev(a) for a in u]
    p = plan.project_vd(*d, dev(C), dev(pn), dev(pm) if hist else None, 0.01, 0.02, *rho)
    for a, b in zip(d + [p], want):
        assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-12 * np.linalg.norm(b)
    pn[2, 15, 30] = np.nan  # in the gas: it has to show
    p = plan.project_vd(*[dev(a) for a in u], dev(C), dev(pn), dev(pm) if hist else None, 0.01, 0.02, *rho)
    assert np.isnan(p.cpu().numpy()).all()
    plan.close()
