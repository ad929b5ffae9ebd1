"""GPU parity of the periodic z pass on equal widths (circulant systems, ``csrc/zcirc.cuh``) against the CPU oracle:
tile widths of 32, 16, 8 and 4 columns, partial tiles, empty and one-row segments, the mean mode of the singular
operator, the three precisions; unequal widths (the general column solver) beside them.  Bars as everywhere:
1e-12 for FP64 plans, 1e-10 for the reduced precisions."""
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


@pytest.mark.parametrize("prec", ["fp64", "mixed", "ff"])
@pytest.mark.parametrize("n,bc", [((33, 6, 3), ("P", "P", "P")), ((5, 4, 9), ("NN", "P", "P")),
                                  ((40, 3, 32), ("P", "DD", "P")), ((7, 35, 65), ("P", "NN", "P")),
                                  ((6, 5, 385), ("P", "P", "P")), ((18, 4, 640), ("P", "P", "P")),
                                  ((9, 3, 1000), ("NN", "NN", "P")), ((4, 3, 2050), ("P", "ND", "P"))])
def test_periodic_z_vs_oracle(vp, n, bc, prec):
    import torch
    dz = synth.uniform_dz(n[2], 1.5)
    g = oracle.Grid(*n, 1.0 / n[0], 0.7 / n[1], dz, bc)
    f = synth.rng(17 + n[2]).standard_normal((n[2], n[1], n[0]))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / n[0], 0.7 / n[1], dz, bc, prec={"fp64": vp.FP64, "mixed": vp.MIXED, "ff": vp.FF}[prec])
    got, info = plan.poisson_solve(torch.tensor(f, device="cuda"), info=True)
    err = np.linalg.norm(got.cpu().numpy() - want) / np.linalg.norm(want)
    assert err <= (1e-12 if prec == "fp64" else 1e-10), err
    if g.singular():
        assert abs(info["compat_defect"] - f.mean()) <= 1e-12
    plan.close()


def test_unequal_periodic_widths(vp):
    import torch
    n, bc = (12, 10, 40), ("P", "P", "P")
    dz = synth.uniform_dz(40)
    dz[7] *= 1.25
    g = oracle.Grid(*n, 1.0 / 12, 1.0 / 10, dz, bc)
    f = synth.rng(5).standard_normal((40, 10, 12))
    want = oracle.poisson_solve(g, f)[0]
    plan = vp.Plan(n, 1.0 / 12, 1.0 / 10, dz, bc)
    got = plan.poisson_solve(torch.tensor(f, device="cuda")).cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    plan.close()
