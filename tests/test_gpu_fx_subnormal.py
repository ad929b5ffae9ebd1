"""Lines near the end of FP64's range through the fixed-point transforms, which lift them into it first: a right-hand side times
2^-960 to 2^-990 (line exponents below 66, values still normal) gives the solution times that, to 1e-15 and the rounding of
subnormal results; one below the normal range is solved as the rounded numbers it holds."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bc", [((128, 64, 6), ("P", "P", "NN")), ((64, 128, 5), ("NN", "DD", "DD")),
                                  ((64, 250, 13), ("ND", "DN", "P"))])
def test_lifted_lines(n, bc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)

    def solve(f):
        return plan.poisson_solve(torch.tensor(f, dtype=torch.float64, device="cuda")).cpu().numpy()

    f = synth.rng(11).standard_normal((n[2], n[1], n[0]))
    p = solve(f)
    for e in (-960, -975, -990):
        q = solve(np.ldexp(f, e))
        assert np.abs(np.ldexp(q, -e) - p).max() <= 1e-15 * np.abs(p).max(), e
    # subnormal inputs, 27 bits of the solution above the smallest number: ten of them, at least, survive
    g = np.ldexp(f, -1040)
    q, want = np.ldexp(solve(g), 1040), solve(np.ldexp(g, 1040))
    assert np.linalg.norm(q - want) <= 1e-3 * np.linalg.norm(want)
    plan.close()
