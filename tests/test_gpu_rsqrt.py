"""The unit normal's reciprocal square root (an FP32 seed and one third-order step) over the whole range of gradients: the source term
s = mdot (1/rho2 - 1/rho1) |grad C| of a plane ramp, whose gradient is one number, against that number in extended precision.
1 / sqrt to 1 ulp, as CUDA's, and four more roundings of half an ulp: 3 ulps of 2^-52."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


def test_gradient_magnitude():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    n = (256, 64, 3)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), ("P", "P", "P"))
    r = synth.rng(3)
    # C differs in x only: |grad C| = |C[i+1] - C[i-1]| n / 2 exactly but for two roundings
    C = np.ldexp(r.uniform(1.0, 2.0, (n[2], n[1], n[0])), r.integers(-480, 480, (n[2], n[1], 1)))
    C[:, :, 0::2] *= 0.5
    C = np.broadcast_to(C[:1, :1, :], C.shape).copy()
    for e in (-900, -480, -30, 0, 30, 430, 480):
        Ce = np.ldexp(C / np.abs(C).max(), e)
        one = np.ones_like(Ce)
        s = plan.stefan_source(torch.tensor(Ce, device="cuda"), torch.tensor(one, device="cuda"), 2.0, 1.0).cpu().numpy()
        d = np.roll(Ce, -1, 2) - np.roll(Ce, 1, 2)
        want = 0.5 * np.abs(d) * (n[0] / 2.0)
        ok = want > 0
        assert np.isfinite(s).all() and (s[~ok] == 0).all()
        tiny = np.abs(d) * n[0] < 2.0 ** -500  # (squares of the gradient leave the normal range)
        assert (np.abs(s - want)[ok & ~tiny] <= 3 * 2.0 ** -52 * want[ok & ~tiny]).all(), e
    plan.close()
