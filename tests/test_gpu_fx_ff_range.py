"""FP32-pair spectra near both ends of the FP32 range through the fixed-point x passes: spectral values from 2^127 to 2^128
stay finite, and subnormal ones are read to the last bit.  A right-hand side times a power of two gives the solution times
it: to the parity bar at the upper end; at the lower one every value stored on the way (some 32 a mode, as the z recurrence
mixes rows) has an absolute rounding of 2^-149, the smallest FP32 number."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu
N, BC = (512, 1, 1400), ("P", "P", "NN")  # one y row: the x spectrum goes straight to the z pass


def solve(f):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    plan = vp.Plan(N, 1.0 / N[0], 1.0, synth.uniform_dz(N[2]), BC, prec=vp.FF, max_refine=0)
    p = plan.poisson_solve(torch.tensor(f, dtype=torch.float64, device="cuda")).cpu().numpy()
    plan.close()
    return p


@pytest.mark.parametrize("top", [126, 127])
def test_upper_end(top):
    # f with one mode in x (its spectral value is 512 f's amplitude), noise in z
    a = synth.rng(5).uniform(0.5, 0.999, N[2])
    f = a[:, None, None] * np.cos(2 * np.pi * 7 * (np.arange(N[0]) + 0.5) / N[0])[None, None, :]
    f = np.ascontiguousarray(np.broadcast_to(f, (N[2], N[1], N[0])))
    want = solve(f)
    e = top + 1 - 9  # amplitudes 2^(e - 1) .. 2^e: spectral values 2^top .. 2^(top + 1)
    got = np.ldexp(solve(np.ldexp(f, e)), -e)
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)


@pytest.mark.parametrize("e", [-90, -100, -106, -110])
def test_lower_end(e):
    f = synth.rng(6).standard_normal((N[2], N[1], N[0]))
    want = solve(f)
    got = np.ldexp(solve(np.ldexp(f, e)), -e)
    bound = 1e-10 * np.abs(want).max() + 32 * N[0] * 2.0 ** (-149 - e)
    assert np.abs(got - want).max() <= bound
