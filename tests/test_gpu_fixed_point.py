"""The fixed-point x and y transforms (``csrc/fxfft.cuh``) of FP64 and FP32-pair plans on the GPU: every compiled-in length
and its neighbours, tile remainders, rolled odd-prime stages, the longest lines, against the CPU oracle at the parity
bars (1e-12, 1e-10); values near both ends of FP64's range (a power-of-two factor on f is a power-of-two factor on p,
exactly); zero lines beside others; an infinity or a NaN anywhere reaches the whole result."""
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


def plan_of(vp, n, bc, prec):
    return vp.Plan(n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc, prec=vp.FP64 if prec == "fp64" else vp.FF,
                   max_refine=0)


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("bc", [("P", "NN", "NN"), ("NN", "P", "DD"), ("ND", "DN", "ND"), ("DD", "DD", "NN")])
@pytest.mark.parametrize("n", [(32, 64, 3), (64, 33, 7), (65, 128, 2), (128, 31, 5), (256, 18, 3), (17, 256, 2),
                               (512, 9, 2), (6, 512, 2), (11 * 13, 49, 2), (1024, 5, 2), (3, 2048, 1)])
def test_lengths_vs_oracle(vp, n, bc, prec):
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], synth.uniform_dz(n[2]), bc)
    f = synth.rng(n[0] + 3 * n[1]).standard_normal((n[2], n[1], n[0]))
    f[:, n[1] // 2:, :] = 0.0  # zero lines beside others
    want = oracle.poisson_solve(g, f)[0]
    plan = plan_of(vp, n, bc, prec)
    got = plan.poisson_solve(dev(f)).cpu().numpy()
    assert np.linalg.norm(got - want) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(want)
    plan.close()


@pytest.mark.parametrize("n,bc", [((128, 64, 6), ("P", "P", "NN")), ((48, 37, 5), ("NN", "DN", "DD"))])
def test_power_of_two_scaling_is_exact(vp, n, bc):
    f = synth.rng(11).standard_normal((n[2], n[1], n[0]))
    plan = plan_of(vp, n, bc, "fp64")
    p = plan.poisson_solve(dev(f)).cpu().numpy()
    for e in (-900, -300, 300, 900):
        q = plan.poisson_solve(dev(np.ldexp(f, e))).cpu().numpy()
        # (the z pass works in FP64 as before; nothing leaves the normal range here)
        assert np.array_equal(q, np.ldexp(p, e)), e
    tiny = plan.poisson_solve(dev(np.ldexp(f, -1060))).cpu().numpy()  # below the normal range: a few bits are left
    assert np.abs(tiny - np.ldexp(p, -1060)).max() <= 2.0 ** -1060 * np.abs(p).max()
    zero = plan.poisson_solve(dev(np.zeros_like(f))).cpu().numpy()
    assert not zero.any()
    plan.close()


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_input_reaches_the_result(vp, bad, prec):
    n, bc = (64, 20, 6), ("P", "NN", "NN")
    f = synth.rng(12).standard_normal((n[2], n[1], n[0]))
    f[3, 7, 41] = bad
    plan = plan_of(vp, n, bc, prec)
    p = plan.poisson_solve(dev(f)).cpu().numpy()
    assert not np.isfinite(p).any()
    with pytest.raises(vp.VofpError):
        plan.poisson_solve(dev(f), info=True)
    plan.close()
