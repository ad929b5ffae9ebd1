"""VoF update where C is constant over most of the grid (such cells take no arithmetic): the oracle's result on blocks of
liquid and gas, a uniform C kept exactly, and non-finite velocities inside a phase still showing in the result."""
import numpy as np
import pytest

import oracle
from oracle.vof import vof_update
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


@pytest.mark.parametrize("n,bc", [((33, 17, 18), ("P", "P", "NN")), ((31, 16, 16), ("NN", "DD", "P")),
                                  ((64, 35, 33), ("DN", "P", "ND")), ((1, 2, 3), ("P", "P", "P"))])
def test_blocks_of_both_phases(vp, n, bc):
    dz = synth.uniform_dz(n[2])
    g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    r = synth.rng(8)
    C = np.zeros((n[2], n[1], n[0]))
    C[n[2] // 3:, n[1] // 4:, n[0] // 5:] = 1.0
    C[n[2] // 2, :, :] = r.random((n[1], n[0]))
    ug = synth.random_velocity(n, bc, 92, sigma=0.5)
    dt = 0.1 / max(n)
    want = vof_update(g, C, *ug, dt)
    plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc)
    got = plan.vof_update(dev(C), *[dev(a) for a in ug], dt).cpu().numpy()
    assert np.abs(got - want).max() <= 1e-12
    for c in (0.0, 1.0, 0.3):
        out = plan.vof_update(dev(np.full_like(C, c)), *[dev(a) for a in ug], dt).cpu().numpy()
        assert np.array_equal(out, np.full_like(C, c))
    plan.close()


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("c", [0.0, 1.0])
def test_nonfinite_velocity_inside_a_phase(vp, axis, c):
    n, bc = (20, 18, 17), ("P", "P", "P")
    plan = vp.Plan(n, 1.0 / 20, 1.0 / 18, synth.uniform_dz(17), bc)
    for bad in (np.nan, np.inf):
        ug = [a.copy() for a in synth.random_velocity(n, bc, 5, sigma=0.1)]
        ug[axis][9, 8, 7] = bad
        out = plan.vof_update(dev(np.full((17, 18, 20), c)), *[dev(a) for a in ug], 1e-3).cpu().numpy()
        assert np.isnan(out[9, 8, 7])
    plan.close()
