"""Bounded z on grids with few systems and many rows: both sides of the line between the staged and the streaming column solver (438
rows, and five or seven tiles of 32 systems an SM above it), with and without the mean mode: the plan's own choice
against the staged and the streaming kernel, asked for through the autotuner's cache file."""
import numpy as np
import pytest

from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "ff"])
@pytest.mark.parametrize("bc", [("P", "NN", "NN"), ("DD", "P", "ND")])
@pytest.mark.parametrize("n", [(3, 760, 440), (3, 768, 440), (3, 768, 438), (3, 1064, 440), (3, 1080, 440)])
def test_both_sides(n, bc, prec, tmp_path, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    pr = vp.FP64 if prec == "fp64" else vp.FF
    dz = synth.stretched_dz(n[2])
    f = torch.tensor(synth.rng(n[1]).standard_normal((n[2], n[1], n[0])), dtype=torch.float64, device="cuda")
    key = "%s|%d|%d|%d|%d|%d|%d|%d" % ((torch.cuda.get_device_name(0).replace(" ", "_"),) + n +
                                       tuple(vp.BC[b] for b in bc) + (pr,))
    p = []
    for zti in (None, 0, 128):
        if zti is not None:
            cache = tmp_path / ("z%d.txt" % zti)
            cache.write_text("%s %d %d %d %d\n" % (key, 4, 8, zti, 0))
            monkeypatch.setenv("VOFP_TUNE_CACHE", str(cache))
        plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc, prec=pr, max_refine=0, tune=0 if zti is None else 1)
        p.append(plan.poisson_solve(f).cpu().numpy())
        plan.close()
    for q in p[1:]:
        assert np.linalg.norm(q - p[0]) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(p[0])
