"""The autotuner on axes in fixed point: a radix order from its cache file (the stages of x and y reversed, as entries from before
those axes ran in fixed point may hold) leaves the compiled-in kernels and their results alone, bit for bit; a search keeps
parity and writes no reversed order for them."""
import numpy as np
import pytest

import oracle
from paper_1907_00890_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "ff"])
def test_cached_order_and_search(tmp_path, monkeypatch, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build()
    from paper_1907_00890_gb300 import vofp as vp
    pr = vp.FP64 if prec == "fp64" else vp.FF
    for n, bc, searched in (((128, 256, 32), ("P", "NN", "NN"), False), ((256, 128, 33), ("NN", "P", "P"), True)):
        dz = synth.uniform_dz(n[2])
        key = "%s|%d|%d|%d|%d|%d|%d|%d" % ((torch.cuda.get_device_name(0).replace(" ", "_"),) + n +
                                           tuple(vp.BC[b] for b in bc) + (pr,))
        cache = tmp_path / ("tune%d.txt" % searched)
        if not searched:
            cache.write_text("%s %d %d %d %d\n" % (key, 8, 8, 0 if prec == "fp64" else -1, 3))
        f = synth.rng(9).standard_normal((n[2], n[1], n[0]))
        tf = torch.tensor(f, dtype=torch.float64, device="cuda")
        plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc, prec=pr, max_refine=0)
        plain = plan.poisson_solve(tf).cpu().numpy()
        plan.close()
        monkeypatch.setenv("VOFP_TUNE_CACHE", str(cache))
        plan = vp.Plan(n, 1.0 / n[0], 1.0 / n[1], dz, bc, prec=pr, max_refine=0, tune=1)
        tuned = plan.poisson_solve(tf).cpu().numpy()
        plan.close()
        assert cache.read_text().startswith(key)
        g = oracle.Grid(*n, 1.0 / n[0], 1.0 / n[1], dz, bc)
        want = oracle.poisson_solve(g, f)[0]
        assert np.linalg.norm(tuned - want) <= (1e-12 if prec == "fp64" else 1e-10) * np.linalg.norm(want)
        if searched:
            assert int(cache.read_text().split()[4]) == 0  # (both axes)
        elif prec == "fp64":
            assert np.array_equal(tuned, plain)
