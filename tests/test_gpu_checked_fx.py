"""The bounds-checked library over the fixed-point transforms, the circulant z pass and the flat face kernels: the files that reach
them, on small grids too (VOFP_FX=1), in a child process; the conftest hook asserts after each test that no index test
failed (see test_gpu_checked.py)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FILES = ["tests/test_gpu_fx_lines.py", "tests/test_gpu_thin_grids.py", "tests/test_gpu_zcirc.py", "tests/test_gpu_fx_sparse.py",
         "tests/test_gpu_ff_xinv_tma.py", "tests/test_gpu_stefan_512.py"]


@pytest.mark.skipif(os.environ.get("VOFP_CHECKED") == "1", reason="the sweep itself")
def test_bounds_checked_fixed_point():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_00890_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider"] + FILES, cwd=ROOT,
                       env=dict(os.environ, VOFP_CHECKED="1", VOFP_FX="1"), capture_output=True, text=True, timeout=600)
    tail = "\n".join((r.stdout + r.stderr).splitlines()[-25:])
    assert r.returncode == 0, tail
    assert " passed" in tail and "failed" not in tail, tail
