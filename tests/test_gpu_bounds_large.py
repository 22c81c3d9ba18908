"""The kernels of grids above the limit of the one-launch stage, of flat axes, of several
waves of blocks and of the state copies on the bounds-checked build of the library (see
test_gpu_bounds.py): no launch forms an index outside its array."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FILES = ["ct_one_launch", "linked_emf", "vector_forms", "flat_axis", "flat_unsound", "divb_waves", "state_lines",
         "state_routes", "2d"]


def test_large_grid_kernels_pass_on_bounds_checked_build():
    from paper_1808_10633_gb300 import build

    env = dict(os.environ, WB_LIBRARY=build.build(variant="check"))
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
           *(os.path.join(ROOT, "tests", f"test_gpu_{f}.py") for f in FILES)]
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    assert "passed" in r.stdout
