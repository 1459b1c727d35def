"""The bounds-checked build on the inputs most likely to leave the volume's padding: one-
voxel axes, 1500-plane rays, rays in or almost in voxel planes, coinciding crossings,
rays that clip an edge, back-projection rays that wait for their level.  Every gather is
checked, and every add of a back-projected segment longer than the rounding of its ends
(a shorter one beyond the exit, of crossings that FP32 cannot order, is dropped)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_walks_stay_in_bounds():
    from paper_2208_12737_gb300 import build
    env = dict(os.environ, DRR_LIBRARY=build.build(checked=True), DRR_EXPECT_CHECKED="1")
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider", "-k", "not cost_no_multiple",
                        "tests/test_gpu_slab.py", "tests/test_gpu_aligned.py", "tests/test_gpu_accuracy.py"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert " passed" in r.stdout
