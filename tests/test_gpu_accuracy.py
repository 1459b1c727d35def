"""How exact the pieces of a registration step are, beyond the parity tolerances: Adam
divides by sqrt(v), so that the rounding of a small, cancelling gradient component shows
in the pose.  The bounds are those of the arithmetic."""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs
from tests._parity import odet, ovol

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


def test_jacobian_renders_sum_their_voxels_to_the_last_bits(drr):
    # A ray sums up to ~250 voxels: in blocks of 8 (a tree), 4 to 8 blocks a piece, the pieces
    # exactly, then one rounding of the product with the path length.  Each of these ~10 roundings at
    # the size of a piece is uniform in 2^-24 of at most an eighth of the sum, the last in 2^-24 of it:
    # rms below 2^-24 / sqrt(12) * sqrt(1 + 8 * 8 / 64 + ...) < 5e-8.  One running sum: 1e-7.
    rng = np.random.default_rng(5)
    vol_np = rng.uniform(0.018, 0.022, (60, 250, 256)).astype(np.float32)
    sp, det = (0.7, 0.7, 2.5), inputs.Detector(510.0, 48, 52, 1.3, 1.3)
    poses = inputs.random_poses(3, seed=6)
    ref = oracle.render(ovol(vol_np, sp), odet(det), poses)
    E, _ = drr.render(drr.Volume(vol_np, sp), det, torch.from_numpy(poses).cuda(), jacobian=True)
    through = ref > 0.3 * ref.max()
    err = (E.cpu().numpy().astype(np.float64) - ref)[through] / ref[through]
    assert through.mean() > 0.5 and np.sqrt((err**2).mean()) < 5e-8, np.sqrt((err**2).mean())
