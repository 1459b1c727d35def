"""ZNCC of images whose mean is large against their deviation, at sizes where a thread
sums hundreds of pixels, and the choice between FP32 pairs and FP64."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


@pytest.mark.parametrize("shape", [(1024, 1024), (1021, 1023), (200, 200), (64, 64), (7, 5)])
@pytest.mark.parametrize("mean", [0.0, 1.0, 7.0, 30.0, 1e3, 1e4])
def test_correlated_images_far_from_zero(drr, shape, mean):
    # FP64 sums over n pixels in 2048 threads round at random: below sqrt(n / 2048 + 32) 2^-53 of
    # the mean square (rms about a third of it), hence that times mean square / variance of a
    # variance; twice this for the three moments, and the FP32 result's last bit
    rng = np.random.default_rng(51)
    n = shape[0] * shape[1]
    x = rng.uniform(-1, 1, (2, *shape))
    I = (mean + x).astype(np.float32)
    F = (0.37 * mean + 0.8 * x + 0.4 * rng.uniform(-1, 1, x.shape)).astype(np.float32)
    tol = 2 * np.sqrt(n / 2048 + 32) * 2.0**-53 * (mean**2 + 1 / 3) / (0.8 / 3)
    loss, g = drr.zncc(torch.from_numpy(I).cuda(), torch.from_numpy(F).cuda(), eps=1e-8)
    ref, g_ref = oracle.zncc_loss(I, F, 1e-8), oracle.zncc_loss_grad(I, F, 1e-8)
    assert np.abs(loss.cpu().numpy() - ref).max() < tol + 2.0**-24
    scale = np.abs(g_ref).max()
    assert np.abs(g.cpu().numpy() - g_ref).max() < (4 * tol + 2.0**-22) * scale


def test_one_small_pixel_does_not_change_the_path(drr):
    # (a ray that clips a corner): once sent the pair through a second pass, in FP64
    rng = np.random.default_rng(52)
    I = torch.from_numpy(rng.uniform(0, 5, (32, 1024, 1024)).astype(np.float32)).cuda()
    F = (0.5 * I + 1.0).contiguous()
    J = I.clone()
    J[:, :, :4] = 0.0  # (all pixels of some threads)
    J[:, 0, 0] = 1e-12

    def ms(A):
        best = np.inf
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            drr.zncc(A, F, grad=False)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    plain, odd = ms(I), ms(J)
    assert odd < 1.5 * plain, (odd, plain)
