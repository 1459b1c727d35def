"""How exact the pieces of a registration step are, beyond the parity tolerances: Adam
divides by sqrt(v), so that the rounding of a small, cancelling gradient component shows
in the pose.  The bounds are those of the arithmetic."""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs
from tests._parity import FP32_TOL, GRAD_TOL, odet, ovol, rel_err

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


@pytest.mark.parametrize("H, W", [(64, 80), (61, 37), (1, 1), (3, 5), (211, 193)])
def test_stored_jacobian_gradient_of_cancelling_sums(drr, H, W):
    # the sum over pixels cancels to ~1e-4 of its terms; value + error sums lose less than
    # 2^-40 of the terms, and the result is rounded once
    rng = np.random.default_rng(H)
    B, n = 2, H * W
    J = rng.normal(size=(B, 6, n)).astype(np.float32)
    g = rng.normal(size=(B, n)).astype(np.float32)
    h = n // 2
    g[:, h:2 * h] = -g[:, :h]
    J[:, :, h:2 * h] = J[:, :, :h] * np.float32(1.0001)
    vol = drr.Volume(np.ones((4, 4, 4), np.float32), (1.0, 1.0, 1.0))
    P = torch.zeros((B, 6), device="cuda")
    G = drr.render_backward(vol, inputs.Detector(100.0, H, W, 1.0, 1.0), P, torch.from_numpy(g.reshape(B, H, W)).cuda(),
                            jac=torch.from_numpy(J.reshape(B, 6, H, W)).cuda()).cpu().numpy()
    terms = J.astype(np.float64) * g[:, None]
    ref = terms.sum(2)
    assert (np.abs(G - ref) <= 2.0**-24 * np.abs(ref) + 2.0**-40 * np.abs(terms).sum(2)).all()


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
def test_stored_jacobian_gradient_stays_infinite(drr, bad):
    H, W = 40, 37
    J = np.ones((1, 6, H, W), np.float32)
    g = np.ones((1, H, W), np.float32)
    g[0, 20, 11] = bad
    vol = drr.Volume(np.ones((4, 4, 4), np.float32), (1.0, 1.0, 1.0))
    G = drr.render_backward(vol, inputs.Detector(100.0, H, W, 1.0, 1.0), torch.zeros((1, 6), device="cuda"),
                            torch.from_numpy(g).cuda(), jac=torch.from_numpy(J).cuda())
    np.testing.assert_array_equal(G.cpu().numpy(), np.full((1, 6), bad, np.float32))


def test_adam_moves_the_pose_by_the_fp64_step(drr):
    # FP32 states, the step between them in FP64: each is the FP64 result rounded once
    rng = np.random.default_rng(9)
    B, lr = 500, np.array([0.01] * 3 + [1.0] * 3, np.float32).astype(np.float64)
    b1, b2, eps = (float(np.float32(x)) for x in (0.9, 0.999, 1e-8))
    p = rng.uniform(-30, 30, (B, 6)).astype(np.float32)
    P = torch.from_numpy(p.copy()).cuda()
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    for t in (1, 2, 3):
        g = (rng.normal(size=(B, 6)) * 10.0 ** rng.uniform(-6, 0, (B, 6))).astype(np.float32)
        m, v, q = (x.cpu().numpy().astype(np.float64) for x in (M, V, P))
        drr.adam_step(P, torch.from_numpy(g).cuda(), M, V, t, 0.01, 1.0)
        g = g.astype(np.float64)
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        q = q - lr * (m / (1 - b1**t)) / (np.sqrt(v / (1 - b2**t)) + eps)
        for x, ref in ((M, m), (V, v), (P, q)):
            np.testing.assert_array_equal(x.cpu().numpy(), ref.astype(np.float32))


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 3, 3), (2, 4, 31)])
def test_jacobian_renders_of_grazing_rays(drr, shape):
    # a detector fine enough for rays that clip an edge inside one slab: their lengths are a
    # small part of a slab, and are held to the per-pixel tolerance all the same
    rng = np.random.default_rng(31)
    vol_np, sp = rng.uniform(0.01, 0.05, shape).astype(np.float32), (1.0, 1.1, 0.9)
    ext = max(n * s for n, s in zip(shape[::-1], sp))
    det = inputs.Detector(510.0, 601, 597, 3.6 * ext / 600, 3.6 * ext / 600)
    poses = inputs.random_poses(4, seed=32, max_angle_deg=40, max_trans_mm=0.3)
    ov = ovol(vol_np, sp)
    ref, J_ref = oracle.render(ov, odet(det), poses, jacobian=True)
    E, J = drr.render(drr.Volume(vol_np, sp), det, torch.from_numpy(poses).cuda(), jacobian=True)
    assert (ref > 0).sum() > 10000 and rel_err(E.cpu().numpy(), ref).max() < FP32_TOL
    J, J_ref = J.cpu().numpy(), np.moveaxis(J_ref, -1, 1)
    for grp in (slice(0, 3), slice(3, 6)):
        assert (np.abs(J[:, grp] - J_ref[:, grp]) / np.abs(J_ref[:, grp]).max()).max() < GRAD_TOL


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
def test_gradient_sums_stay_infinite(drr, bad):
    # one infinite upstream gradient, without a stored Jacobian and with one, pose and detector parameters
    vol = drr.Volume(np.random.default_rng(33).uniform(0.01, 0.05, (20, 22, 24)).astype(np.float32), (1.0, 1.1, 0.9))
    det = inputs.Detector(150.0, 45, 37, 0.8, 0.8)
    P = torch.from_numpy(inputs.random_poses(2, seed=34)).cuda()
    E, J = drr.render(vol, det, P, jacobian=True)
    g = torch.ones_like(E)
    h, w = (int(x) for x in torch.nonzero((J[1] != 0).all(0))[50])
    g[1, h, w] = bad
    G = drr.render_backward(vol, det, P, g).cpu().numpy()
    np.testing.assert_array_equal(G[1], bad * np.sign(J[1, :, h, w].cpu().numpy()))
    np.testing.assert_array_equal(G[1], drr.render_backward(vol, det, P, g, jac=J).cpu().numpy()[1])
    assert np.isfinite(G[0]).all()
    assert np.isinf(drr.geometry_grad(vol, det, P, g).cpu().numpy()[1]).all()


def test_gradient_sums_beyond_fp32_that_cancel(drr):
    # rows of tiles of opposite signs, each tile's sum just within FP32: 32 of one sign are not
    vol = drr.Volume(np.full((20, 60, 60), 0.03, np.float32), (3.0, 1.0, 1.0))
    det = inputs.Detector(200.0, 16, 512, 1.0, 0.1)
    P = torch.from_numpy(np.array([[0.02, 0.03, 0.01, 1.0, 0.5, 0.3]], np.float32)).cuda()
    E, J = drr.render(vol, det, P, jacobian=True)
    J = J[0].cpu().numpy().astype(np.float64)
    tiles = np.abs(J).reshape(6, 4, 4, 64, 8).sum((2, 4))
    sign = np.repeat([1.0, -1.0, -1.0, 1.0], 4)[:, None]
    g = (np.broadcast_to(sign, (16, 512)) * (2.5e38 / tiles[0].max())).astype(np.float32)  # (rz's tiles; ry's overflow)
    ref, terms = (J * g).sum((1, 2)), np.abs(J * g).sum((1, 2))
    G = drr.render_backward(vol, det, P, torch.from_numpy(g[None].copy()).cuda()).cpu().numpy()[0].astype(np.float64)
    assert terms[0] > 8 * 2 * 3.4e38 and abs(ref[0]) < 3e38  # eight warps of 32 tiles each
    assert abs(G[0] - ref[0]) <= 1e-5 * terms[0]  # (1e-5: what the two walks' Jacobians may differ by)
