"""The slab walk of the Jacobian modes (each axis' crossings in a loop of its own)
and the forward walk where they can go wrong: volumes of one to three voxels along an axis, strong
anisotropy (an axis crossed once or never), rays parallel or almost parallel to
voxel planes, crossings that coincide on a lattice, a source inside the volume,
ragged detectors, and voxels that are not finite.  Against the FP64 oracle, with
the tolerances of the other parity tests: 2e-5 per pixel, and 1e-4 of a
parameter group's largest entry for every ray's Jacobian.  (At crossings that
coincide exactly the gradient has no value, so those cases check E alone.)"""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs
from tests._parity import odet, osp, ovol, FP32_TOL, GRAD_TOL, grad_err, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


def _noise(shape, seed):
    return np.random.default_rng(seed).uniform(0.0, 0.05, shape).astype(np.float32)


_Q = np.pi / 2
# name: volume (nz, ny, nx), spacing, detector, poses, gradient defined
CASES = {
    "one_slab": ((7, 9, 1), (30.0, 1.1, 1.3), inputs.Detector(200.0, 13, 11, 1.0, 1.2), inputs.random_poses(3, seed=71), True),
    "two_thin_axes": ((2, 40, 3), (2.0, 1.0, 9.0), inputs.Detector(150.0, 10, 21, 1.5, 1.5),
                      inputs.random_poses(3, seed=72, max_angle_deg=80), True),
    "anisotropic": ((90, 33, 5), (40.0, 2.0, 0.31), inputs.Detector(600.0, 17, 19, 1.9, 3.0),
                    inputs.random_poses(4, seed=73, max_angle_deg=170), True),
    "any_direction": ((41, 50, 37), (1.0, 0.9, 1.3), inputs.Detector(300.0, 21, 27, 2.0, 2.0),
                      inputs.random_poses(8, seed=74, max_angle_deg=180, max_trans_mm=4), True),
    "nearly_parallel": ((24, 31, 40), (1.0, 1.0, 1.0), inputs.Detector(250.0, 9, 9, 1.0, 1.0),
                        np.array([[1e-6, 2e-6, 0, 0.1, 0.23, 0.31], [_Q + 3e-7, 1e-7, 0, 0.2, 0.31, -0.17]], np.float32), True),
    "lattice": ((32, 32, 32), (1.0, 1.0, 1.0), inputs.Detector(128.0, 33, 32, 1.0, 1.0),
                np.array([[0, 0, 0, 0, 0, 0], [_Q, 0, 0, 0, 0, 0], [0, _Q, 0, 0, 0, 0]], np.float32), False),
    "inside": ((30, 34, 38), (1.0, 1.0, 1.0), inputs.Detector(24.0, 15, 18, 0.9, 0.9),
               inputs.random_poses(3, seed=75, max_angle_deg=180, max_trans_mm=4), True),
}


@pytest.mark.parametrize("layout", ["x", "z"])
@pytest.mark.parametrize("name", list(CASES))
def test_slab_walk_against_the_oracle(drr, name, layout):
    shape, sp, det, poses_np, smooth = CASES[name]
    vol_np = _noise(shape, len(name))
    vol = drr.Volume(vol_np, sp, layout=layout)
    P = torch.from_numpy(poses_np).cuda()
    ov = ovol(vol_np, sp)
    E_ref, J_ref = oracle.render(ov, odet(det), poses_np, jacobian=True)
    J_ref = np.moveaxis(J_ref, -1, 1)
    E, J = drr.render(vol, det, P, jacobian=True)
    assert rel_err(E.cpu().numpy(), E_ref).max() < FP32_TOL
    if not smooth:
        return
    J = J.cpu().numpy()
    for grp in (slice(0, 3), slice(3, 6)):
        assert (np.abs(J[:, grp] - J_ref[:, grp]) / np.abs(J_ref[:, grp]).max()).max() < GRAD_TOL
    g_np = inputs.upstream_grad(E.shape, seed=76)
    G = drr.render_backward(vol, det, P, torch.from_numpy(g_np).cuda()).cpu().numpy()
    G_ref = oracle.pose_grad(ov, odet(det), poses_np, g_np.astype(np.float64))
    assert grad_err(G, G_ref).max() < GRAD_TOL
    K = drr.geometry_grad(vol, det, P, torch.from_numpy(g_np).cuda()).cpu().numpy()
    K_ref = oracle.geometry_grad(ov, odet(det), poses_np, g_np.astype(np.float64))
    assert (np.abs(K - K_ref) / np.abs(K_ref).max(axis=0)).max() < GRAD_TOL


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_voxels_that_are_not_finite_reach_only_their_rays(drr, bad):
    vol_np = _noise((20, 22, 24), 3)
    vol_np[9, 12, 11] = bad
    vol = drr.Volume(vol_np, (1.0, 1.1, 0.9))
    det = inputs.Detector(150.0, 30, 34, 1.0, 1.0)
    P = torch.from_numpy(inputs.random_poses(3, seed=77)).cuda()
    E, _ = drr.render(vol, det, P, jacobian=True)
    E, F = E.cpu().numpy(), drr.render(vol, det, P).cpu().numpy()
    assert not np.isfinite(F).all() and np.isfinite(F).sum() > F.size // 2
    np.testing.assert_array_equal(np.isfinite(E), np.isfinite(F))
    np.testing.assert_array_equal(E[~np.isfinite(F)], F[~np.isfinite(F)])
    np.testing.assert_allclose(E[np.isfinite(F)], F[np.isfinite(F)], rtol=FP32_TOL, atol=1e-3 * FP32_TOL)


@pytest.mark.parametrize("layout", ["x", "y"])
@pytest.mark.parametrize("name", list(CASES))
def test_forward_walk_against_the_oracle(drr, name, layout):
    # a small launch (split over the warps of a tile) and one that fills the GPU give the
    # same bits, with ties at the ends of chunks among them, and both match the oracle
    shape, sp, det, poses_np, _ = CASES[name]
    vol_np = _noise(shape, len(name))
    vol = drr.Volume(vol_np, sp, layout=layout)
    B = poses_np.shape[0]
    E = drr.render(vol, det, torch.from_numpy(poses_np).cuda()).cpu().numpy()
    assert rel_err(E, oracle.render(ovol(vol_np, sp), odet(det), poses_np)).max() < FP32_TOL
    tiles = -(-det.height // 4) * -(-det.width // 8) * B
    many = -(-6000 // tiles)  # past the split kernel's resident tiles
    F = drr.render(vol, det, torch.from_numpy(np.tile(poses_np, (many, 1))).cuda()).cpu().numpy()
    np.testing.assert_array_equal(F.reshape(many, *E.shape), np.broadcast_to(E, (many, *E.shape)))


def test_forward_walk_of_long_rays(drr):
    # more crossings than one FP32 frame would hold: 1500 planes along the rays
    vol_np = _noise((3, 40, 1500), 5)
    vol = drr.Volume(vol_np, (0.2, 0.25, 1.0))
    det = inputs.Detector(700.0, 9, 17, 0.4, 0.4)
    poses_np = np.array([[0.01, 0.002, 0.1, 0.0, 0.3, 0.1], [0.004, -0.001, 0.0, 1.0, 0.0, 0.0]], np.float32)
    P = torch.from_numpy(poses_np).cuda()
    ov = ovol(vol_np, (0.2, 0.25, 1.0))
    E_ref, J_ref = oracle.render(ov, odet(det), poses_np, jacobian=True)
    assert rel_err(drr.render(vol, det, P).cpu().numpy(), E_ref).max() < FP32_TOL
    E, J = drr.render(vol, det, P, jacobian=True)
    assert rel_err(E.cpu().numpy(), E_ref).max() < FP32_TOL
    J_ref = np.moveaxis(J_ref, -1, 1)
    for grp in (slice(0, 3), slice(3, 6)):
        assert (np.abs(J.cpu().numpy()[:, grp] - J_ref[:, grp]) / np.abs(J_ref[:, grp]).max()).max() < GRAD_TOL


BP_CASES = {**CASES,
            # pixels many voxels apart, so that a tile's rays enter at far levels (stepped without waiting),
            # and pixels closer than voxels, with rays of one tile entering through different faces
            "coarse": ((60, 50, 70), (0.4, 0.5, 0.3), inputs.Detector(90.0, 17, 14, 5.0, 4.0), inputs.random_poses(3, seed=78), True),
            "fine": ((9, 30, 28), (1.0, 1.0, 3.0), inputs.Detector(120.0, 61, 45, 0.9, 0.9),
                     inputs.random_poses(3, seed=80, max_angle_deg=60, max_trans_mm=5), True),
            "long": ((3, 40, 1500), (0.2, 0.25, 1.0), inputs.Detector(700.0, 9, 17, 0.4, 0.4),
                     np.array([[0.01, 0.002, 0.1, 0.0, 0.3, 0.1], [0.004, -0.001, 0.0, 1.0, 0.0, 0.0]], np.float32), True)}


@pytest.mark.parametrize("layout", ["x", "z"])
@pytest.mark.parametrize("name", list(BP_CASES))
def test_back_projection_walk_against_the_oracle(drr, name, layout):
    # rays that wait for their voxel level, rays left to FP64 (in voxel planes), zero upstream gradients
    shape, sp, det, poses_np, _ = BP_CASES[name]
    vol = drr.Volume(_noise(shape, 1), sp, layout=layout)
    g_np = inputs.upstream_grad((poses_np.shape[0], det.height, det.width), seed=81)
    g_np[:, ::5, ::3] = 0.0
    gv = torch.zeros(shape, device="cuda")
    drr.render_backward(vol, det, torch.from_numpy(poses_np).cuda(), torch.from_numpy(g_np).cuda(), pose_grad=False,
                        grad_volume=gv)
    ref = oracle.backproject(shape, osp(sp), odet(det), poses_np, g_np.astype(np.float64))
    np.testing.assert_allclose(gv.cpu().numpy(), ref, atol=FP32_TOL * np.abs(ref).max())
