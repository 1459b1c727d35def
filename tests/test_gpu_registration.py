"""GPU tests of the registration pieces (Sec. 3.2): the ZNCC kernel against the
FP64 oracle, the Adam kernel against its update rule, and end-to-end gradient
registration that recovers ground-truth poses."""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


def test_zncc_kernel_vs_oracle(drr):
    rng = np.random.default_rng(111)
    I = rng.uniform(0, 5, (5, 37, 41)).astype(np.float32)
    F = (0.7 * I + rng.normal(0, 0.5, I.shape)).astype(np.float32)
    loss, g = drr.zncc(torch.from_numpy(I).cuda(), torch.from_numpy(F).cuda(), eps=1e-8)
    np.testing.assert_allclose(loss.cpu().numpy(), oracle.zncc_loss(I, F, 1e-8), rtol=1e-5, atol=1e-6)
    g_ref = oracle.zncc_loss_grad(I, F, 1e-8)
    assert np.abs(g.cpu().numpy() - g_ref).max() < 1e-5 * np.abs(g_ref).max()
    # identical images: loss -1
    l2 = drr.zncc(torch.from_numpy(I).cuda(), torch.from_numpy(I).cuda(), eps=1e-8, grad=False)
    np.testing.assert_allclose(l2.cpu().numpy(), -1.0, atol=1e-6)


def test_adam_kernel_update_rule(drr):
    rng = np.random.default_rng(112)
    p = rng.normal(size=(4, 6)).astype(np.float32)
    P = torch.from_numpy(p.copy()).cuda()
    m = torch.zeros_like(P)
    v = torch.zeros_like(P)
    pm, mm, vm = p.astype(np.float64), np.zeros((4, 6)), np.zeros((4, 6))
    for t in range(1, 4):
        g = rng.normal(size=(4, 6)).astype(np.float32)
        drr.adam_step(P, torch.from_numpy(g).cuda(), m, v, t, 0.01, 0.5)
        mm = 0.9 * mm + 0.1 * g
        vm = 0.999 * vm + 0.001 * g.astype(np.float64) ** 2
        lr = np.array([0.01] * 3 + [0.5] * 3)
        pm = pm - lr * (mm / (1 - 0.9 ** t)) / (np.sqrt(vm / (1 - 0.999 ** t)) + 1e-8)
    np.testing.assert_allclose(P.cpu().numpy(), pm, rtol=1e-5, atol=1e-6)


def test_registration_recovers_poses(drr):
    shape, sp = (60, 96, 96), (2.0, 2.0, 3.0)
    hu = inputs.ct_phantom_hu(shape, sp, seed=113)
    vol = drr.Volume(hu, sp, hu=True)
    det = inputs.Detector(510.0, 96, 96, 3.0, 3.0)
    truth = inputs.random_poses(6, seed=114, max_angle_deg=20, max_trans_mm=10)
    fixed = drr.render(vol, det, torch.from_numpy(truth).cuda())
    init = truth + inputs.pose_offsets(6, seed=115, max_angle_deg=4, max_trans_mm=4)
    # 250 iterations, the paper's budget per registration (Sec. 3.2).  Gradient descent on
    # this non-convex loss is sensitive to last-bit changes of the gradient, so the test asks
    # for 5 of the 6 problems to converge (-ZNCC < -0.999) and checks their poses.
    poses, hist, first = drr.register(vol, det, fixed, torch.from_numpy(init).cuda(), steps=250,
                                      lr_rot=5e-3, lr_trans=0.5)
    conv = hist[-1] < -0.999
    assert conv.sum() >= 5, hist[-1]
    assert np.all(first[conv] >= 0)
    err = (poses - truth)[conv]
    assert np.abs(err[:, :3]).max() < np.deg2rad(0.5) and np.abs(err[:, 3:]).max() < 1.0, err


def test_registration_step_gradient_full_size(drr):
    # the registration workload at its full sizes (512x512x133 CT, 256x256 detector,
    # 64 problems): the loss and the pose gradient of one step, as the loop composes
    # them (fused forward + Jacobian, ZNCC and its gradient, the reduction), for two
    # of the 64 problems at the initial poses and after 10 Adam steps, against the
    # oracle's render, ZNCC gradient and pose gradient of the same definitions (the
    # oracle renders its own fixed images)
    from tests._parity import GRAD_TOL, grad_err, odet, ovol
    cfg = inputs.REGISTRATION
    hu = inputs.ct_volume_hu()
    vol = drr.Volume(hu, cfg["spacing"], hu=True)
    det = cfg["detector"]
    B = cfg["batch"]
    truth = inputs.random_poses(B, seed=cfg["truth_seed"])
    init = truth + inputs.pose_offsets(B, seed=cfg["offset_seed"])
    fixed = drr.render(vol, det, torch.from_numpy(truth).cuda())
    after, _, _ = drr.register(vol, det, fixed, torch.from_numpy(init).cuda(), steps=10)
    ov = ovol(oracle.hu_to_mu(hu, inputs.MU_WATER).astype(np.float32), cfg["spacing"])
    picks = (0, 37)
    fixed_ref = oracle.render(ov, odet(det), truth[list(picks)])
    for poses_np in (init.astype(np.float32), after.astype(np.float32)):
        poses = torch.from_numpy(poses_np).cuda()
        E, J = drr.render(vol, det, poses, jacobian=True)
        loss, g = drr.zncc(E, fixed, eps=1e-8)
        G = drr.render_backward(vol, det, poses, g, jac=J).cpu().numpy()
        sub = poses_np[list(picks)]
        E_ref = oracle.render(ov, odet(det), sub)
        L_ref = oracle.zncc_loss(E_ref, fixed_ref, 1e-8)
        gE = oracle.zncc_loss_grad(E_ref, fixed_ref, 1e-8)
        G_ref = oracle.pose_grad(ov, odet(det), sub, gE)
        np.testing.assert_allclose(loss.cpu().numpy()[list(picks)], L_ref, atol=1e-5)
        assert grad_err(G[list(picks)], G_ref).max() < GRAD_TOL


@pytest.mark.parametrize("npix", [1, 2, 3, 7, 31, 256, 1023, 4096, 40000, 65537])
@pytest.mark.parametrize("scale,offset", [(1.0, 0.0), (1.0, 1e4), (1e-20, 0.0), (1e20, 0.0)])
def test_zncc_sizes_and_ranges(drr, npix, scale, offset):
    # pixel counts around the shares of a cluster's blocks and of their vector loads,
    # nearly constant images and magnitudes whose squares leave FP32, against NumPy in
    # FP64: the loss to 2e-7 (its own rounding to FP32 is 6e-8) and the gradient to 1e-6
    # of its largest entry, widened where the images' variance is a small part of their
    # mean square (FP64 sums of the squares then lose that much)
    rng = np.random.default_rng(npix)
    I = (scale * (offset + rng.uniform(0.5, 3.0, (3, npix)))).astype(np.float32)
    F = (scale * (offset + rng.uniform(0.5, 3.0, (3, npix)))).astype(np.float32)
    eps = 1e-8 * scale
    loss, g = drr.zncc(torch.from_numpy(I).cuda(), torch.from_numpy(F).cuda(), eps)
    i, f = I.astype(np.float64), F.astype(np.float64)
    c, d = i - i.mean(1, keepdims=True), f - f.mean(1, keepdims=True)
    si, sf = np.sqrt((c * c).mean(1, keepdims=True)), np.sqrt((d * d).mean(1, keepdims=True))
    e = float(np.float32(eps))
    z = (c * d).mean(1, keepdims=True) / ((si + e) * (sf + e))
    if npix == 1:  # no variance: only that nothing breaks
        assert np.isfinite(loss.cpu().numpy()).all()
        return
    g_ref = -(d / (sf + e) - z * c / si) / (npix * (si + e))
    cond = 1e-15 * float(((i * i).mean() + (f * f).mean()) / min((si * si).min(), (sf * sf).min()))
    assert np.abs(loss.cpu().numpy() + z[:, 0]).max() < 2e-7 + cond
    if npix > 2:  # (two pixels: the gradient is zero)
        assert np.abs(g.cpu().numpy() - g_ref).max() < (1e-6 + cond) * np.abs(g_ref).max()
