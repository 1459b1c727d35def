"""The Jacobian modes at axis-aligned poses, the usual starting poses of a registration:
crossings of several axes coincide there by the thousand, or lie closer than the walk's
fixed-point coordinates resolve, and are put in order by their FP64 positions."""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs
from tests._parity import FP32_TOL, GRAD_TOL, grad_err, odet, ovol, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


_Q = np.pi / 2
# volume (nz, ny, nx), spacing, detector; with lattice coincidences on the aligned poses
GEOMETRIES = {
    "cube": ((48, 48, 48), (1.0, 1.0, 1.0), inputs.Detector(128.0, 44, 47, 1.0, 1.0)),
    "flat": ((3, 40, 56), (2.0, 1.0, 0.5), inputs.Detector(96.0, 32, 61, 0.5, 1.0)),
    "wide": ((40, 44, 2), (1.0, 1.0, 16.0), inputs.Detector(200.0, 40, 41, 1.0, 2.0)),
}
ALIGNED = np.array([[0, 0, 0, 0, 0, 0], [_Q, 0, 0, 0, 0, 0], [0, _Q, 0, 0, 0, 0], [0, 0, _Q, 0, 0, 0],
                    [0, 0, 0, 0.5, 1.0, -2.0], [0, 0, 0, 3.1, 5.2, 0.7], [2 * _Q, 0, 0, 0, 0.5, 0.5]], np.float32)
# near-coincidences of a definite order (1e-8 voxels and more; FP64 holds 1e-13)
NEAR = np.array([[0, 0, 0, 1e-8, 2.3e-8, -1.7e-8], [0, 0, 0, -3.1e-8, 4.7e-8, 7.9e-8], [3e-10, 7e-10, -5e-10, 0.5, 1.0, 0.5]],
                np.float32)


@pytest.mark.parametrize("layout", ["x", "z"])
@pytest.mark.parametrize("name", list(GEOMETRIES))
def test_coinciding_crossings(drr, name, layout):
    shape, sp, det = GEOMETRIES[name]
    vol_np = np.random.default_rng(41).uniform(0.0, 0.05, shape).astype(np.float32)
    vol, ov = drr.Volume(vol_np, sp, layout=layout), ovol(vol_np, sp)
    for poses, smooth in ((ALIGNED, False), (NEAR, True)):
        P = torch.from_numpy(poses).cuda()
        E_ref, J_ref = oracle.render(ov, odet(det), poses, jacobian=True)
        E, J = drr.render(vol, det, P, jacobian=True)
        assert rel_err(E.cpu().numpy(), E_ref).max() < FP32_TOL
        assert torch.isfinite(J).all()
        g_np = inputs.upstream_grad(E.shape, seed=42)
        g = torch.from_numpy(g_np).cuda()
        G, K = drr.render_backward(vol, det, P, g), drr.geometry_grad(vol, det, P, g)
        if smooth:  # (where crossings coincide exactly, the gradient has no value)
            J_np, J_ref = J.cpu().numpy(), np.moveaxis(J_ref, -1, 1)
            for grp in (slice(0, 3), slice(3, 6)):
                assert (np.abs(J_np[:, grp] - J_ref[:, grp]) / np.abs(J_ref[:, grp]).max()).max() < GRAD_TOL
            assert grad_err(G.cpu().numpy(), oracle.pose_grad(ov, odet(det), poses, g_np.astype(np.float64))).max() < GRAD_TOL
            K_ref = oracle.geometry_grad(ov, odet(det), poses, g_np.astype(np.float64))
            assert (np.abs(K.cpu().numpy() - K_ref) / np.abs(K_ref).max(axis=0)).max() < GRAD_TOL
        # the split walk of a small launch and the whole one of a large give the same bits
        many = -(-6000 // (-(-det.height // 4) * -(-det.width // 8) * len(poses)))
        Em, Jm = drr.render(vol, det, P.repeat(many, 1), jacobian=True)
        assert torch.equal(Em.view(many, *E.shape), E.expand(many, *E.shape))
        assert torch.equal(Jm.view(many, *J.shape), J.expand(many, *J.shape))


@pytest.mark.parametrize("pose", [0, 1, 3])
def test_aligned_poses_cost_no_multiple(drr, pose):
    # a third of these rays have coinciding crossings; one after another they took 3 to 12
    # times a generic pose's time
    vol = drr.Volume(np.random.default_rng(43).uniform(0.0, 0.05, (256, 256, 256)).astype(np.float32), (1.0, 1.0, 1.0))
    det = inputs.Detector(1000.0, 256, 256, 1.0, 1.0)

    def ms(p):
        P = torch.from_numpy(np.tile(np.asarray(p, np.float32), (16, 1))).cuda()
        E, J = drr.render(vol, det, P, jacobian=True)
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            drr.render(vol, det, P, jacobian=True, out=E, jac=J)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert ms(ALIGNED[pose]) < 2.0 * ms([0.3, -0.2, 0.4, 5.0, -3.0, 2.0])
