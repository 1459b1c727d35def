"""Precision sweep (512^3 at 0.5 mm, air / soft tissue / bone ellipsoids, 1024x1024
detector at 0.4 mm, 8 poses): the volume stored as FP32, BF16 and FP16, each against
the FP64 oracle on 4096 seeded pixels per pose.  FP32 must meet 2e-5; 16-bit volumes
5e-3 against the oracle on the FP32 volume and 2e-5 against the oracle on their own
de-quantised values (the kernel's arithmetic error alone).  Also the plain FP32
baseline walk, whose error is reported, not bounded."""
import numpy as np
import pytest

import oracle
from paper_2208_12737_gb300 import inputs
from tests._parity import FP32_TOL, HALF_TOL, odet, ovol, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def drr():
    from paper_2208_12737_gb300 import build
    build.build()
    from paper_2208_12737_gb300 import drr as d
    d.load()
    return d


@pytest.fixture(scope="module")
def case():
    cfg = inputs.PRECISION
    vol = inputs.bone_tissue_phantom(cfg["shape_zyx"], cfg["spacing"], seed=cfg["phantom_seed"])
    det = cfg["detector"]
    poses = inputs.random_poses(cfg["batch"], seed=cfg["pose_seed"])
    pix = np.random.default_rng(66).choice(det.height * det.width, size=4096, replace=False)
    ref = oracle.render(ovol(vol, cfg["spacing"]), odet(det), poses, pixels=pix)
    return cfg, vol, det, poses, pix, ref


def _sampled(E, pix):
    return E.reshape(E.shape[0], -1)[:, pix]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
def test_precision_per_storage(drr, case, storage):
    cfg, vol, det, poses, pix, ref = case
    v = drr.Volume(vol, cfg["spacing"], storage=storage)
    E = _sampled(drr.render(v, det, torch.from_numpy(poses).cuda()).cpu().numpy(), pix)
    err = rel_err(E, ref).max()
    if storage == "f32":
        assert err < FP32_TOL, err
        return
    assert err < HALF_TOL, err
    if storage == "bf16":
        deq = oracle.round_bf16(vol)
    else:
        sc = oracle.f16_scale(float(np.abs(vol).max()))
        deq = (oracle.round_f16(vol * np.float32(sc)).astype(np.float64) / sc).astype(np.float32)
    ref_deq = oracle.render(ovol(deq, cfg["spacing"]), odet(det), poses, pixels=pix)
    err_deq = rel_err(E, ref_deq).max()
    assert err_deq < FP32_TOL, err_deq


def test_plain_fp32_baseline_is_close_but_unbounded(drr, case):
    cfg, vol, det, poses, pix, ref = case
    v = drr.Volume(vol, cfg["spacing"])
    E = _sampled(drr.render_plain_fp32(v, det, torch.from_numpy(poses).cuda()).cpu().numpy(), pix)
    err = rel_err(E, ref)
    # the textbook FP32 walk computes the same integral to FP32 accuracy, but its drift is not
    # held to the product tolerance
    assert np.median(err) < 1e-4 and err.max() < 1e-1, (np.median(err), err.max())


@pytest.mark.parametrize("layout", ["x", "y", "z"])
@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 30), (2, 4, 31), (5, 3, 255), (4, 2, 300)])
def test_ingest_row_lengths(drr, shape, storage, layout):
    # rows at the edges of a warp's share; values that every storage holds exactly
    vol_np = (np.arange(np.prod(shape)).reshape(shape) % 251 + 1).astype(np.float32)
    det = inputs.Detector(2000.0, 2 * max(shape[:2]) + 3, 2 * max(shape) + 3, 1.0, 1.0)
    poses_np = inputs.random_poses(2, seed=5, max_angle_deg=60, max_trans_mm=0.2)
    E = drr.render(drr.Volume(vol_np, (1.0, 1.0, 1.0), storage=storage, layout=layout), det, torch.from_numpy(poses_np).cuda())
    ref = oracle.render(ovol(vol_np, (1.0, 1.0, 1.0)), odet(det), poses_np)
    assert ref.max() > 0 and rel_err(E.cpu().numpy(), ref).max() < FP32_TOL
