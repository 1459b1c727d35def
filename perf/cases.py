"""The work that users of this framework have it do, as cases with sizes, inputs and FP64 results.

A case names an operation ("op") of the public binding, a volume (voxel counts,
spacing, storage, phantom kind), a detector and a number of poses:

  render        E = drr.render(volume, detector, poses)
  jacobian      E and the per-ray pose Jacobian, then the pose gradient from it
  autograd      E = drr.drr(volume, detector, poses) and dL/d poses by autograd
  calibrate     gradients without a stored Jacobian: the pose gradient and the
                detector-parameter gradient of an upstream gradient
  register      drr.register: Adam steps on -ZNCC of B poses (render with Jacobian,
                ZNCC, reduction, update), poses and loss history back on the host
  reconstruct   drr.drr_volume: E, dL/d volume and dL/d poses of a volume tensor
  landscape     drr.loss_landscape: -ZNCC at N displaced poses against one image
  serve         requests of mixed volumes, sizes and kinds through drr.Server

Volumes are synthesised on the GPU from the seed: "ct" is a chest-like phantom in
int16 HU (air, body, lungs, vertebrae, ribs, noise inside the body), "soft" a sum
of ellipsoids in attenuation, "bone" air, tissue and bone in attenuation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2208_12737_gb300 import drr

DEV = "cuda"
CT133 = dict(kind="ct", nx=512, ny=512, nz=133, dx=0.703, dy=0.703, dz=2.5)
CT300 = dict(kind="ct", nx=512, ny=512, nz=300, dx=0.703, dy=0.703, dz=1.1)
CUBE256 = dict(kind="soft", nx=256, ny=256, nz=256, dx=1.0, dy=1.0, dz=1.0)


def _det(H, W=None, sdr=510.0, dh=1.4, dw=None):
    return dict(H=H, W=H if W is None else W, sdr=sdr, dh=dh, dw=dh if dw is None else dw)


def listed():
    return [
        # the smallest call: one small DRR of a small volume (a preview, a unit of a data loader)
        dict(name="tiny_forward", op="render", kind="soft", nx=64, ny=64, nz=64, dx=1.0, dy=1.0, dz=1.0, storage="f32",
             B=1, **_det(64, sdr=300.0, dh=2.0)),
        # one interactive DRR of a mid-size volume in 16-bit storage
        dict(name="lone_forward_bf16", op="render", **CUBE256, storage="bf16", B=1, **_det(128, dh=280.0 / 128)),
        # one step of a single registration: DRR, per-ray Jacobian, pose gradient
        dict(name="lone_jacobian", op="jacobian", **CUBE256, storage="f32", B=1, **_det(150, 141, dh=280.0 / 150)),
        # a batch of DRRs of a CT (training data, pose search)
        dict(name="ct_forward", op="render", **CT133, storage="f32", B=16, **_det(200)),
        # the same batch with pose gradients through autograd (pose estimation, the headline workload)
        dict(name="ct_gradient", op="autograd", **CT133, storage="f32", B=16, **_det(200)),
        # a longer CT in 16-bit storage at a large ragged detector, gradients through autograd
        dict(name="ct300_gradient_bf16", op="autograd", **CT300, storage="bf16", B=4, **_det(509, 451, dh=0.6, dw=0.62)),
        # calibration: pose and detector-parameter gradients without storing a Jacobian
        dict(name="ct_calibrate_bf16", op="calibrate", **CT133, storage="bf16", B=3, **_det(331, 255, dh=0.85, dw=1.1)),
        # the high-resolution sweep: 512^3 at 0.5 mm, 1024^2 detector, 16-bit storage (the largest call)
        dict(name="sweep_forward_f16", op="render", kind="bone", nx=512, ny=512, nz=512, dx=0.5, dy=0.5, dz=0.5,
             storage="f16", B=8, **_det(1024, dh=0.4)),
        # concurrent registrations of a CT, two Adam steps
        dict(name="register_b16", op="register", **CT133, storage="f32", B=16, steps=2, **_det(256)),
        # reconstruction: DRR of a volume tensor with gradients to the voxels and the poses
        dict(name="reconstruct", op="reconstruct", kind="soft", nx=200, ny=216, nz=180, dx=1.2, dy=1.2, dz=1.5,
             storage="f32", B=12, **_det(181, 217)),
        # a loss landscape around one pose
        dict(name="landscape", op="landscape", **CT133, storage="f32", B=256, **_det(200)),
        # a burst of requests at a server that holds several volumes
        dict(name="serve_burst", op="serve", kind="mixed", nx=512, ny=512, nz=133, dx=0.703, dy=0.703, dz=2.5,
             storage="mixed", B=16, lo=128, hi=512, **_det(512, dh=280.0 / 512)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any operation, volumes from 40 voxels to 512 a side in any storage, detectors
    of 32 to 1024 pixels a side (ragged), one to 64 poses, at most the largest listed case's work."""
    op = rng.choice(["render", "render", "jacobian", "autograd", "autograd", "calibrate", "register", "reconstruct",
                     "landscape", "serve"])
    if op == "serve":
        return dict(op="serve", kind="mixed", nx=512, ny=512, nz=133, dx=0.703, dy=0.703, dz=2.5, storage="mixed",
                    B=rng.randint(1, 32), lo=rng.randint(64, 160), hi=rng.randint(200, 512), **_det(512, dh=280.0 / 512))
    vol = rng.randint(0, 3)
    if vol == 0 and op != "reconstruct":
        v = dict(CT133)
    elif vol == 1 and op != "reconstruct":
        v = dict(CT300)
    else:
        top = 256 if op == "reconstruct" else 512
        nx, ny, nz = (_log_int(rng, 40, top) for _ in range(3))
        ext = rng.uniform(60.0, 360.0)
        v = dict(kind=rng.choice(["soft", "bone"]), nx=nx, ny=ny, nz=nz, dx=round(ext / nx, 3), dy=round(ext / ny, 3),
                 dz=round(ext / nz, 3))
    storage = "f32" if op == "reconstruct" else rng.choice(["f32", "bf16", "f16"])
    H, W = _log_int(rng, 32, 1024), _log_int(rng, 32, 1024)
    most = 6.0e9 if op in ("render", "landscape") else 1.0e9
    B = max(1, min(_log_int(rng, 1, 64), int(most / (H * W * (v["nx"] + v["ny"] + v["nz"])))))
    if op == "landscape":
        B = max(2, min(4 * B, 256))
        H, W = min(H, 256), min(W, 256)
    case = dict(op=op, **v, storage=storage, B=B,
                **_det(H, W, sdr=float(rng.randint(480, 1020)), dh=round(290.0 / H, 3), dw=round(290.0 / W, 3)))
    if op == "register":
        case["steps"] = 2
        case["B"] = min(B, 16)
    return case


# --- inputs --------------------------------------------------------------------


def _paint(vol, spacing, centre, semi, rot, value, add):
    """Set or add `value` inside the ellipsoid (world mm; the volume is centred at the origin)."""
    n = vol.shape  # (nz, ny, nx)
    ax = [(torch.arange(n[2 - a], device=vol.device, dtype=torch.float32) - 0.5 * (n[2 - a] - 1)) * spacing[a] - centre[a]
          for a in range(3)]
    r = float(max(semi))
    sl = []
    for a in (2, 1, 0):
        idx = torch.nonzero(ax[a].abs() <= r).flatten()
        if idx.numel() == 0:
            return
        sl.append(slice(int(idx[0]), int(idx[-1]) + 1))
    x, y, z = ax[0][sl[2]], ax[1][sl[1]], ax[2][sl[0]]
    q = 0.0
    for k in range(3):
        u = (x[None, None, :] * float(rot[0, k]) + y[None, :, None] * float(rot[1, k]) + z[:, None, None] * float(rot[2, k]))
        q = q + (u / float(semi[k])) ** 2
    sub = vol[sl[0], sl[1], sl[2]]
    if add:
        sub += torch.where(q <= 1.0, float(value), 0.0)
    else:
        sub.masked_fill_(q <= 1.0, float(value))


def _rotation(rng):
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    return q


def _volume(kind, nx, ny, nz, dx, dy, dz, seed):
    """(nz, ny, nx) CUDA tensor: int16 HU for "ct", float32 attenuation (/mm) otherwise."""
    rng = np.random.default_rng([seed, nx, ny, nz])
    sp = (dx, dy, dz)
    ext = np.array([nx * dx, ny * dy, nz * dz])
    eye = np.eye(3)
    if kind == "ct":
        hu = torch.full((nz, ny, nx), -1000.0, device=DEV)
        _paint(hu, sp, np.zeros(3), ext * [0.42, 0.32, 0.68], eye, 40.0, False)
        body = hu > -999.0
        for side in (-1.0, 1.0):
            _paint(hu, sp, ext * [0.17 * side, 0.02, 0.05], ext * [0.13, 0.2, 0.42] * rng.uniform(0.9, 1.1, 3), eye, -800.0, False)
        for v in range(8):
            _paint(hu, sp, ext * [0.0, -0.22, -0.45 + 0.9 * (v + 0.5) / 8],
                   np.array([18.0, 16.0, 0.45 * ext[2] / 8]) * rng.uniform(0.9, 1.1, 3), eye, rng.uniform(700, 1400), False)
        for _ in range(12):
            t = rng.uniform(0, 2 * np.pi)
            c = np.array([0.38 * ext[0] * np.cos(t), 0.28 * ext[1] * np.sin(t), rng.uniform(-0.4, 0.4) * ext[2]])
            rot = np.array([[-np.sin(t), np.cos(t), 0], [-np.cos(t), -np.sin(t), 0], [0, 0, 1.0]]).T
            _paint(hu, sp, c, [rng.uniform(25, 45), 4.0, 4.0], rot, rng.uniform(1000, 2000), False)
        gen = torch.Generator(device=DEV).manual_seed(seed + 17)
        noise = torch.randn(hu.shape, generator=gen, device=DEV) * 10.0
        hu = torch.where(body, hu + noise, hu)
        return hu.round_().clamp_(-1000, 2000).to(torch.int16)
    vol = torch.zeros((nz, ny, nx), device=DEV)
    small = float(ext.min())
    if kind == "soft":
        for _ in range(6):
            _paint(vol, sp, rng.uniform(-0.3, 0.3, 3) * ext, rng.uniform(0.08, 0.4, 3) * small, _rotation(rng),
                   rng.uniform(0.0005, 0.005), True)
        return vol
    _paint(vol, sp, np.zeros(3), 0.4 * ext * rng.uniform(0.9, 1.0, 3), eye, 0.02, False)
    for _ in range(6):
        _paint(vol, sp, rng.uniform(-0.2, 0.2, 3) * ext, rng.uniform(0.05, 0.15, 3) * small, _rotation(rng), 0.021, False)
    for _ in range(8):
        _paint(vol, sp, rng.uniform(-0.25, 0.25, 3) * ext, rng.uniform(0.02, 0.08, 3) * small, _rotation(rng),
               rng.uniform(0.04, 0.06), False)
    return vol


def _poses(B, rng, deg=30.0, mm=10.0):
    return np.concatenate([np.deg2rad(rng.uniform(-deg, deg, (B, 3))), rng.uniform(-mm, mm, (B, 3))], axis=1).astype(np.float32)


def _detector(case):
    return (case["sdr"], case["H"], case["W"], case["dh"], case["dw"])


def _vol_args(case):
    return [case[k] for k in ("kind", "nx", "ny", "nz", "dx", "dy", "dz")]


def _spacing(case):
    return (case["dx"], case["dy"], case["dz"])


SERVED = (  # the server's resident volumes: (volume, storage)
    (dict(kind="soft", nx=128, ny=128, nz=128, dx=2.0, dy=2.0, dz=2.0), "f32"),
    (CUBE256, "bf16"),
    (CUBE256, "f32"),
    (CT133, "f32"),
    (CT133, "bf16"),
)


def _inputs(case, seed):
    """Everything the seed decides but the volume: poses, upstream gradients, targets, requests (numpy)."""
    rng = np.random.default_rng([seed, case["B"], case["H"]])
    B, H, W = case["B"], case["H"], case["W"]
    op = case["op"]
    if op == "serve":  # the burst's sizes, volumes and kinds are the case's, its poses and gradients the seed's
        mix = np.random.default_rng([B, case["lo"], case["hi"]])
        reqs = []
        for _ in range(B):
            n, m = (int(mix.integers(case["lo"], case["hi"] + 1)) for _ in range(2))
            r = dict(vol=int(mix.integers(len(SERVED))), det=(510.0, n, m, 280.0 / n, 280.0 / m), poses=_poses(1, rng), grad=None)
            if mix.uniform() < 0.5:
                r["grad"] = rng.uniform(-1, 1, (1, n, m)).astype(np.float32)
            reqs.append(r)
        return dict(reqs=reqs)
    poses = _poses(B, rng)
    out = dict(poses=poses)
    if op in ("jacobian", "autograd", "calibrate", "reconstruct"):
        out["grad"] = rng.uniform(-1, 1, (B, H, W)).astype(np.float32)
    if op == "register":
        out["init"] = poses + _poses(B, rng, 15.0, 20.0)
    if op == "landscape":
        half = np.concatenate([np.deg2rad([45.0, 45.0, 22.5]), [15.0] * 3])
        out["truth"] = poses[:1]
        out["poses"] = (poses[:1] + rng.uniform(-half, half, (B, 6))).astype(np.float32)
    return out


def _make_volume(v, storage, seed):
    data = _volume(v["kind"], v["nx"], v["ny"], v["nz"], v["dx"], v["dy"], v["dz"], seed)
    return drr.Volume(data, (v["dx"], v["dy"], v["dz"]), storage=storage, hu=v["kind"] == "ct")


def _cuda(a):
    return torch.from_numpy(a).to(DEV)


def prepare(case, seed):
    i = _inputs(case, seed)
    op = case["op"]
    st = dict(op=op, det=_detector(case))
    if op == "serve":
        vols = [_make_volume(v, s, seed) for v, s in SERVED]
        for r in i["reqs"]:
            _, n, m, _, _ = r["det"]
            r["vol"] = vols[r["vol"]]
            r["out"] = np.zeros((1, n, m), np.float32)  # a client keeps and reuses its result buffers
        st.update(reqs=i["reqs"], vols=vols, server=drr.Server(device_budget=1 << 30))
        return st
    if op == "reconstruct":
        st.update(mu=_volume(*_vol_args(case), seed).requires_grad_(True), spacing=_spacing(case),
                  poses=_cuda(i["poses"]).requires_grad_(True), grad=_cuda(i["grad"]))
        return st
    st["vol"] = _make_volume(case, case["storage"], seed)
    st["poses"] = _cuda(i["poses"])
    if op == "autograd":
        st["poses"].requires_grad_(True)
    if "grad" in i:
        st["grad"] = _cuda(i["grad"])
    if op == "register":
        st["init"] = _cuda(i["init"])
        st["fixed"] = drr.render(st["vol"], st["det"], st["poses"])
        st["steps"] = case["steps"]
    if op == "landscape":
        st["fixed"] = drr.render(st["vol"], st["det"], _cuda(i["truth"]))[0]
    torch.cuda.synchronize()
    return st


def run(state):
    op, det = state["op"], state["det"]
    if op == "render":
        return drr.render(state["vol"], det, state["poses"])
    if op == "jacobian":
        E, J = drr.render(state["vol"], det, state["poses"], jacobian=True)
        return E, J, drr.render_backward(state["vol"], det, state["poses"], state["grad"], jac=J)
    if op == "autograd":
        E = drr.drr(state["vol"], det, state["poses"])
        (g,) = torch.autograd.grad(E, state["poses"], state["grad"])
        return E.detach(), g
    if op == "calibrate":
        return (drr.render_backward(state["vol"], det, state["poses"], state["grad"]),
                drr.geometry_grad(state["vol"], det, state["poses"], state["grad"]))
    if op == "register":
        poses, hist, first = drr.register(state["vol"], det, state["fixed"], state["init"], steps=state["steps"])
        return poses, hist, first
    if op == "reconstruct":
        E = drr.drr_volume(state["mu"], state["spacing"], det, state["poses"])
        g_mu, g_pose = torch.autograd.grad(E, (state["mu"], state["poses"]), state["grad"])
        return E.detach(), g_mu, g_pose
    if op == "landscape":
        return drr.loss_landscape(state["vol"], det, state["fixed"], state["poses"])
    tickets = [state["server"].submit(r["vol"], r["det"], r["poses"], r["grad"], out=r["out"]) for r in state["reqs"]]
    out = []
    for t in tickets:
        E, g = t.wait(60000)
        out.append([E] if g is None else [E, g])
    return out


def _ray_work(rays, n, elem, flops):
    """One voxel per crossed segment (about 0.6 of a ray's plane count are crossed), at most the volume once."""
    seg = 0.6 * rays * sum(n)
    return min(float(n[0]) * n[1] * n[2], seg) * elem, seg * flops


def work(case):
    op, B, H, W = case["op"], case["B"], case["H"], case["W"]
    if op == "serve":  # mean size of the drawn detectors
        side = 0.5 * (case["lo"] + case["hi"])
        b, f = 0.0, 0.0
        for v, s in SERVED:
            vb, vf = _ray_work(B / len(SERVED) * side * side, (v["nx"], v["ny"], v["nz"]), 4 if s == "f32" else 2, 5.0)
            b, f = b + vb, f + vf
        return {"bytes": b + 6.0 * B * side * side, "flops": f}
    rays = float(B) * H * W
    steps = case.get("steps", 1)
    per_ray = {"render": 4, "jacobian": 4 + 24 + 4, "autograd": 4 + 4, "calibrate": 4, "register": 4, "reconstruct": 8,
               "landscape": 0}[op]
    flops = {"render": 3.0, "landscape": 3.0, "reconstruct": 11.0, "calibrate": 16.0}.get(op, 8.0)
    b, f = _ray_work(rays, (case["nx"], case["ny"], case["nz"]), 4 if case["storage"] == "f32" else 2, flops)
    b = b * (2 if op == "reconstruct" else 1) + per_ray * rays + 48.0 * B
    if op == "landscape":
        b += 4.0 * H * W
    return {"bytes": b, "flops": f * steps}


# --- the same results in FP64, plain torch -------------------------------------


def _f32(x):
    return float(np.float32(x))


def _stored(v, storage, seed):
    """The volume's values as stored (HU mapped, rounded to the storage type), float64."""
    data = _volume(v["kind"], v["nx"], v["ny"], v["nz"], v["dx"], v["dy"], v["dz"], seed)
    mu = torch.clamp(0.02 * (1.0 + data.double() / 1000.0), min=0.0) if data.dtype == torch.int16 else data.double()
    if storage == "bf16":
        mu = mu.float().to(torch.bfloat16).double()
    elif storage == "f16":
        e = math.frexp(float(mu.abs().max()))[1]
        mu = (mu.float() * 2.0 ** (14 - e)).half().double() * 2.0 ** (e - 14)
    return mu


def _frame(eta, det):
    """R, dR/d(rz, ry, rx) and the canonical source and pixel grid, FP64 on the GPU."""
    sdr, H, W, dh, dw = det
    sdr, dh, dw = _f32(sdr), _f32(dh), _f32(dw)
    rz, ry, rx, *t = [float(x) for x in eta]

    def mats(a, which):
        c, s = math.cos(a), math.sin(a)
        r = {"z": [[c, -s, 0], [s, c, 0], [0, 0, 1]], "y": [[c, 0, s], [0, 1, 0], [-s, 0, c]], "x": [[1, 0, 0], [0, c, -s], [0, s, c]]}[which]
        d = {"z": [[-s, -c, 0], [c, -s, 0], [0, 0, 0]], "y": [[-s, 0, c], [0, 0, 0], [-c, 0, -s]], "x": [[0, 0, 0], [0, -s, -c], [0, c, -s]]}[which]
        return torch.tensor(r, dtype=torch.float64, device=DEV), torch.tensor(d, dtype=torch.float64, device=DEV)

    (Rz, dRz), (Ry, dRy), (Rx, dRx) = mats(rz, "z"), mats(ry, "y"), mats(rx, "x")
    R, dR = Rz @ Ry @ Rx, [dRz @ Ry @ Rx, Rz @ dRy @ Rx, Rz @ Ry @ dRx]
    h = (torch.arange(H, dtype=torch.float64, device=DEV) - 0.5 * (H - 1))
    w = (torch.arange(W, dtype=torch.float64, device=DEV) - 0.5 * (W - 1))
    sc = torch.tensor([0.5 * sdr, 0.0, 0.0], dtype=torch.float64, device=DEV)
    pc = torch.stack([torch.full((H, W), -0.5 * sdr, dtype=torch.float64, device=DEV), (w * dw)[None, :].expand(H, W),
                      (h * dh)[:, None].expand(H, W)], dim=-1).reshape(-1, 3)
    return R, dR, torch.tensor(t, dtype=torch.float64, device=DEV), sc, pc, h, w


def _sums64(mu, spacing, s, p, want):
    """Per ray: the radiologic path length E (Eq. 2) as a sum over plane crossings of weight times
    position, and (want) the per-axis sums of the weights and of weight times position."""
    nz, ny, nx = mu.shape
    n = (nx, ny, nz)
    sp = [_f32(x) for x in spacing]
    b = [-0.5 * n[a] * sp[a] for a in range(3)]
    flat = mu.reshape(-1)
    d = p - s
    L = d.norm(dim=1)
    G, A = [], []
    for a in range(3):
        planes = torch.arange(n[a] + 1, dtype=torch.float64, device=DEV)
        da = d[:, a:a + 1]
        alpha = (b[a] + planes * sp[a] - s[a]) / da
        base = None
        ok = (alpha > 0.0) & (alpha < 1.0)
        for c in range(3):
            if c == a:
                continue
            i = torch.floor((s[c] - b[c] + alpha * d[:, c:c + 1]) / sp[c])
            ok &= (i >= 0) & (i < n[c])
            i = i.clamp_(0, n[c] - 1).long() * (1, nx, nx * ny)[c]
            base = i if base is None else base + i
        st = (1, nx, nx * ny)[a]
        k = torch.arange(n[a] + 1, device=DEV)
        v_hi = torch.where(ok & (k < n[a]), flat[base + (k.clamp(max=n[a] - 1) * st)], 0.0)   # voxel above the plane
        v_lo = torch.where(ok & (k > 0), flat[base + ((k - 1).clamp(min=0) * st)], 0.0)       # voxel below it
        wgt = (v_lo - v_hi) * torch.sign(da)
        G.append(wgt.sum(1))
        A.append((wgt * alpha).sum(1))
        del alpha, base, ok, v_hi, v_lo, wgt
    i = [torch.floor((p[:, c] - b[c]) / sp[c]) for c in range(3)]
    inside = (i[0] >= 0) & (i[0] < nx) & (i[1] >= 0) & (i[1] < ny) & (i[2] >= 0) & (i[2] < nz)
    q = [i[c].clamp(0, n[c] - 1).long() for c in range(3)]
    end = torch.where(inside, flat[q[0] + nx * (q[1] + ny * q[2])], 0.0)  # pixel inside the volume: ends at alpha = 1
    F = A[0] + A[1] + A[2] + end
    E = L * F
    if not want:
        return E, None, None
    gp = torch.stack([d[:, a] / L * F - L * A[a] / d[:, a] for a in range(3)], 1)             # dE/dp
    gs = torch.stack([-d[:, a] / L * F + L * (A[a] - G[a]) / d[:, a] for a in range(3)], 1)   # dE/ds
    return E, gs, gp


def _render64(mu, spacing, det, eta, want=False, geometry=False):
    """E (H, W), with want the pose Jacobian (6, H, W), with geometry dE/d(sdr, dh, dw) (3, H, W)."""
    H, W = det[1], det[2]
    R, dR, t, sc, pc, h, w = _frame(eta, det)
    s, p = R @ sc + t, pc @ R.T + t
    chunk = max(1, int(4.0e7 / max(mu.shape)))
    Es, Js, Ks = [], [], []
    for lo in range(0, H * W, chunk):
        E, gs, gp = _sums64(mu, spacing, s, p[lo:lo + chunk], want or geometry)
        Es.append(E)
        c = pc[lo:lo + chunk]
        if want:
            rot = [gs @ (dR[j] @ sc) + (gp * (c @ dR[j].T)).sum(1) for j in range(3)]
            Js.append(torch.stack(rot + [gs[:, a] + gp[:, a] for a in range(3)]))
        if geometry:
            hh = h.repeat_interleave(W)[lo:lo + chunk]
            ww = w.repeat(H)[lo:lo + chunk]
            Ks.append(torch.stack([0.5 * ((gs - gp) @ R[:, 0]), hh * (gp @ R[:, 2]), ww * (gp @ R[:, 1])]))
    return (torch.cat(Es).reshape(H, W), torch.cat(Js, 1).reshape(6, H, W) if want else None,
            torch.cat(Ks, 1).reshape(3, H, W) if geometry else None)


def _adjoint64(shape, spacing, det, eta, grad, out):
    """out += the transpose of the forward map applied to grad: crossings sorted along each ray."""
    nz, ny, nx = shape
    n = (nx, ny, nz)
    sp = [_f32(x) for x in spacing]
    R, _, t, sc, pc, _, _ = _frame(eta, det)
    s, p = R @ sc + t, pc @ R.T + t
    b = [-0.5 * n[a] * sp[a] for a in range(3)]
    chunk = max(1, int(4.0e7 / sum(n)))
    for lo in range(0, p.shape[0], chunk):
        d = p[lo:lo + chunk] - s
        al = torch.cat([(b[a] + torch.arange(n[a] + 1, dtype=torch.float64, device=DEV) * sp[a] - s[a]) / d[:, a:a + 1]
                        for a in range(3)], 1)
        al = al.clamp_(0.0, 1.0).sort(dim=1).values
        ln = al[:, 1:] - al[:, :-1]
        mid = 0.5 * (al[:, 1:] + al[:, :-1])
        idx, ok = None, ln > 0
        for a in (2, 1, 0):
            i = torch.floor((s[a] - b[a] + mid * d[:, a:a + 1]) / sp[a])
            ok &= (i >= 0) & (i < n[a])
            i = i.clamp_(0, n[a] - 1).long()
            idx = i if idx is None else idx * n[a] + i
        val = ln * (grad.reshape(-1)[lo:lo + chunk] * d.norm(dim=1))[:, None]
        out.index_add_(0, idx[ok], val[ok])


def _zncc64(E, F, eps=1e-8, grad=False):
    """-ZNCC of one pair and, with grad, its image gradient."""
    c, f = E - E.mean(), F - F.mean()
    si, sf = c.square().mean().sqrt(), f.square().mean().sqrt()
    fh = f / (sf + eps)
    z = (c * fh).mean() / (si + eps)
    if not grad:
        return -z, None
    return -z, -(fh - z * c / si) / (E.numel() * (si + eps))


def exact(case, seed):
    op, B = case["op"], case["B"]
    det = _detector(case)
    rays = B * case["H"] * case["W"] * case.get("steps", 1)
    if op != "serve" and rays * (case["nx"] + case["ny"] + case["nz"]) > 4.0e10:
        return None
    i = _inputs(case, seed)
    host = lambda x: x.cpu().numpy()
    if op == "serve":
        out, keep = [], {}
        for r in i["reqs"]:
            if r["vol"] not in keep:
                keep = {r["vol"]: _stored(*SERVED[r["vol"]], seed)}
            v = SERVED[r["vol"]][0]
            E, J, _ = _render64(keep[r["vol"]], (v["dx"], v["dy"], v["dz"]), r["det"], r["poses"][0], want=r["grad"] is not None)
            out.append([host(E[None])] + ([] if r["grad"] is None else [host((J * _cuda(r["grad"])).sum((1, 2))[None])]))
        return out
    sp = _spacing(case)
    mu = _stored(case, case["storage"], seed)
    g = _cuda(i["grad"]).double() if "grad" in i else None
    if op == "render":
        return torch.stack([_render64(mu, sp, det, e)[0] for e in i["poses"]])
    if op in ("jacobian", "autograd"):
        r = [_render64(mu, sp, det, e, want=True)[:2] for e in i["poses"]]
        E, J = torch.stack([x[0] for x in r]), torch.stack([x[1] for x in r])
        G = (J * g[:, None]).sum((2, 3))
        return (E, J, G) if op == "jacobian" else (E, G)
    if op == "calibrate":
        r = [_render64(mu, sp, det, e, want=True, geometry=True)[1:] for e in i["poses"]]
        return tuple(torch.stack([(x[k] * g[b]).sum((1, 2)) for b, x in enumerate(r)]) for k in (0, 1))
    if op == "reconstruct":
        r = [_render64(mu, sp, det, e, want=True)[:2] for e in i["poses"]]
        gm = torch.zeros(mu.numel(), dtype=torch.float64, device=DEV)
        for b, e in enumerate(i["poses"]):
            _adjoint64(mu.shape, sp, det, e, g[b], gm)
        return (torch.stack([x[0] for x in r]), gm.reshape(mu.shape),
                torch.stack([(x[1] * g[b]).sum((1, 2)) for b, x in enumerate(r)]))
    if op == "landscape":
        F = _render64(mu, sp, det, i["truth"][0])[0]
        return torch.stack([_zncc64(_render64(mu, sp, det, e)[0], F)[0] for e in i["poses"]])
    # register: Adam on -ZNCC, separate rates for angles and translations
    p = i["init"].astype(np.float64)
    m, v = np.zeros_like(p), np.zeros_like(p)
    lr = np.array([1e-2] * 3 + [1.0] * 3)
    fixed = [_render64(mu, sp, det, e)[0] for e in i["poses"]]
    hist = np.zeros((case["steps"], B))
    for t in range(case["steps"]):
        G = np.zeros_like(p)
        for k in range(B):
            E, J, _ = _render64(mu, sp, det, p[k], want=True)
            loss, gi = _zncc64(E, fixed[k], grad=True)
            hist[t, k] = float(loss)
            G[k] = host((J * gi).sum((1, 2)))
        m, v = 0.9 * m + 0.1 * G, 0.999 * v + 0.001 * G * G
        p = p - lr * (m / (1 - 0.9 ** (t + 1))) / (np.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
    return p, hist, None
