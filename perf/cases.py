"""The work whose speed is measured: calls that a program using this library makes, over the range of sizes it makes
them at. `listed()` names twelve of them, `draw()` gives others of the same ranges; `prepare()` makes a case's inputs
on the GPU from a seed, `run()` is one pass through the public entry points and returns everything it computed,
`work()` counts what the pass cannot do without, and `exact()` computes the same values in 64 bits with plain PyTorch
and NumPy."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_05558_gb300 import gs, synth
from paper_2506_05558_gb300.autograd import rasterize
from paper_2506_05558_gb300.raster import Rasterizer

DEV = "cuda"


def listed():
    return [
        # The smallest render: one 64x64 view of 1,000 Gaussians (degree-0 colour), forward and adjoint. Unit-sized
        # problems, previews and thumbnails: launches and latency are all of it.
        dict(name="step_64", kind="raster", scene="frustum", n=1000, views=1, width=64, height=64, sh=0),
        # One training view at 720p: 200k Gaussians, degree-3 colour, forward and adjoint.
        dict(name="step_720p", kind="raster", scene="box", n=200_000, views=1, width=1280, height=720, sh=3),
        # One iteration of a keyframe's joint optimisation: 1M Gaussians, eight 1080p views, forward and adjoint
        # with every parameter's and every pose's gradient. The library's headline workload.
        dict(name="step_8x1080p", kind="raster", scene="path", n=1_000_000, views=8, width=1920, height=1080, sh=3),
        # The same with 2M Gaussians and 16 views of four different sizes in one launch: mixed captures.
        dict(name="step_16_uneven", kind="raster", scene="path", n=2_000_000, views=16, width=0, height=0, sh=3),
        # A novel view of a finished reconstruction with its depth integral: forward only, a ragged size.
        dict(name="view_1901x1077", kind="view", scene="path", n=1_000_000, views=1, width=1901, height=1077, sh=3),
        # A coarse level of the coarse-to-fine schedule through torch.autograd: four window frames at a quarter of
        # 720p, all of the scene's Gaussians in few tiles, the integral-keeping filter on.
        dict(name="autograd_4x320x180", kind="autograd", scene="path", n=200_000, views=4, width=320, height=180,
             sh=0),
        # What closes the iteration: L1 loss with its gradient over eight 1080p views, sparse Adam on 1M Gaussians,
        # the pose step.
        dict(name="loss_adam_8x1080p", kind="optim", n=1_000_000, views=8, width=1920, height=1080),
        # A new frame's spawn proposal by direct sampling, 1080p, with the probability maps.
        dict(name="spawn_1080p", kind="spawn", width=1920, height=1080),
        # One training step of the learned spawn proposal on a 1080p frame (tcgen05 path), Adam included.
        dict(name="mlp_train_1080p", kind="mlp", width=1920, height=1080),
        # Bootstrapping bundle adjustment: 8 frames, 6,144 keypoints, 200 Levenberg-Marquardt iterations.
        dict(name="ba_8x6144", kind="ba", frames=8, points=6144, iterations=200),
        # A new frame's pose refinement: 6,144 matched points, 20 iterations.
        dict(name="ba_pose_6144", kind="ba_pose", points=6144, iterations=20),
        # Guided-matching depth of a new 1080p frame: four neighbours, 32 channels, 32 candidates.
        dict(name="guided_1080p", kind="guided", width=1920, height=1080, neighbours=4, channels=32, candidates=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["raster", "raster", "raster", "view", "autograd", "optim", "spawn", "mlp", "ba", "ba_pose",
                       "guided"])
    if kind == "raster":
        width = _log_int(rng, 160, 1920)
        return dict(kind=kind, scene="path", n=_log_int(rng, 2000, 1_000_000), views=rng.randint(1, 8), width=width,
                    height=max(96, int(width * rng.uniform(0.5, 0.8))), sh=rng.randint(0, 3))
    if kind == "view":
        width = _log_int(rng, 320, 1920)
        return dict(kind=kind, scene="path", n=_log_int(rng, 20_000, 1_500_000), views=1, width=width,
                    height=max(180, int(width * rng.uniform(0.5, 0.8))), sh=rng.randint(0, 3))
    if kind == "autograd":
        return dict(kind=kind, scene="path", n=_log_int(rng, 10_000, 500_000), views=rng.randint(1, 4),
                    width=rng.randint(160, 640), height=rng.randint(90, 360), sh=rng.choice([0, 0, 2, 3]))
    if kind == "optim":
        return dict(kind=kind, n=_log_int(rng, 5000, 2_000_000), views=rng.randint(1, 8),
                    width=rng.randint(320, 1920), height=rng.randint(180, 1080))
    if kind == "spawn":
        return dict(kind=kind, width=_log_int(rng, 320, 1920), height=_log_int(rng, 200, 1080))
    if kind == "mlp":  # whole 8x8 patches
        return dict(kind=kind, width=8 * _log_int(rng, 40, 240), height=8 * _log_int(rng, 25, 135))
    if kind == "ba":
        return dict(kind=kind, frames=rng.randint(3, 8), points=_log_int(rng, 600, 6144), iterations=rng.randint(20, 100))
    if kind == "ba_pose":
        return dict(kind=kind, points=_log_int(rng, 500, 20_000), iterations=20)
    return dict(kind=kind, width=_log_int(rng, 320, 1600), height=_log_int(rng, 200, 900), neighbours=rng.randint(1, 4),
                channels=rng.choice([16, 32, 64]), candidates=rng.choice([16, 32, 48]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))


def _np_rng(seed):
    return np.random.Generator(np.random.PCG64(int(seed) % (1 << 62)))


def _sizes(case):
    if case["width"] == 0:
        return [synth.UNEVEN_SIZES[v % 4] for v in range(case["views"])]
    return [(case["width"], case["height"])] * case["views"]


def _gaussians(case, seed):
    """The attribute rows of a case's scene (the recipes of the synthetic workloads, drawn on the GPU)."""
    gen, n, scene = _gen(seed), case["n"], case["scene"]
    uni = lambda *s: torch.rand(*s, generator=gen, device=DEV)
    nrm = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    mo = torch.empty((n, 4), device=DEV)
    if scene == "frustum":
        z = 2.0 + 4.0 * uni(n)
        mo[:, 0] = (uni(n) - 0.5) * case["width"] * z / 80.0
        mo[:, 1] = (uni(n) - 0.5) * case["height"] * z / 80.0
        mo[:, 2] = z
        mu, sd = -3.0, 0.5
    else:
        lo, hi = ([-10, -5, 2], [10, 5, 32]) if scene == "box" else ([-15, -7.5, 2], [15, 7.5, 52])
        lo, hi = torch.tensor(lo, device=DEV), torch.tensor(hi, device=DEV)
        mo[:, :3] = lo + (hi - lo) * uni(n, 3)
        mu, sd = -4.0, 0.7
    mo[:, 3] = nrm(n)
    scale = torch.zeros((n, 4), device=DEV)
    scale[:, :3] = mu + sd * nrm(n, 3)
    quat = nrm(n, 4)
    sh = torch.zeros((n, 48), device=DEV)
    sh[:, :3] = synth.DC_STD * nrm(n, 3)
    nc = 3 * (case["sh"] + 1) ** 2
    if nc > 3:
        sh[:, 3:nc] = 0.05 * nrm(n, nc - 3)
    return mo, scale, quat, sh


def _cameras(case, seed):
    sizes = _sizes(case)
    if case["scene"] == "frustum":
        return [synth.camera(np.eye(3), np.zeros(3), 80.0, *sizes[0])]
    if case["scene"] == "box":
        return [synth.camera(np.eye(3), np.zeros(3), 1000.0 / 1280.0 * sizes[0][0], *sizes[0])]
    rng = _np_rng(seed)
    return [synth.camera(*synth.world_to_camera(R, c), 1500.0 / 1920.0 * w, w, h)
            for (R, c), (w, h) in zip(synth.camera_path(rng, len(sizes)), sizes)]


def _config(case):
    if case["kind"] == "autograd":
        return gs.config(sh_degree=case["sh"], mip_filter=1, dilation=0.1)
    return gs.config(sh_degree=case["sh"])


def _loss_gradient(n_pix, seed):
    """The gradient of an L1 loss over all pixels and channels: +-1 / (3 n_pix)."""
    s = torch.randint(0, 2, (3 * n_pix,), generator=_gen(seed + 77), device=DEV, dtype=torch.int8)
    return (2.0 * s.float() - 1.0) / (3 * n_pix)


def _image(w, h, seed):
    """A structured picture in [0, 1]: random sinusoids and a little noise, [3][h][w]."""
    rng = _np_rng(seed)
    y, x = torch.meshgrid(torch.arange(h, device=DEV).float(), torch.arange(w, device=DEV).float(), indexing="ij")
    img = torch.full((3, h, w), 0.5, device=DEV)
    for _ in range(6):
        kx, ky, ph = rng.uniform(-0.6, 0.6), rng.uniform(-0.6, 0.6), rng.uniform(0, 6.28)
        img += torch.tensor(rng.uniform(0.02, 0.08, 3), dtype=torch.float32, device=DEV)[:, None, None] * torch.sin(kx * x + ky * y + ph)
    img += 0.02 * torch.randn((3, h, w), generator=_gen(seed + 5), device=DEV)
    return img.clamp_(0.0, 1.0).contiguous()


def _f32(a):
    return torch.tensor(np.asarray(a, np.float32), device=DEV).contiguous()


def _exp_se3(xi):
    """4x4 matrix exponential of a tangent (rho, phi) in 64 bits."""
    rho, w = np.asarray(xi[:3], np.float64), np.asarray(xi[3:], np.float64)
    K = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    th = float(np.linalg.norm(w))
    if th < 1e-6:
        A, B, C = 1 - th * th / 6, 0.5 - th * th / 24, 1 / 6 - th * th / 120
    else:
        A, B, C = math.sin(th) / th, (1 - math.cos(th)) / th ** 2, (th - math.sin(th)) / th ** 3
    T = np.eye(4)
    T[:3, :3] = np.eye(3) + A * K + B * K @ K
    T[:3, 3] = (np.eye(3) + B * K + C * K @ K) @ rho
    return T


def _ba_inputs(case, seed):
    pr = synth.ba_problem(seed=int(seed) % (1 << 62), n_frames=case["frames"], n_points=case["points"])
    w = pr["width"]
    cx, cy = w / 2.0, w * 9 // 16 / 2.0
    T = [_exp_se3(x) for x in pr["xi"]]
    q = np.einsum("fij,pj->pfi", np.stack([t[:3, :3] for t in T]), pr["X"]) + np.stack([t[:3, 3] for t in T])
    obs = np.stack([pr["fl"] * q[..., 0] / q[..., 2] + cx, pr["fl"] * q[..., 1] / q[..., 2] + cy], -1) + pr["noise"]
    sx = pr["start_xi"].copy()
    sx[0] = 0.0
    T0 = [_exp_se3(x) @ t for x, t in zip(sx, T)]
    poses = np.stack([np.concatenate([t[:3, :3].reshape(9), t[:3, 3]]) for t in T0])
    pts = np.concatenate([pr["X"] * pr["start_X_scale"], np.zeros((case["points"], 1))], 1)
    return obs.astype(np.float32), cx, cy, np.float32([pr["fl"] * pr["start_fl"]]), poses.astype(np.float32), pts.astype(np.float32)


def _ba_pose_inputs(case, seed):
    pr = synth.ba_pose_problem(seed=int(seed) % (1 << 62), n_obs=case["points"])
    w = pr["width"]
    cx, cy = w / 2.0, w * 9 // 16 / 2.0
    T = _exp_se3(pr["xi"])
    q = pr["X"] @ T[:3, :3].T + T[:3, 3]
    obs = np.stack([pr["fl"] * q[:, 0] / q[:, 2] + cx, pr["fl"] * q[:, 1] / q[:, 2] + cy], -1) + pr["noise"]
    T0 = _exp_se3(pr["start_xi"]) @ T
    pose = np.concatenate([T0[:3, :3].reshape(9), T0[:3, 3]])
    pts = np.concatenate([pr["X"], np.zeros((case["points"], 1))], 1)
    return obs.astype(np.float32), cx, cy, np.float32([pr["fl"]]), pose.astype(np.float32), pts.astype(np.float32)


def _guided_inputs(case, seed):
    """Feature maps of a ray-cast room (a box with four fronto-parallel boxes in it) seen by a path's newest frame and
    its neighbours, and a monocular depth 5% off with 1% holes."""
    W, H, J, C = case["width"], case["height"], case["neighbours"], case["channels"]
    rng, gen = _np_rng(seed), _gen(seed)
    f = 1500.0 / 1920.0 * W
    path = synth.camera_path(rng, J + 1)
    cams = [synth.camera(*synth.world_to_camera(*path[k]), f, W, H) for k in [J] + list(range(J))]
    planes = [((0, 0, 1), 9.0, None), ((0, 1, 0), 1.6, None), ((0, 1, 0), -1.8, None), ((1, 0, 0), -3.5, None),
              ((1, 0, 0), 3.5, None)]
    for _ in range(4):
        zc, xc, yc = rng.uniform(3, 6), rng.uniform(-2, 2), rng.uniform(-1, 1)
        hw, hh = rng.uniform(0.3, 1.0), rng.uniform(0.3, 1.0)
        planes.append(((0, 0, 1), zc, (xc - hw, xc + hw, yc - hh, yc + hh)))
    d = rng.normal(size=(8, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    omega = _f32(d * (2 * np.pi / rng.uniform(8.0 * 5.0 / f, 40.0 * 5.0 / f, 8))[:, None])
    phase, mix = _f32(rng.uniform(0, 6.28, 8)), _f32(rng.normal(size=(8, C)))
    feats = torch.empty((J + 1, H, W, C), dtype=torch.bfloat16, device=DEV)
    y, x = torch.meshgrid(torch.arange(H, device=DEV).float(), torch.arange(W, device=DEV).float(), indexing="ij")
    z_true = None
    for k, c in enumerate(cams):
        R, t = _f32(c["R"]), _f32(c["t"])
        ray = torch.stack([(x + 0.5 - c["cx"]) / c["fx"], (y + 0.5 - c["cy"]) / c["fy"], torch.ones_like(x)], -1).view(-1, 3)
        dw, o = ray @ R, -(R.T @ t)
        best = torch.full((H * W,), math.inf, device=DEV)
        for n, off, rect in planes:
            n = _f32(n)
            s = (off - n @ o) / (dw @ n)
            hit = torch.isfinite(s) & (s > 0.05) & (s < best)
            if rect is not None:
                p = o + s[:, None] * dw
                hit &= (p[:, 0] >= rect[0]) & (p[:, 0] <= rect[1]) & (p[:, 1] >= rect[2]) & (p[:, 1] <= rect[3])
            best = torch.where(hit, s, best)
        best = torch.where(torch.isfinite(best), best, torch.full_like(best, 50.0))
        fv = torch.sin((o + best[:, None] * dw) @ omega.T + phase) @ mix
        feats[k] = (fv / (fv.norm(dim=1, keepdim=True) + 1e-12)).view(H, W, C).to(torch.bfloat16)
        if k == 0:
            z_true = best.view(H, W)
    z = z_true * torch.exp(0.05 * torch.randn((H, W), generator=gen, device=DEV))
    z[torch.rand((H, W), generator=gen, device=DEV) < 0.01] = 0.0
    return cams, feats, z


def _mlp_layers(seed):
    rng = _np_rng(seed)
    return [(rng.uniform(-1, 1, (o, i)) / np.sqrt(i), rng.uniform(-1, 1, o) / np.sqrt(i))
            for o, i in ((128, 194), (128, 128), (128, 128), (3, 128))]


def _mlp_inputs(case, seed):
    img = _image(case["width"], case["height"], seed)
    n_p = (case["width"] // 8) * (case["height"] // 8)
    gen = _gen(seed + 3)
    u = torch.rand((n_p, 4), generator=gen, device=DEV)
    tg = torch.stack([u[:, 0], 2.0 + 18.0 * u[:, 1], -4.0 + 0.5 * torch.randn(n_p, generator=gen, device=DEV),
                      (u[:, 3] < 0.5).float()], 1).contiguous()
    return img, tg


def _optim_inputs(case, seed):
    n, npx, gen = case["n"], case["views"] * case["width"] * case["height"], _gen(seed)
    color = torch.rand((3 * npx,), generator=gen, device=DEV)
    target = torch.rand((3 * npx,), generator=gen, device=DEV)
    rows = lambda s: [s * torch.randn((n, k), generator=gen, device=DEV) for k in (4, 4, 4, 48)]
    visible = (torch.rand((n,), generator=gen, device=DEV) < 0.78).to(torch.uint8)
    return color, target, rows(1.0), rows(1e-6), visible, 1e-3 * torch.randn((case["views"], 6), generator=gen, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("raster", "view", "autograd"):
        mo, sc, q, sh = _gaussians(case, seed)
        cams, cfg, sizes = _cameras(case, seed), _config(case), _sizes(case)
        n_pix = sum(w * h for w, h in sizes)
        s.update(cams=gs.cameras_tensor(cams), cfg=cfg, sizes=sizes, dL=_loss_gradient(n_pix, seed))
        if kind == "autograd":
            s["leaves"] = [t.requires_grad_(True) for t in (mo, sc, q, sh, torch.zeros((case["views"], 6), device=DEV))]
            return s
        s["g"] = gs.Gaussians(mo, sc, q, sh)
        s["r"] = Rasterizer(case["n"], sizes, 1 << 20, cfg)
        s["r"].fit_capacity(s["g"], s["cams"])
        if kind == "view":
            s["r"].img.depth = torch.zeros_like(s["r"].img.t_final)
    elif kind == "optim":
        color, target, p, g, visible, dpose = _optim_inputs(case, seed)
        cams = dict(case, scene="path")
        s.update(color=color, target=target, dL=torch.empty_like(color), loss=torch.zeros(1, device=DEV),
                 ws=gs.workspace(4 * 4096), p=gs.Gaussians(*p), grads=gs.Grads(*g, visible), m=gs.Gaussians.zeros(case["n"]),
                 v=gs.Gaussians.zeros(case["n"]), cams=gs.cameras_tensor(_cameras(cams, seed)), nv=case["views"], dpose=dpose,
                 pm=torch.zeros_like(dpose), pv=torch.zeros_like(dpose), adam=gs.adam_config(),
                 step=torch.ones(1, dtype=torch.int32, device=DEV))
    elif kind == "spawn":
        w, h = case["width"], case["height"]
        img = _image(w, h, seed)
        render = img + 0.01 * torch.randn(img.shape, generator=_gen(seed + 1), device=DEV)
        render[:, :, :w // 2] = 0.0  # the left half of the frame is not reconstructed yet
        depth = 1.0 + 19.0 * torch.rand((h, w), generator=_gen(seed + 2), device=DEV)
        depth[torch.rand((h, w), generator=_gen(seed + 4), device=DEV) < 0.01] = 0.0
        cam = synth.camera(np.eye(3), np.array([0.1, -0.2, 0.3]), 1500.0 / 1920.0 * w, w, h)
        s.update(img=img, render=render, depth=depth, w=w, h=h, cam=gs.cameras_tensor([cam]), seed=int(seed) % (1 << 30),
                 out=gs.Spawned.alloc(w * h, w * h), ws=gs.workspace(gs.gs_spawn_workspace_size(w, h)))
    elif kind == "mlp":
        img, tg = _mlp_inputs(case, seed)
        w, h = case["width"], case["height"]
        n_p = gs.gs_mlp_patches(w, h)
        s.update(img=img, tg=tg, w=w, h=h, p=gs.MlpParams.from_numpy(_mlp_layers(seed)), m=gs.MlpParams.zeros(),
                 v=gs.MlpParams.zeros(), cfg=gs.mlp_config(tensor_path=1), loss=torch.zeros(1, device=DEV),
                 out=torch.zeros((n_p, 3), device=DEV), grads=torch.zeros(gs.gs_mlp_param_count(), device=DEV),
                 ws=gs.workspace(gs.gs_mlp_workspace_size(n_p)), step=torch.ones(1, dtype=torch.int32, device=DEV))
    elif kind == "ba":
        obs, cx, cy, fl, poses, pts = _ba_inputs(case, seed)
        s.update(obs=_f32(obs), cx=cx, cy=cy, start=[_f32(a) for a in (fl, poses, pts, [1e-5])],
                 x=[_f32(a) for a in (fl, poses, pts, [1e-5])], it=case["iterations"],
                 ws=gs.workspace(gs.gs_ba_workspace_size(case["frames"], case["points"])),
                 failed=torch.zeros(1, dtype=torch.int32, device=DEV))
    elif kind == "ba_pose":
        obs, cx, cy, fl, pose, pts = _ba_pose_inputs(case, seed)
        s.update(obs=_f32(obs), cx=cx, cy=cy, fl=_f32(fl), pts=_f32(pts), start=[_f32(pose), _f32([1e-5])],
                 x=[_f32(pose), _f32([1e-5])], it=case["iterations"],
                 ws=gs.workspace(gs.gs_ba_pose_workspace_size(case["points"])),
                 failed=torch.zeros(1, dtype=torch.int32, device=DEV))
    else:
        cams, feats, z = _guided_inputs(case, seed)
        s.update(cams=gs.cameras_tensor(cams), feats=feats, z=z, n=case["candidates"], depth=torch.empty_like(z),
                 nb=torch.empty(z.shape, dtype=torch.int32, device=DEV), corr=torch.empty_like(z))
    return s


def run(s):
    kind = s["kind"]
    if kind in ("raster", "view"):
        r = s["r"]
        img = r.forward(s["g"], s["cams"])
        out = dict(color=img.color, t_final=img.t_final, n_contrib=img.n_contrib)
        if kind == "view":
            return dict(out, depth=img.depth)
        grads, dpose = r.backward(s["g"], s["cams"], s["dL"])
        return dict(out, mean_opa=grads.mean_opa, scale=grads.scale, quat=grads.quat, sh=grads.sh, visible=grads.visible,
                    pose=dpose)
    if kind == "autograd":
        color, t_final = rasterize(*s["leaves"], s["cams"], s["sizes"], s["cfg"])
        grads = torch.autograd.grad(color, s["leaves"], s["dL"])
        return dict(zip(("mean_opa", "scale", "quat", "sh", "pose"), grads), color=color.detach(), t_final=t_final)
    if kind == "optim":
        p, m, v = s["p"], s["m"], s["v"]
        gs.gs_l1_loss(s["color"], s["target"], s["dL"], s["loss"], s["ws"])
        gs.gs_adam_step(p, s["grads"], m, v, s["adam"], 0, step_dev=s["step"])
        gs.gs_pose_step(s["cams"], s["nv"], s["dpose"], s["pm"], s["pv"], 1e-3, 1e-3, 0, step_dev=s["step"])
        gs.gs_counter_add(s["step"], 1)
        return dict(dL=s["dL"], loss=s["loss"], p=[p.mean_opa, p.scale, p.quat, p.sh], m=[m.mean_opa, m.scale, m.quat, m.sh],
                    v=[v.mean_opa, v.scale, v.quat, v.sh], cams=s["cams"].view(torch.float32), pm=s["pm"], pv=s["pv"])
    if kind == "spawn":
        o = s["out"]
        gs.gs_spawn_propose(s["img"], s["render"], s["depth"], s["w"], s["h"], s["cam"], 1.0, s["seed"], 3, o, s["ws"])
        return dict(mean_opa=o.g.mean_opa, scale=o.g.scale, quat=o.g.quat, sh=o.g.sh, pixel=o.pixel, count=o.count,
                    status=o.status, p_l=o.p_l, p_pen=o.p_pen, p_s=o.p_s)
    if kind == "mlp":
        gs.gs_mlp_train_step(s["p"], s["m"], s["v"], s["img"], s["w"], s["h"], s["tg"], s["cfg"], 0, s["loss"], s["ws"],
                             out=s["out"], grads=s["grads"], step_dev=s["step"])
        gs.gs_counter_add(s["step"], 1)
        return dict(loss=s["loss"], out=s["out"], grads=s["grads"])
    if kind == "ba":
        for a, b in zip(s["x"], s["start"]):
            a.copy_(b)
        fl, poses, pts, lam = s["x"]
        gs.gs_ba_lm(s["obs"], s["cx"], s["cy"], fl, poses, pts, lam, s["it"], s["ws"], s["failed"])
        return dict(fl=fl, poses=poses, points=pts, failed=s["failed"])
    if kind == "ba_pose":
        for a, b in zip(s["x"], s["start"]):
            a.copy_(b)
        gs.gs_ba_pose_lm(s["pts"], s["obs"], s["fl"], s["cx"], s["cy"], s["x"][0], s["x"][1], s["it"], s["ws"], s["failed"])
        return dict(pose=s["x"][0], failed=s["failed"])
    gs.gs_guided_depth(s["feats"], s["cams"], s["z"], n_cand=s["n"], depth=s["depth"], nb=s["nb"], corr=s["corr"])
    return dict(depth=s["depth"], nb=s["nb"], corr=s["corr"])


def work(case):
    kind = case["kind"]
    if kind in ("raster", "view", "autograd"):
        n, px = case["n"], sum(w * h for w, h in _sizes(case))
        # attribute rows in use read, colour, transmittance and contributor count written; backward: the loss
        # gradient read, the gradient rows written. About 30 Gaussians composite per pixel on the synthetic scenes
        # (20 flops forward, 63 backward each); a projection with its colour is about 400 flops per view, its
        # adjoint about 900.
        rows = 48 + 12 * (case["sh"] + 1) ** 2
        b, fl = n * rows + 20 * px, 30 * 20 * px + 400 * n * case["views"]
        if kind == "view":
            return {"bytes": b + 4 * px, "flops": fl}
        return {"bytes": b + 12 * px + 240 * n, "flops": fl + 30 * 63 * px + 900 * n * case["views"]}
    if kind == "optim":
        px = case["views"] * case["width"] * case["height"]
        return {"bytes": 36 * px + 0.78 * 7 * 240 * case["n"], "flops": 9 * px + 0.78 * 60 * 12 * case["n"]}
    if kind == "spawn":
        # image, render and depth read, three maps written, a row per spawn (about 7% of the pixels)
        px = case["width"] * case["height"]
        return {"bytes": (28 + 12 + 0.07 * 244) * px, "flops": 2 * 6 * 14 * px}
    if kind == "mlp":
        m = (case["width"] // 8) * (case["height"] // 8)
        return {"bytes": m * 64 * 12 + m * 28 + 7 * 4 * 58_400, "flops": 6 * m * (194 * 128 + 2 * 128 * 128 + 3 * 128)}
    if kind == "ba":
        p, f, nc = case["points"], case["frames"], 6 * case["frames"] - 5
        per = p * (nc * (nc + 1) * 3 + f * 300 + nc * 30) + nc ** 3 / 3
        return {"bytes": p * f * 8 + 32 * p, "flops": case["iterations"] * per}
    if kind == "ba_pose":
        return {"bytes": 24 * case["points"], "flops": case["iterations"] * case["points"] * 220}
    px = case["width"] * case["height"]
    return {"bytes": 2 * px * (2 * case["channels"]) + 16 * px, "flops": px * case["candidates"] * (8 * case["channels"] + 18)}


# ---------------------------------------------------------------------------
# the same values in 64 bits
# ---------------------------------------------------------------------------

def _sh_basis(deg, d):
    x, y, z = d.unbind(-1)
    c = lambda v: math.sqrt(v / math.pi)
    Y = [torch.full_like(x, 0.5 * c(1))]
    if deg > 0:
        Y += [-c(0.75) * y, c(0.75) * z, -c(0.75) * x]
    if deg > 1:
        Y += [c(15) / 2 * x * y, -c(15) / 2 * y * z, c(5) / 4 * (2 * z * z - x * x - y * y), -c(15) / 2 * x * z,
              c(15) / 4 * (x * x - y * y)]
    if deg > 2:
        Y += [-c(35 / 2) / 4 * y * (3 * x * x - y * y), c(105) / 2 * x * y * z, -c(21 / 2) / 4 * y * (4 * z * z - x * x - y * y),
              c(7) / 4 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c(21 / 2) / 4 * x * (4 * z * z - x * x - y * y),
              c(105) / 4 * z * (x * x - y * y), -c(35 / 2) / 4 * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _project64(leaves, xi, cam, deg, mip, dil):
    """EWA projection of every Gaussian in one view, differentiable in its parameters and the pose tangent xi."""
    mo, sc, q4, sh = leaves
    R, t = (torch.tensor(np.asarray(cam[k], np.float32).astype(np.float64), device=DEV) for k in ("R", "t"))
    fx, fy, cx, cy, W, H = (float(np.float32(cam[k])) for k in ("fx", "fy", "cx", "cy", "width", "height"))
    zero = torch.zeros((), dtype=torch.float64, device=DEV)
    ph = torch.stack([torch.stack([zero, -xi[5], xi[4]]), torch.stack([xi[5], zero, -xi[3]]), torch.stack([-xi[4], xi[3], zero])])
    Rp = R + ph @ R
    p = mo[:, :3] @ Rp.T + (t + ph @ t + xi[:3])
    x, y, z = p.unbind(-1)
    near = z > float(np.float32(0.2))
    zs = torch.where(near, z, torch.ones_like(z))
    w, a, b, c = (q4 / q4.norm(dim=1, keepdim=True)).unbind(-1)
    Rq = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b), 2 * (a * b + w * c), 1 - 2 * (a * a + c * c),
                      2 * (b * c - w * a), 2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], -1).view(-1, 3, 3)
    T = Rp @ (Rq * torch.exp(sc[:, None, :3]))
    lx, ly = 0.65 * W / fx, 0.65 * H / fy
    tx, ty = torch.clamp(x / zs, -lx, lx), torch.clamp(y / zs, -ly, ly)
    M0 = fx / zs[:, None] * (T[:, 0] - tx[:, None] * T[:, 2])
    M1 = fy / zs[:, None] * (T[:, 1] - ty[:, None] * T[:, 2])
    Sa, Sb, Sc = (M0 * M0).sum(-1) + dil, (M0 * M1).sum(-1), (M1 * M1).sum(-1) + dil
    det = Sa * Sc - Sb * Sb
    o = torch.sigmoid(mo[:, 3])
    if mip:
        o = o * torch.sqrt(torch.clamp(torch.linalg.cross(M0, M1).square().sum(-1) / det, min=1e-6))
    u, v = fx * x / zs + cx, fy * y / zs + cy
    dirs = mo[:, :3] + (R.T @ t)
    dirs = dirs / dirs.norm(dim=1, keepdim=True)
    nc = (deg + 1) ** 2
    rgb = torch.clamp(0.5 + torch.einsum("nk,nkc->nc", _sh_basis(deg, dirs), sh[:, :3 * nc].reshape(-1, nc, 3)), min=0.0)
    with torch.no_grad():
        mid = 0.5 * (Sa + Sc)
        r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt(torch.clamp(mid * mid - det, min=0.1))))
        gx, gy = -(-int(W) // 16), -(-int(H) // 16)
        lim = lambda e, m: torch.clamp(torch.nan_to_num(torch.floor(e)), 0, m)
        x0, y0, x1, y1 = lim((u - r) / 16, gx), lim((v - r) / 16, gy), lim((u + r + 15) / 16, gx), lim((v + r + 15) / 16, gy)
        keep = near & (det > 0) & (o >= float(np.float32(1 / 255)))
        # only tiles where the Gaussian's alpha can reach 1/255: the others add nothing
        ta = 2 * torch.log(torch.clamp(o * 255, min=1.0))
        hx, hy = torch.sqrt(ta * Sa) + 0.05, torch.sqrt(ta * Sc) + 0.05
        x0, y0 = torch.maximum(x0, lim((u - hx) / 16, gx)), torch.maximum(y0, lim((v - hy) / 16, gy))
        x1, y1 = torch.minimum(x1, lim((u + hx) / 16 + 1, gx)), torch.minimum(y1, lim((v + hy) / 16 + 1, gy))
        keep &= (x1 > x0) & (y1 > y0)
        rect = torch.stack([x0, y0, x1, y1], -1).long()
    return torch.stack([u, v, Sc / det, -Sb / det, Sa / det, o], -1), rgb, z, rect, keep


def _composite64(items, rgb, z, rect, keep, W, H, dL, back):
    """Front-to-back compositing of one view; with back, the gradients of sum(color * dL) at the items and colours."""
    gx, gy = -(-W // 16), -(-H // 16)
    idx = torch.nonzero(keep)[:, 0]
    idx = idx[torch.sort(z[idx].float(), stable=True).indices]
    r = rect[idx]
    wx = r[:, 2] - r[:, 0]
    cnt = wx * (r[:, 3] - r[:, 1])
    rep = torch.repeat_interleave(torch.arange(len(idx), device=DEV), cnt)
    loc = torch.arange(len(rep), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[rep]
    tile = (r[rep, 1] + loc // wx[rep]) * gx + r[rep, 0] + loc % wx[rep]
    tile, order = torch.sort(tile, stable=True)
    who = idx[rep[order]]
    n_t = torch.bincount(tile, minlength=gx * gy)
    start = torch.cumsum(n_t, 0) - n_t
    color = torch.zeros((3, gy * 16, gx * 16), dtype=torch.float64, device=DEV)
    tfin, dep = torch.ones_like(color[0]), torch.zeros_like(color[0])
    dLp = torch.zeros_like(color)
    dLp[:, :H, :W] = dL.view(3, H, W).double()
    g_it, g_rgb = torch.zeros_like(items), torch.zeros_like(rgb)
    ln, tiles = torch.sort(n_t, descending=True)
    ln = ln.tolist()
    ly, lx = torch.meshgrid(torch.arange(16, device=DEV), torch.arange(16, device=DEV), indexing="ij")
    ly, lx = ly.reshape(-1), lx.reshape(-1)
    at = 0
    while at < len(ln) and ln[at] > 0:
        L = ln[at]
        B = max(1, min(len(ln) - at, (1 << 26) // (256 * L)))
        tb = tiles[at:at + B]
        at += B
        k = start[tb][:, None] + torch.arange(L, device=DEV)
        live = torch.arange(L, device=DEV) < n_t[tb][:, None]
        sel = who[torch.where(live, k, 0)]
        py, px = (tb // gx * 16)[:, None] + ly, (tb % gx * 16)[:, None] + lx
        with torch.enable_grad():
            it, cc = items[sel].requires_grad_(back), rgb[sel].requires_grad_(back)
            u, v, A, Bc, C, o = (e[..., None] for e in it.unbind(-1))
            dx, dy = px[:, None, :] + 0.5 - u, py[:, None, :] + 0.5 - v
            pw = -0.5 * (A * dx * dx + C * dy * dy) - Bc * dx * dy
            al = torch.clamp(o * torch.exp(pw), max=float(np.float32(0.99)))
            ok = (pw <= 0) & (al >= float(np.float32(1 / 255))) & live[..., None]
            with torch.no_grad():
                T = torch.cumprod(torch.where(ok, 1 - al, 1.0), 1)
                ok &= T >= float(np.float32(1e-4))
            al = torch.where(ok, al, 0.0)
            T = torch.cumprod(1 - al, 1)
            Te = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
            wgt = al * Te
            col = torch.einsum("blp,blc->bcp", wgt, cc)
            if back:
                gi, gc = torch.autograd.grad((col * dLp[:, py, px].transpose(0, 1)).sum(), (it, cc))
                g_it.index_put_((sel,), gi, accumulate=True)
                g_rgb.index_put_((sel,), gc, accumulate=True)
        color[:, py, px] = col.detach().transpose(0, 1)
        tfin[py, px] = T[:, -1].detach()
        dep[py, px] = torch.einsum("blp,bl->bp", wgt.detach(), z[sel])
    return color[:, :H, :W].reshape(-1), tfin[:H, :W].reshape(-1), dep[:H, :W].reshape(-1), g_it, g_rgb


def _exact_raster(case, seed):
    kind, V = case["kind"], case["views"]
    # more than about 20 seconds: the largest renders
    if case["n"] * V > 8_000_000:
        return None
    leaves = [t.double().requires_grad_(True) for t in _gaussians(case, seed)]
    cams, sizes = _cameras(case, seed), _sizes(case)
    n_pix = sum(w * h for w, h in sizes)
    dL = _loss_gradient(n_pix, seed)
    back = kind != "view"
    dil, mip = (float(np.float32(0.1)), True) if kind == "autograd" else (float(np.float32(0.3)), False)
    grads = [torch.zeros_like(t) for t in leaves]
    pose = torch.zeros((V, 6), dtype=torch.float64, device=DEV)
    colors, tfins, deps, base = [], [], [], 0
    for v, (cam, (W, H)) in enumerate(zip(cams, sizes)):
        xi = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
        items, rgb, z, rect, keep = _project64(leaves, xi, cam, case["sh"], mip, dil)
        c, t, d, gi, gc = _composite64(items.detach(), rgb.detach(), z.detach(), rect, keep, W, H, dL[3 * base:3 * (base + W * H)], back)
        base += W * H
        colors.append(c)
        tfins.append(t)
        deps.append(d)
        if back:
            got = torch.autograd.grad((items, rgb), (*leaves, xi), (gi * keep[:, None], gc * keep[:, None]))
            for a, b in zip(grads, got):
                a += torch.nan_to_num(b)
            pose[v] = got[4]
    out = dict(color=torch.cat(colors), t_final=torch.cat(tfins))
    if kind == "view":
        return dict(out, n_contrib=None, depth=torch.cat(deps))
    out.update(zip(("mean_opa", "scale", "quat", "sh"), grads), pose=pose)
    if kind == "raster":
        out.update(n_contrib=None, visible=None)
    return out


def _exact_optim(case, seed):
    color, target, p, g, visible, dpose = _optim_inputs(case, seed)
    d = color.double() - target.double()
    b1, b2, eps = (float(np.float32(x)) for x in (0.9, 0.999, 1e-15))
    f = lambda x: float(np.float32(x))
    rates = [torch.full((k,), f(r), dtype=torch.float64, device=DEV) for k, r in ((4, 1.6e-4), (4, 5e-3), (4, 1e-3), (48, 1.25e-4))]
    rates[0][3] = f(0.05)
    rates[1][3] = 0.0
    rates[3][:3] = f(2.5e-3)
    vis = (visible > 0)[:, None]
    m = [torch.where(vis, (1 - b1) * x.double(), 0.0) for x in g]
    v = [torch.where(vis, (1 - b2) * x.double() ** 2, 0.0) for x in g]
    step = lambda mm, vv: (mm / (1 - b1)) / (torch.sqrt(vv / (1 - b2)) + eps)
    p = [torch.where(vis, x.double() - r * step(mm, vv), x.double()) for x, r, mm, vv in zip(p, rates, m, v)]
    pm, pv = (1 - b1) * dpose.double(), (1 - b2) * dpose.double() ** 2
    delta = (-f(1e-3) * step(pm, pv)).cpu().numpy()
    raw = gs.cameras_tensor(_cameras(dict(case, scene="path"), seed)).view(torch.float32).view(-1, 18).double().cpu().numpy()
    for i, row in enumerate(raw):
        T = np.eye(4)
        T[:3, :3], T[:3, 3] = row[:9].reshape(3, 3), row[9:12]
        T = _exp_se3(delta[i]) @ T
        row[:9], row[9:12] = T[:3, :3].reshape(9), T[:3, 3]
    return dict(dL=torch.sign(d) / d.numel(), loss=d.abs().mean().reshape(1), p=p, m=m, v=v,
                cams=torch.tensor(raw).reshape(-1), pm=pm, pv=pv)


def _exact_spawn(case, seed):
    st = prepare(case, seed)
    t = np.arange(-3, 4, dtype=np.float64)
    r2 = t[:, None] ** 2 + t[None, :] ** 2
    k = (r2 - 2) * np.exp(-r2 / 2) / (2 * np.pi)
    k = torch.tensor(k - k.mean(), device=DEV)
    res = []
    for a in (st["img"], st["render"]):
        a = torch.nn.functional.pad(a.double()[None], (3, 3, 3, 3), mode="replicate")[0]
        acc = torch.zeros((3, case["height"], case["width"]), dtype=torch.float64, device=DEV)
        for j in range(7):
            for i in range(7):
                acc += k[j, i] * a[:, j:j + case["height"], i:i + case["width"]]
        res.append(torch.clamp(acc.square().sum(0).sqrt(), max=1.0).reshape(-1))
    # which pixels spawn hangs on draws against p_s: the rows have no value that a rounding could not move
    return dict(mean_opa=None, scale=None, quat=None, sh=None, pixel=None, count=None, status=None, p_l=res[0], p_pen=res[1],
                p_s=torch.clamp(res[0] - res[1], min=0.0))


def _exact_mlp(case, seed):
    img, tg = _mlp_inputs(case, seed)
    w, h = case["width"], case["height"]
    nx, ny = w // 8, h // 8
    x = img[:, :ny * 8, :nx * 8].double().view(3, ny, 8, nx, 8).permute(1, 3, 0, 2, 4).reshape(ny * nx, 192)
    iy, ix = torch.meshgrid(torch.arange(ny, device=DEV).double(), torch.arange(nx, device=DEV).double(), indexing="ij")
    pos = torch.stack([2 * (ix + 0.5) / nx - 1, 2 * (iy + 0.5) / ny - 1], -1).view(-1, 2)
    hid = torch.cat([x, pos], 1)
    params = [torch.tensor(np.asarray(a, np.float32), device=DEV).double().requires_grad_(True) for l in _mlp_layers(seed) for a in l]
    for l in range(4):
        hid = torch.nn.functional.linear(hid, params[2 * l], params[2 * l + 1])
        if l < 3:
            hid = torch.nn.functional.gelu(hid)
    tg = tg.double()
    loss = (torch.nn.functional.softplus(hid[:, 0]) - tg[:, 0] * hid[:, 0] + tg[:, 3] * ((hid[:, 1] - tg[:, 1]).abs() + (hid[:, 2] - tg[:, 2]).abs())).mean()
    grads = torch.autograd.grad(loss, params)
    return dict(loss=loss.detach().reshape(1), out=hid.detach(), grads=torch.cat([g.reshape(-1) for g in grads]))


def _robust(e, delta=2.0):
    """Which residual norms are kept (median + 4 MAD, lower medians) and their Huber weights."""
    med = torch.sort(e.reshape(-1)).values[(e.numel() - 1) // 2]
    mad = torch.sort((e - med).abs().reshape(-1)).values[(e.numel() - 1) // 2]
    return (e <= med + 4 * mad).double()


def _robust_cost(e, keep, delta=2.0):
    return (keep * torch.where(e <= delta, 0.5 * e * e, delta * (e - 0.5 * delta))).sum()


def _exact_ba(case, seed):
    pose_only = case["kind"] == "ba_pose"
    obs, cx, cy, fl, poses, pts = (_ba_pose_inputs if pose_only else _ba_inputs)(case, seed)
    t64 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64)
    M = case["points"]
    F = 1 if pose_only else case["frames"]
    obs, fl = t64(obs).view(M, F, 2), float(fl[0])
    poses = [np.vstack([np.hstack([r[:9].reshape(3, 3), r[9:, None]]), [[0, 0, 0, 1]]]) for r in poses.astype(np.float64).reshape(F, 12)]
    X, lam = t64(pts[:, :3]), float(np.float32(1e-5))
    nc = 6 if pose_only else 6 * (F - 1) + 1

    def look(fl, poses, X):
        R, t = t64(np.stack([p[:3, :3] for p in poses])), t64(np.stack([p[:3, 3] for p in poses]))
        q = torch.einsum("fij,pj->pfi", R, X) + t
        r = fl * q[..., :2] / q[..., 2:] + t64([cx, cy]) - obs
        return R, q, r, r.norm(dim=-1)

    for _ in range(case["iterations"]):
        R, q, r, e = look(fl, poses, X)
        keep = _robust(e)
        wgt = keep * torch.where(e <= 2.0, 1.0, 2.0 / torch.clamp(e, min=1e-300))
        cost = _robust_cost(e, keep)
        x, y, z = q.unbind(-1)
        zero = torch.zeros_like(x)
        jq = torch.stack([torch.stack([fl / z, zero, -fl * x / z ** 2], -1), torch.stack([zero, fl / z, -fl * y / z ** 2], -1)], -2)
        sk = torch.stack([torch.stack([zero, z, -y], -1), torch.stack([-z, zero, x], -1), torch.stack([y, -x, zero], -1)], -2)
        jp = torch.cat([jq, jq @ sk], -1)  # d residual / d (rho, phi)
        Jc = torch.zeros((M, F, 2, nc), dtype=torch.float64)
        if pose_only:
            Jc[:, 0] = jp[:, 0]
        else:
            for f in range(1, F):
                Jc[:, f, :, 6 * (f - 1):6 * f] = jp[:, f]
            Jc[..., -1] = q[..., :2] / q[..., 2:]
        wJ = Jc * wgt[..., None, None]
        Hcc = torch.einsum("pfka,pfkb->ab", wJ, Jc)
        gc = torch.einsum("pfka,pfk->a", wJ, r)
        Hd = Hcc + torch.diag(lam * Hcc.diagonal() + 1e-9)
        if pose_only:
            dc, dX = torch.linalg.solve(Hd, -gc), None
        else:
            Jx = jq @ R
            wx = Jx * wgt[..., None, None]
            Hpp = torch.einsum("pfka,pfkb->pab", wx, Jx)
            gp = torch.einsum("pfka,pfk->pa", wx, r)
            K = torch.einsum("pfka,pfkb->pab", wJ, Jx)
            Hpp = Hpp + torch.diag_embed(lam * Hpp.diagonal(dim1=1, dim2=2) + 1e-9)
            Hi = torch.linalg.inv(Hpp)
            S = Hd - torch.einsum("pai,pij,pbj->ab", K, Hi, K)
            dc = torch.linalg.solve(S, -gc + torch.einsum("pai,pij,pj->a", K, Hi, gp))
            dX = -torch.einsum("pij,pj->pi", Hi, gp + torch.einsum("pai,a->pi", K, dc))
        d = dc.numpy()
        if pose_only:
            fl_t, poses_t, X_t = fl, [_exp_se3(d) @ poses[0]], X
        else:
            fl_t, poses_t, X_t = fl + d[-1], poses[:1] + [_exp_se3(d[6 * (f - 1):6 * f]) @ poses[f] for f in range(1, F)], X + dX
        better = bool(_robust_cost(look(fl_t, poses_t, X_t)[3], keep) < cost)
        if better:
            fl, poses, X = fl_t, poses_t, X_t
        lam = min(1e10, max(1e-12, lam / 2 if better else lam * 2))
    rows = t64(np.stack([np.concatenate([p[:3, :3].reshape(9), p[:3, 3]]) for p in poses]))
    if pose_only:
        return dict(pose=rows.reshape(12), failed=None)
    return dict(fl=t64([fl]), poses=rows, points=torch.cat([X, torch.zeros((M, 1), dtype=torch.float64)], 1), failed=None)


def _exact_guided(case, seed):
    cams, feats, zm = _guided_inputs(case, seed)
    W, H, J, n = case["width"], case["height"], case["neighbours"], case["candidates"]
    t64 = lambda a: torch.tensor(np.asarray(a, np.float32).astype(np.float64), device=DEV)
    ci, win = cams[0], float(np.float32(0.1))
    y, x = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(), indexing="ij")
    ray = torch.stack([(x + 0.5 - ci["cx"]) / ci["fx"], (y + 0.5 - ci["cy"]) / ci["fy"], torch.ones_like(x)], -1).view(-1, 3)
    z = zm.double().view(-1)
    ok = z > 0
    dc = 1.0 / torch.where(ok, z, 1.0)
    lo, hi = torch.clamp(dc - win, min=0.0), dc + win
    rel = []
    for c in cams[1:]:
        R = t64(c["R"]) @ t64(ci["R"]).T
        rel.append((R, t64(c["t"]) - R @ t64(ci["t"])))

    def at(j, a, d):
        p = a + d[..., None] * rel[j][1]
        c = cams[1 + j]
        return c["fx"] * p[..., 0] / p[..., 2] + c["cx"] - 0.5, c["fy"] * p[..., 1] / p[..., 2] + c["cy"] - 0.5, p[..., 2]

    best, nb = torch.full_like(z, -1.0), torch.full_like(z, -1, dtype=torch.long)
    for j in range(J):
        a = ray @ rel[j][0].T
        e = [at(j, a, d) for d in (lo, hi)]
        use = ok.clone()
        for sx, sy, sz in e:
            use &= (sz > 0) & (sx >= 0) & (sx <= W - 1) & (sy >= 0) & (sy <= H - 1)
        ln = torch.where(use, torch.hypot(e[0][0] - e[1][0], e[0][1] - e[1][1]), -1.0)
        nb = torch.where(ln > best, j, nb)
        best = torch.maximum(best, ln)
    depth, corr = z.clone(), torch.zeros_like(z)
    ref = feats[0].view(H * W, -1)
    for j in range(J):
        for idx in torch.nonzero(nb == j)[:, 0].split(200_000):
            a, f0, fj = ray[idx] @ rel[j][0].T, ref[idx].double(), feats[1 + j].view(H * W, -1)
            step = (hi[idx] - lo[idx]) / (n - 1)
            Cs = []
            for k in range(n):
                sx, sy, _ = at(j, a, lo[idx] + step * k)
                x0, y0 = torch.clamp(sx.floor(), 0, W - 2), torch.clamp(sy.floor(), 0, H - 2)
                wx, wy, cell = sx - x0, sy - y0, (y0 * W + x0).long()
                dot = lambda o: (f0 * fj[cell + o].double()).sum(1)
                Cs.append((1 - wx) * (1 - wy) * dot(0) + wx * (1 - wy) * dot(1) + (1 - wx) * wy * dot(W) + wx * wy * dot(W + 1))
            Cs = torch.stack(Cs, 1)
            cb, kb = Cs.max(1)
            cm, cp = (Cs.gather(1, torch.clamp(kb + s, 0, n - 1)[:, None])[:, 0] for s in (-1, 1))
            den = cm - 2 * cb + cp
            mid = (kb > 0) & (kb < n - 1) & (den < 0)
            ds = lo[idx] + step * (kb + torch.where(mid, (cm - cp) / (2 * torch.where(mid, den, 1.0)), 0.0))
            good = ds > 0
            depth[idx] = torch.where(good, 1 / torch.where(good, ds, 1.0), z[idx])
            corr[idx] = torch.where(good, cb, 0.0)
    return dict(depth=depth.view(H, W), nb=None, corr=corr.view(H, W))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("raster", "view", "autograd"):
        return _exact_raster(case, seed)
    if kind in ("ba", "ba_pose"):
        return _exact_ba(case, seed)
    return {"optim": _exact_optim, "spawn": _exact_spawn, "mlp": _exact_mlp, "guided": _exact_guided}[kind](case, seed)
