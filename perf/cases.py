"""Timed cases of the library's main paths: rendering, the differentiable render with its
adjoint, whole mapping iterations, the losses, and the learned initializer, each through the
calls a mapping program makes.  Sizes are those of the repository's own workloads and tests
(160x120 cloud, ragged 157x91 pyramid, 640x480 and 1200x680 rooms, the batched keyframes) and
of the ranges between them.

A case is a flat dict.  kind:
  splat   pyramid_splat (torch.autograd.Function): images, and the gradients of every parameter
          for a given upstream gradient
  render  a novel view: set_cameras + PyramidRasterizer.forward, no gradient
  step    one MappingStep iteration (render, loss, adjoint, Adam), eager or as a graph replay
  loss    PyramidRasterizer.loss alone: terms, dL/dimage, decoder gradient
  insert  the learned insertion of B pixels of a keyframe: heuristic init, patch features,
          network, application of its outputs
  train   one training step of the learned initializer on a batch
"""
import ctypes
import math

import numpy as np
import torch

from paper_2412_01217_gb300 import (LossConfig, MappingStep, PyramidRasterizer, RenderConfig, build_pyramid,
                                    pyramid_splat)
from paper_2412_01217_gb300._lib import call
from paper_2412_01217_gb300.learned_init import MLPInit
from paper_2412_01217_gb300.splat import DEFAULT_LR, camera_struct, gaussians_struct

# Launch shapes: the package's default, and the ones its autotuner picks on the room workloads.
CONFIGS = {
    "default": dict(),
    "tile8": dict(tile_w=8, tile_h=8, batch=64, batch_bwd=16, pixels_per_thread=1, pixels_per_thread_bwd=1),
    "half": dict(tile_w=8, tile_h=8, batch=64, batch_bwd=16, pixels_per_thread=1, pixels_per_thread_bwd=1,
                 half_masks=True),
    "half2": dict(tile_w=8, tile_h=8, batch=64, batch_bwd=16, pixels_per_thread=1, pixels_per_thread_bwd=1,
                  half_masks=True, half_tile_fwd=True),
    "wide": dict(tile_w=32, tile_h=8, batch=128, pixels_per_thread=1, pixels_per_thread_bwd=1),
}
# contributing Gaussians per pixel of a finished room map (about; for the flop counts only)
DEPTH_COMPLEXITY = 40


def listed():
    return [
        # the smallest call: a 2000-Gaussian cloud at 160x120, where launches and host time count
        dict(name="splat_160x120", kind="splat", scene="cloud", N=2000, C=8, W=160, H=120, kf=1, levels=1, sh=0,
             sem_sh=False, iso=False, cfg="default"),
        # ragged sizes at every level, view-dependent colour and semantics of degree 3
        dict(name="splat_157x91_sh3", kind="splat", scene="cloud", N=800, C=4, W=157, H=91, kf=2, levels=3, sh=3,
             sem_sh=True, iso=False, cfg="default"),
        # the Eq. 2 projection on a small room, two keyframes (preview quality mapping)
        dict(name="splat_320x180_iso", kind="splat", scene="room", N=30_000, C=16, W=320, H=180, kf=2, levels=3,
             sh=0, sem_sh=False, iso=True, cfg="tile8"),
        # evaluation of a map: one 640x480 novel view, default launch shape
        dict(name="render_640x480", kind="render", scene="room", N=200_000, C=16, W=640, H=480, levels=1, iso=False,
             cfg="default"),
        # an ordinary mapping iteration run eagerly (the first ones of every keyframe are)
        dict(name="step_320x180_eager", kind="step", scene="room", N=30_000, C=16, K=32, decoder=True, W=320, H=180,
             kf=1, kf_small=0, levels=3, cfg="default", graph=False),
        # the Replica-like iteration: one 1200x680 keyframe x 3 levels, replayed as a graph
        dict(name="step_1200x680", kind="step", scene="room", N=300_000, C=16, K=32, decoder=True, W=1200, H=680,
             kf=1, kf_small=0, levels=3, cfg="half", graph=True),
        # the ScanNet-like iteration: a dense map, class logits without a decoder
        dict(name="step_640x480_1m", kind="step", scene="room", N=1_000_000, C=40, K=40, decoder=False, W=640, H=480,
             kf=1, kf_small=0, levels=4, cfg="half2", graph=True),
        # the batched iteration: 4 x 1200x680 and 4 x 640x480 keyframes x 3 levels in one launch
        # per kernel (the largest)
        dict(name="step_batched", kind="step", scene="room", N=500_000, C=16, K=32, decoder=True, W=1200, H=680, kf=4,
             kf_small=4, levels=3, cfg="half2", graph=True),
        # the losses alone: cross-entropy through the decoder, and L1 + D-SSIM on a semantic
        # colour image at an odd size
        dict(name="loss_ce_1200x680", kind="loss", mode="ce", C=16, K=32, decoder=True, W=1200, H=680, kf=1, levels=3),
        dict(name="loss_paper_637x477", kind="loss", mode="paper", C=4, K=4, decoder=False, W=637, H=477, kf=1,
             levels=3),
        # learned insertion of one keyframe's new Gaussians, and one training step
        dict(name="insert_5000", kind="insert", B=5000, C=16, K=32, W=1200, H=680),
        dict(name="train_16384", kind="train", B=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["splat", "splat", "splat", "render", "step", "step", "loss", "loss", "insert", "train"])
    if kind == "insert":
        W = _log_int(rng, 160, 1200)
        return dict(kind=kind, B=_log_int(rng, 100, 20_000), C=16, K=32, W=W, H=max(91, int(W * rng.uniform(0.55, 0.8))))
    if kind == "train":
        return dict(kind=kind, B=128 * _log_int(rng, 4, 256))
    W = _log_int(rng, 100, 1200)
    H = max(75, int(W * rng.uniform(0.5, 0.8)))
    levels = rng.randint(1, 4)
    if kind == "loss":
        mode = rng.choice(["ce", "paper"])
        C, K, dec = rng.choice([(16, 32, True), (32, 32, True), (16, 16, True), (8, 8, True), (40, 40, False)]
                               if mode == "ce" else [(4, 4, False), (8, 8, False)])
        return dict(kind=kind, mode=mode, C=C, K=K, decoder=dec, W=W, H=H, kf=rng.randint(1, 2), levels=levels)
    if kind == "render":
        return dict(kind=kind, scene=rng.choice(["cloud", "room"]), N=_log_int(rng, 500, 400_000),
                    C=rng.choice([4, 8, 16, 32, 40]), W=W, H=H, levels=levels, iso=rng.random() < 0.25,
                    cfg=rng.choice(sorted(CONFIGS)))
    if kind == "step":
        C, K, dec = rng.choice([(16, 32, True), (32, 32, True), (40, 40, False), (8, 8, False)])
        return dict(kind=kind, scene="room", N=_log_int(rng, 5_000, 400_000), C=C, K=K, decoder=dec, W=W, H=H,
                    kf=rng.randint(1, 2), kf_small=rng.randint(0, 1), levels=levels, cfg=rng.choice(sorted(CONFIGS)),
                    graph=rng.random() < 0.5)
    sh = rng.choice([0, 0, 1, 2, 3])
    return dict(kind=kind, scene=rng.choice(["cloud", "room"]), N=_log_int(rng, 500, 100_000),
                C=rng.choice([4, 8, 16, 32, 40]), W=W, H=H, kf=rng.randint(1, 3), levels=levels, sh=sh,
                sem_sh=sh > 0 and rng.random() < 0.3, iso=rng.random() < 0.25, cfg=rng.choice(sorted(CONFIGS)))


# ------------------------------------------------------------------------------------------
# Scenes: a 6 x 5 x 3 m room with 20 boxes (Gaussians on its surfaces, ray-cast frames), and a
# random cloud in front of the camera.  Everything from the seed, on the GPU.
# ------------------------------------------------------------------------------------------

ROOM = (6.0, 5.0, 3.0)
DEV = "cuda"


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1_000_003 + salt * 7919) % (1 << 62))


def _boxes(seed):
    """(20, 3) lower and upper corners of boxes resting on the floor."""
    u = torch.rand(20, 6, generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
    size = 0.2 + 0.8 * u[:, :3]
    lo = torch.zeros(20, 3, device=DEV, dtype=torch.float64)
    for a in range(2):
        lo[:, a] = 0.1 + u[:, 3 + a] * (ROOM[a] - size[:, a] - 0.2)
    return lo, lo + size


def _texture(p, sid, seed):
    """RGB of the points p (n, 3) on surface sid (n): a base colour per surface, checkers."""
    base = 0.15 + 0.75 * torch.rand(6 + 20 * 6, 3, generator=_gen(seed, 2), device=DEV, dtype=torch.float64)
    s = p.sum(-1, keepdim=True)
    ch = 0.55 + 0.2 * (torch.floor(p / 0.5).sum(-1, keepdim=True) % 2) \
        + 0.12 * (torch.floor(p / 0.17).sum(-1, keepdim=True) % 2) + 0.06 * torch.sin(40 * s)
    return (base[sid] * ch).clamp(0, 1)


def _label(sid, K):
    return torch.where(sid < 6, sid, 6 + (sid - 6) // 6) % K


def _room_gaussians(N, C, seed):
    g = _gen(seed, 3)
    lo, hi = _boxes(seed)
    size = hi - lo
    room = torch.tensor(ROOM, device=DEV, dtype=torch.float64)
    o = torch.cat([torch.zeros(1, 3, device=DEV, dtype=torch.float64), lo])
    e = torch.cat([room[None], size])
    # faces 2 a (low side) and 2 a + 1 (high side) of axis a of the room (0) and the boxes
    area = torch.stack([e[:, 1] * e[:, 2], e[:, 0] * e[:, 2], e[:, 0] * e[:, 1]], 1).repeat_interleave(2, 1)
    area[1:, 4] = 0  # a box stands on the floor
    sid = torch.multinomial(area.reshape(-1), N, replacement=True, generator=g)
    b, face = sid // 6, sid % 6
    p = torch.rand(N, 3, generator=g, device=DEV, dtype=torch.float64)
    ax = (face // 2)[:, None]
    p.scatter_(1, ax, (face % 2).double()[:, None])
    mean = o[b] + p * e[b] + 0.002 * torch.randn(N, 3, generator=g, device=DEV, dtype=torch.float64)
    q = torch.randn(N, 4, generator=g, device=DEV)
    return dict(mean=mean, log_scale=math.log(0.005) + math.log(10) * torch.rand(N, 3, generator=g, device=DEV),
                quat=q / q.norm(dim=1, keepdim=True),
                opacity_logit=2 + 0.5 * torch.randn(N, generator=g, device=DEV),
                rgb=_texture(o[b] + p * e[b], sid, seed), sem=0.5 * torch.randn(N, C, generator=g, device=DEV))


def _cloud_gaussians(N, C, seed):
    g = _gen(seed, 3)
    u = torch.rand(N, 3, generator=g, device=DEV)
    mean = torch.stack([2 * u[:, 0] - 1, 2 * u[:, 1] - 1, 1 + 3 * u[:, 2]], 1)
    q = torch.randn(N, 4, generator=g, device=DEV)
    return dict(mean=mean, log_scale=math.log(0.005) + math.log(10) * torch.rand(N, 3, generator=g, device=DEV),
                quat=q / q.norm(dim=1, keepdim=True), opacity_logit=torch.randn(N, generator=g, device=DEV),
                rgb=torch.rand(N, 3, generator=g, device=DEV), sem=torch.randn(N, C, generator=g, device=DEV))


def _gaussians(case, seed):
    g = (_room_gaussians if case["scene"] == "room" else _cloud_gaussians)(case["N"], case["C"], seed)
    if case.get("sh"):
        K = (case["sh"] + 1) ** 2 - 1
        l = torch.floor(torch.sqrt(torch.arange(1, K + 1, device=DEV).double()))[None, :, None]
        g["sh"] = 0.2 / l * torch.randn(case["N"], K, 3, generator=_gen(seed, 4), device=DEV)
        if case["sem_sh"]:
            g["sem_sh"] = 0.5 / l * torch.randn(case["N"], K, case["C"], generator=_gen(seed, 5), device=DEV)
    return {k: v.float().contiguous() for k, v in g.items()}


def _cameras(case, seed):
    """kf cameras of size W x H (and kf_small of 8/15 of it): inside the room at seeded places
    and headings, or in front of the cloud."""
    rng = np.random.default_rng(seed + 17)
    cams = []
    for i in range(case.get("kf", 1) + case.get("kf_small", 0)):
        W, H = case["W"], case["H"]
        if i >= case.get("kf", 1):
            W, H = max(16, W * 8 // 15), max(16, H * 8 // 15)
        f = W * (150 / 160 if case.get("scene") == "cloud" else 0.5)
        if case.get("scene") == "cloud":
            a = rng.uniform(-0.1, 0.1)
            R = np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]])
            t = rng.uniform(-0.1, 0.1, 3)
        else:
            c = np.array([rng.uniform(1, ROOM[0] - 1), rng.uniform(1, ROOM[1] - 1), rng.uniform(1.3, 1.9)])
            yaw, pitch = rng.uniform(0, 2 * math.pi), rng.uniform(-0.35, -0.15)
            fw = np.array([math.cos(yaw) * math.cos(pitch), math.sin(yaw) * math.cos(pitch), math.sin(pitch)])
            right = np.array([fw[1], -fw[0], 0.0])
            right /= np.linalg.norm(right)
            R = np.stack([right, np.cross(fw, right), fw])
            t = -R @ c
        r32 = lambda x: np.asarray(x, np.float32).astype(np.float64)
        cams.append(dict(W=W, H=H, fx=float(np.float32(f)), fy=float(np.float32(f)), cx=W / 2 - 0.5, cy=H / 2 - 0.5,
                         R_cw=r32(R), t_cw=r32(t)))
    return cams


def _frame(cam, K, seed):
    """Ray-cast level-0 frame of the room: rgb (3, H, W), depth (H, W) with 2 % missing, label."""
    W, H = cam["W"], cam["H"]
    R = torch.tensor(cam["R_cw"], device=DEV)
    c = -(R.T @ torch.tensor(cam["t_cw"], device=DEV))
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(), indexing="ij")
    d = torch.stack([(xs - cam["cx"]) / cam["fx"], (ys - cam["cy"]) / cam["fy"], torch.ones_like(xs)], -1)
    d = d.reshape(-1, 3) @ R
    d = torch.where(d.abs() < 1e-9, torch.full_like(d, 1e-9), d)
    room = torch.tensor(ROOM, device=DEV, dtype=torch.float64)
    t, ax = torch.maximum(-c / d, (room - c) / d).min(1)
    sid = 2 * ax + (d.gather(1, ax[:, None])[:, 0] > 0)
    for k, (lo, hi) in enumerate(zip(*_boxes(seed))):
        a, b = (lo - c) / d, (hi - c) / d
        t0, ax = torch.minimum(a, b).max(1)
        hit = (t0 <= torch.maximum(a, b).min(1)[0]) & (t0 > 1e-6) & (t0 < t)
        t = torch.where(hit, t0, t)
        sid = torch.where(hit, 6 + 6 * k + 2 * ax + (d.gather(1, ax[:, None])[:, 0] < 0), sid)
    rgb = _texture(c + t[:, None] * d, sid, seed)
    depth = t + 0.01 * torch.randn(t.shape, generator=_gen(seed, 6), device=DEV, dtype=torch.float64)
    depth = torch.where(torch.rand(t.shape, generator=_gen(seed, 7), device=DEV) < 0.02, torch.zeros_like(t), depth)
    return dict(rgb=rgb.T.reshape(3, H, W).float(), depth=depth.reshape(H, W).float(),
                label=_label(sid, K).reshape(H, W).int())


def _config(case):
    return RenderConfig(**CONFIGS[case.get("cfg", "default")], isotropic=bool(case.get("iso", False)))


def _targets(rast, cams, case, seed, sem=False):
    fr = [_frame(c, case["K"], seed + i) for i, c in enumerate(cams)]
    host = lambda k: [f[k].cpu().numpy() for f in fr]
    sem0 = None
    if sem:  # a semantic colour image: C channels per class
        code = torch.rand(case["K"], case["C"], generator=_gen(seed, 8), device=DEV)
        sem0 = [code[f["label"].long()].permute(2, 0, 1).contiguous().cpu().numpy() for f in fr]
    return build_pyramid(rast, host("rgb"), host("depth"), host("label"), sem0)


def _decoder(case, seed):
    if not case["decoder"]:
        return None
    return 0.3 * torch.randn(case["K"], case["C"], generator=_gen(seed, 9), device=DEV)


def _upstream(rast, seed):
    g = _gen(seed, 10)
    return [torch.randn(n * rast.P, generator=g, device=DEV) / rast.P for n in (3, 1, rast.C)]


# ------------------------------------------------------------------------------------------
# prepare / run
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    k = case["kind"]
    if k == "train":
        B = case["B"]
        mlp = MLPInit(seed=seed)
        X = torch.randn(B, 2048, generator=_gen(seed, 11), device=DEV) * 0.5
        X[:, 2009:] = 0
        X = X.to(torch.bfloat16)
        T = torch.randn(B, 32, generator=_gen(seed, 12), device=DEV)
        return dict(case=case, mlp=mlp, X=X, Xt=X.T.contiguous(), T=T, loss=torch.zeros(1, device=DEV))
    cams = _cameras(case, seed)
    if k == "insert":
        B = case["B"]
        fr = _frame(cams[0], case["K"], seed)
        valid = torch.nonzero(fr["depth"] > 0)
        pix = valid[torch.randint(len(valid), (B,), generator=_gen(seed, 13), device=DEV)].flip(1).int().contiguous()
        mlp = MLPInit(seed=seed)
        mlp.y_mean = torch.randn(32, generator=_gen(seed, 14), device=DEV)
        mlp.y_std = 0.5 + torch.rand(32, generator=_gen(seed, 15), device=DEV)
        z = lambda *s: torch.zeros(*s, device=DEV)
        out = dict(mean=z(B, 3), log_scale=z(B, 3), quat=z(B, 4), opacity_logit=z(B), rgb=z(B, 3), sem=z(B, case["C"]))
        code = 0.3 * torch.randn(case["K"], case["C"], generator=_gen(seed, 16), device=DEV)
        return dict(case=case, cam=cams[0], frame={a: b.contiguous() for a, b in fr.items()}, pix=pix, mlp=mlp,
                    out=out, code=code)
    if k == "loss":
        rast = PyramidRasterizer(1, case["C"], cams, case["levels"], RenderConfig(), capacity=1 << 16,
                                 loss_cfg=LossConfig(sem_mode=case["mode"], n_classes=case["K"]))
        gt = _targets(rast, cams, case, seed, sem=case["mode"] == "paper")
        g = _gen(seed, 17)
        # a map still being fitted: the targets with an error on them
        noise = lambda t, s: (t + s * torch.randn(t.shape, generator=g, device=DEV)).contiguous()
        sem = noise(gt["sem"], 0.05) if case["mode"] == "paper" else torch.randn(case["C"] * rast.P, generator=g, device=DEV)
        dec = _decoder(case, seed)
        return dict(case=case, rast=rast, gt=gt, rendered=(noise(gt["rgb"], 0.05), noise(gt["depth"], 0.05), sem),
                    decoder=dec, decoder_grad=torch.zeros_like(dec) if dec is not None else None)
    g = _gaussians(case, seed)
    K = case.get("K", case["C"])
    rast = PyramidRasterizer(case["N"], case["C"], cams, case["levels"], _config(case),
                             loss_cfg=LossConfig(n_classes=K), sh_degree=case.get("sh", 0) if "sh" in g else 0,
                             sem_sh="sem_sh" in g)
    if k == "render":
        return dict(case=case, rast=rast, p=g, cams=cams)
    if k == "splat":
        return dict(case=case, rast=rast, p={a: b.requires_grad_(True) for a, b in g.items()},
                    up=_upstream(rast, seed))
    # a map late in its optimisation: decayed learning rates, so that passes do alike work
    lr = {a: 1e-3 * b for a, b in DEFAULT_LR.items()}
    step = MappingStep(rast, g, _targets(rast, cams, case, seed), lr=lr, decoder=_decoder(case, seed))
    if case["graph"]:
        step.capture()
    return dict(case=case, rast=rast, step=step)


def run(s):
    k = s["case"]["kind"]
    if k == "splat":
        rast = s["rast"]
        leaves = list(s["p"].values())
        images = pyramid_splat(rast, s["p"])
        grads = torch.autograd.grad(images, leaves, s["up"])
        return dict(images=list(images), grads=dict(zip(s["p"], grads)), T=rast.T_final, contributors=rast.n_contrib)
    if k == "render":
        rast = s["rast"]
        rast.set_cameras(s["cams"])
        rast.forward(s["p"])
        return dict(rgb=rast.img_rgb, depth=rast.img_depth, sem=rast.img_sem, T=rast.T_final,
                    contributors=rast.n_contrib, last=rast.last)
    if k == "step":
        st = s["step"]
        st.replay() if s["case"]["graph"] else st.step()
        return dict(params=st.p, m=st.m, v=st.v, terms=s["rast"].terms,
                    decoder_grad=[] if st.decoder_grad is None else st.decoder_grad)
    if k == "loss":
        rast = s["rast"]
        if s["decoder_grad"] is not None:
            s["decoder_grad"].zero_()
        rast.loss(s["gt"], rendered=s["rendered"], decoder=s["decoder"], decoder_grad=s["decoder_grad"])
        return dict(terms=rast.terms, d_rgb=rast.dL_rgb, d_depth=rast.dL_depth, d_sem=rast.dL_sem,
                    decoder_grad=[] if s["decoder_grad"] is None else s["decoder_grad"])
    if k == "train":
        s["loss"].zero_()
        m = s["mlp"]
        m.train_step(s["X"], s["Xt"], s["T"], s["case"]["B"], s["loss"])
        return dict(params=m.params, m=m.m, v=m.v, loss=s["loss"])
    # insertion, as the mapper does it
    f, out, mlp, B = s["frame"], s["out"], s["mlp"], s["case"]["B"]
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    cam, og = camera_struct(s["cam"]), gaussians_struct(out)
    call("sg_init_gaussians", ptr(f["rgb"]), ptr(f["depth"]), ptr(f["label"]), ctypes.byref(cam), ptr(s["pix"]), B,
         ptr(s["code"]), s["case"]["K"], 1.0, ctypes.byref(og), st)
    Bp = (B + 127) // 128 * 128
    X = torch.empty(Bp, 2048, dtype=torch.bfloat16, device=DEV)
    call("sg_extract_patches", ptr(f["rgb"]), ptr(f["depth"]), ptr(f["label"]), ctypes.byref(cam), ptr(s["pix"]), B,
         Bp, ptr(X), None, st)
    Y = mlp.forward(X, Bp)
    call("sg_apply_mlp_init", ptr(Y), B, ptr(mlp.y_mean), ptr(mlp.y_std), ctypes.byref(og), st)
    return dict(X=X, Y=Y, out=out)


# ------------------------------------------------------------------------------------------
# work: bytes and flops of one pass that the path cannot do without
# ------------------------------------------------------------------------------------------

def _pixels(case):
    P = 0
    for i in range(case.get("kf", 1) + case.get("kf_small", 0)):
        W, H = (case["W"], case["H"]) if i < case.get("kf", 1) else (case["W"] * 8 // 15, case["H"] * 8 // 15)
        for _ in range(case["levels"]):
            P += W * H
            W, H = W // 2, H // 2
    return P


def work(case):
    k = case["kind"]
    if k == "train":
        B = case["B"]
        macs = 2048 * 128 * 2 + 128 * 128 * 3 + 128 * 32 * 3
        return dict(bytes=B * (2 * 2048 * 2 + 32 * 4) + 32 * (2048 + 128 + 32) * 128, flops=2 * B * macs)
    if k == "insert":
        B, C = case["B"], case["C"]
        return dict(bytes=B * (2048 * 2 + 32 * 4 + 4 * (14 + C) + 49 * 20), flops=2 * B * (2048 * 128 + 128 * 128 + 128 * 32))
    P, C = _pixels(case), case["C"]
    if k == "loss":
        # reads the rendered and target images, writes the image gradients
        targets = 4 + (C if case["mode"] == "paper" else 1)
        ssim = (3 + (C if case["mode"] == "paper" else 0)) * 8 * 2 * 22
        ce = 6 * C * case["K"] if case["decoder"] else (4 * C if case["mode"] == "ce" else 0)
        return dict(bytes=4 * P * (4 + C + targets + 4 + C), flops=P * (ssim + ce))
    N, nf = case["N"], 4 + C
    sh = ((case.get("sh", 0) + 1) ** 2 - 1) * (3 + (C if case.get("sem_sh") else 0))
    par = 4 * N * (14 + C + sh)
    V = (case.get("kf", 1) + case.get("kf_small", 0)) * case["levels"]
    fwd_flops = P * DEPTH_COMPLEXITY * (15 + 2 * nf) + 200 * N * V
    if k == "render":
        return dict(bytes=par + P * 4 * (nf + 3), flops=fwd_flops)
    bwd_flops = P * DEPTH_COMPLEXITY * (40 + 4 * nf) + 300 * N
    if k == "splat":
        return dict(bytes=2 * par + P * 4 * (2 * nf + 3), flops=fwd_flops + bwd_flops)
    # a step reads and writes the parameters and both moments and reads the targets
    return dict(bytes=6 * par + P * 4 * 5, flops=fwd_flops + bwd_flops + P * (1056 + 6 * C * case["K"]))


# ------------------------------------------------------------------------------------------
# exact: the same results in 64-bit torch, from the definitions
# ------------------------------------------------------------------------------------------

_SH = [lambda x, y, z: -0.4886025119029199 * y, lambda x, y, z: 0.4886025119029199 * z,
       lambda x, y, z: -0.4886025119029199 * x,
       lambda x, y, z: 1.0925484305920792 * x * y, lambda x, y, z: -1.0925484305920792 * y * z,
       lambda x, y, z: 0.31539156525252005 * (3 * z * z - 1), lambda x, y, z: -1.0925484305920792 * x * z,
       lambda x, y, z: 0.5462742152960396 * (x * x - y * y),
       lambda x, y, z: -0.5900435899266435 * y * (3 * x * x - y * y), lambda x, y, z: 2.890611442640554 * x * y * z,
       lambda x, y, z: -0.4570457994644658 * y * (5 * z * z - 1),
       lambda x, y, z: 0.3731763325901154 * z * (5 * z * z - 3),
       lambda x, y, z: -0.4570457994644658 * x * (5 * z * z - 1),
       lambda x, y, z: 1.445305721320277 * z * (x * x - y * y),
       lambda x, y, z: -0.5900435899266435 * x * (x * x - 3 * y * y)]


def _levels(cams, n):
    out = []
    for c in cams:
        fx, fy, cx, cy, W, H = c["fx"], c["fy"], c["cx"], c["cy"], c["W"], c["H"]
        for _ in range(n):
            out.append(dict(c, fx=fx, fy=fy, cx=cx, cy=cy, W=W, H=H))
            fx, fy, cx, cy, W, H = fx / 2, fy / 2, (cx - 0.5) / 2, (cy - 0.5) / 2, W // 2, H // 2
    return out


def _project64(p, cam, iso):
    """Differentiable screen-space quantities (u, v, conic, opacity, depth, features) of the
    Gaussians in front of the camera, in depth order."""
    R, tc = torch.tensor(cam["R_cw"], device=DEV), torch.tensor(cam["t_cw"], device=DEV)
    t = p["mean"] @ R.T + tc
    o = torch.sigmoid(p["opacity_logit"])
    keep = torch.nonzero((t[:, 2].detach() > float(np.float32(0.2))) & (o.detach() >= float(np.float32(1 / 255))))[:, 0]
    keep = keep[torch.argsort(t[keep, 2].detach().float(), stable=True)]
    t, o = t[keep], o[keep]
    x, y, z = t.unbind(1)
    s = torch.exp(p["log_scale"][keep])
    if iso:
        a, b, c = (cam["fx"] * s[:, 0] / z) ** 2 + 0.3, torch.zeros_like(z), (cam["fy"] * s[:, 0] / z) ** 2 + 0.3
    else:
        q = p["quat"][keep]
        w, i, j, k = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        Rq = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                          2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                          2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)], 1).reshape(-1, 3, 3)
        M = Rq * s[:, None, :]
        lx, ly = 1.3 * 0.5 * cam["W"] / cam["fx"], 1.3 * 0.5 * cam["H"] / cam["fy"]
        rx, ry = (x / z).clamp(-lx, lx), (y / z).clamp(-ly, ly)
        T0 = (cam["fx"] / z)[:, None] * (R[0] - rx[:, None] * R[2])
        T1 = (cam["fy"] / z)[:, None] * (R[1] - ry[:, None] * R[2])
        A0, A1 = (T0[:, None] @ M)[:, 0], (T1[:, None] @ M)[:, 0]
        a, b, c = (A0 * A0).sum(1) + 0.3, (A0 * A1).sum(1), (A1 * A1).sum(1) + 0.3
    det = a * c - b * b
    rgb, sem = p["rgb"][keep], p["sem"][keep]
    if "sh" in p:
        d = p["mean"][keep] + R.T @ tc
        dx, dy, dz = (d / d.norm(dim=1, keepdim=True)).unbind(1)
        Y = torch.stack([f(dx, dy, dz) for f in _SH[:p["sh"].shape[1]]], 1)
        rgb = rgb + torch.einsum("nk,nkc->nc", Y, p["sh"][keep])
        if "sem_sh" in p:
            sem = sem + torch.einsum("nk,nkc->nc", Y, p["sem_sh"][keep])
    F = torch.cat([rgb, z[:, None], sem], 1)
    return torch.stack([cam["fx"] * x / z + cam["cx"], cam["fy"] * y / z + cam["cy"], c / det, -b / det, a / det, o],
                       1), F, (a, c)


def _render64(p, cams, levels, iso, up=None, block=32):
    """Packed images and T of every view-level; with up (a function of the packed images that
    gives the upstream gradients) their gradients are left in the parameters' .grad."""
    amax, amin, tmin = (float(np.float32(v)) for v in (0.99, 1 / 255, 1e-4))
    views = _levels(cams, levels)
    proj, parts = [], []

    def blocks(cam, q, F, ext):
        with torch.no_grad():
            thr = torch.log(q[:, 5] / amin)
            ex, ey = (2 * thr * ext[0]).sqrt() + 0.1, (2 * thr * ext[1]).sqrt() + 0.1
        for y0 in range(0, cam["H"], block):
            for x0 in range(0, cam["W"], block):
                y1, x1 = min(cam["H"], y0 + block), min(cam["W"], x0 + block)
                with torch.no_grad():
                    sel = torch.nonzero((q[:, 0] + ex > x0) & (q[:, 0] - ex < x1) & (q[:, 1] + ey > y0) &
                                        (q[:, 1] - ey < y1))[:, 0]
                qs, Fs = q[sel], F[sel]
                yy, xx = torch.meshgrid(torch.arange(y0, y1, device=DEV).double(),
                                        torch.arange(x0, x1, device=DEV).double(), indexing="ij")
                dx, dy = xx.reshape(-1, 1) - qs[:, 0], yy.reshape(-1, 1) - qs[:, 1]
                raw = qs[:, 5] * torch.exp(-0.5 * (qs[:, 2] * dx * dx + qs[:, 4] * dy * dy) - qs[:, 3] * dx * dy)
                al = torch.where(raw < amax, raw, torch.full_like(raw, amax))
                al = torch.where(al >= amin, al, torch.zeros_like(al))
                lt = torch.log1p(-al)
                T = torch.exp(torch.cumsum(lt, 1))
                ok = (T >= tmin).double()
                w = al * torch.exp(torch.cumsum(lt, 1) - lt) * ok
                yield (slice(y0, y1), slice(x0, x1)), w @ Fs, torch.exp((lt.detach() * ok.detach()).sum(1))

    for cam in views:
        q, F, ext = _project64(p, cam, iso)
        with torch.no_grad():
            img = torch.zeros(F.shape[1], cam["H"], cam["W"], device=DEV, dtype=torch.float64)
            Tf = torch.ones(cam["H"], cam["W"], device=DEV, dtype=torch.float64)
            for (ys, xs), v, t in blocks(cam, q.detach(), F.detach(), ext):
                img[:, ys, xs] = v.T.reshape(-1, ys.stop - ys.start, xs.stop - xs.start)
                Tf[ys, xs] = t.reshape(ys.stop - ys.start, -1)
        parts.append((img, Tf))
        proj.append((cam, q, F, ext))
    pack = lambda lo, hi: torch.cat([i[lo:hi].reshape(-1) for i, _ in parts])
    images = [pack(0, 3), pack(3, 4), pack(4, None)]
    T = torch.cat([t.reshape(-1) for _, t in parts])
    if up is not None:
        ups, off = up(images), 0
        C = parts[0][0].shape[0] - 4
        for cam, q, F, ext in proj:
            n = cam["H"] * cam["W"]
            u = torch.cat([ups[0][3 * off:3 * (off + n)].reshape(3, -1), ups[1][off:off + n].reshape(1, -1),
                           ups[2][C * off:C * (off + n)].reshape(C, -1)]).reshape(-1, cam["H"], cam["W"])
            off += n
            ql, Fl = q.detach().requires_grad_(True), F.detach().requires_grad_(True)
            for (ys, xs), v, _ in blocks(cam, ql, Fl, ext):
                v.backward(u[:, ys, xs].reshape(u.shape[0], -1).T)
            torch.autograd.backward([q, F], [ql.grad, Fl.grad], retain_graph=True)
    return images, T


def _loss64(images, gt, views, case, decoder=None):
    """Terms (V x 4), dL/dimages and the decoder gradient for packed 64-bit images."""
    C, K = case["C"], case["K"]
    ims = [i.detach().clone().requires_grad_(True) for i in images]
    dec = decoder.double().requires_grad_(True) if decoder is not None else None
    g = torch.exp(-(torch.arange(11, device=DEV).double() - 5) ** 2 / (2 * 1.5 ** 2))
    g = g / g.sum()

    def blur(a):
        a = torch.nn.functional.conv2d(a[:, None], g.reshape(1, 1, 11, 1), padding=(5, 0))
        return torch.nn.functional.conv2d(a, g.reshape(1, 1, 1, 11), padding=(0, 5))[:, 0]

    def l1_ssim(a, b):
        mx, my = blur(a), blur(b)
        sx, sy, sxy = blur(a * a) - mx * mx, blur(b * b) - my * my, blur(a * b) - mx * my
        s = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
        return 0.8 * (a - b).abs().mean() + 0.2 * (1 - s.mean())

    terms, off = [], 0
    for cam in views:
        H, W = cam["H"], cam["W"]
        cut = lambda t, n: t[n * off:n * (off + H * W)].reshape(n, H, W)
        Lr = l1_ssim(cut(ims[0], 3), cut(gt["rgb"], 3).double())
        gd = cut(gt["depth"], 1).double()
        Ld = (cut(ims[1], 1) - gd).abs()[gd > 0].mean()
        S = cut(ims[2], C)
        if case.get("mode", "ce") == "paper":
            Ls = l1_ssim(S, cut(gt["sem"], C).double())
        else:
            z = S.reshape(C, -1).T
            z = z @ dec.T if dec is not None else z
            Ls = torch.nn.functional.cross_entropy(z, cut(gt["label"], 1).reshape(-1).long(), ignore_index=-1)
        terms.append(torch.stack([Lr, Ld, Ls, Lr + Ld + Ls]))
        off += H * W
    terms = torch.stack(terms)
    grads = torch.autograd.grad(terms[:, 3].sum(), ims + ([dec] if dec is not None else []))
    return terms.detach().reshape(-1), list(grads[:3]), grads[3] if dec is not None else None


def _adam64(p, g, lr, eps):
    """Parameters and moments after the first Adam step from zero moments."""
    m, v = 0.1 * g, 0.001 * g * g
    return p - lr * (m / 0.1) / ((v / 0.001).sqrt() + eps), m, v


def exact(case, seed):
    k = case["kind"]
    if k == "train":
        s = prepare(case, seed)
        m, B = s["mlp"], case["B"]
        W = [t.double().requires_grad_(True) for t in m.params]
        Y = _mlp64(s["X"].double(), W)
        loss = (m.out_w.double() * (Y - s["T"].double()) ** 2).sum() / B
        out = [_adam64(w.detach(), g, 1e-3, 1e-8) for w, g in zip(W, torch.autograd.grad(loss, W))]
        return dict(params=[o[0] for o in out], m=[o[1] for o in out], v=[o[2] for o in out],
                    loss=loss.detach().reshape(1))
    if k == "insert":
        return _insert64(case, seed)
    cams = _cameras(case, seed)
    views = _levels(cams, case["levels"])
    if k == "loss":
        s = prepare(case, seed)
        terms, d, dd = _loss64([r.double() for r in s["rendered"]], s["gt"], views, case, s["decoder"])
        return dict(terms=terms, d_rgb=d[0], d_depth=d[1], d_sem=d[2], decoder_grad=[] if dd is None else dd)
    # the per-block renderer takes about 10 ms per 32 x 32 block with gradients (launches), more
    # with many Gaussians; a captured step has already run once when it is first replayed
    blocks = sum(-(-v["W"] // 32) * -(-v["H"] // 32) for v in views)
    if blocks * (1 + case["N"] / 1e5) > 900 or case.get("graph"):
        return None
    if k == "render":
        p = {a: b.double() for a, b in _gaussians(case, seed).items()}
        im, T = _render64(p, cams, case["levels"], case["iso"])
        return dict(rgb=im[0], depth=im[1], sem=im[2], T=T, contributors=None, last=None)
    s = prepare(case, seed)
    if k == "splat":
        p = {a: b.detach().double().requires_grad_(True) for a, b in s["p"].items()}
        im, T = _render64(p, cams, case["levels"], case["iso"], up=lambda _: [u.double() for u in s["up"]])
        return dict(images=im, grads={a: b.grad for a, b in p.items()}, T=T, contributors=None)
    st, got = s["step"], {}
    p = {a: b.double().requires_grad_(True) for a, b in st.p.items()}

    def up(images):
        got["terms"], d, got["dec"] = _loss64(images, st.gt, views, case, st.decoder)
        return d

    _render64(p, cams, case["levels"], False, up=up)
    out = {a: _adam64(b.detach(), b.grad, st.lr[a], 1e-15) for a, b in p.items()}
    return dict(params={a: o[0] for a, o in out.items()}, m={a: o[1] for a, o in out.items()},
                v={a: o[2] for a, o in out.items()}, terms=got["terms"],
                decoder_grad=[] if got["dec"] is None else got["dec"])


def _mlp64(X, W):
    H = torch.relu(X @ W[0].T + W[3])
    H = torch.relu(H @ W[1].T + W[4])
    return H @ W[2].T + W[5]


def _insert64(case, seed):
    s = prepare(case, seed)
    f, cam, B, mlp = s["frame"], s["cam"], case["B"], s["mlp"]
    W, H = cam["W"], cam["H"]
    px, py = s["pix"].long().unbind(1)
    d0 = f["depth"].double()[py, px]
    xc, yc = (px - cam["cx"]) / cam["fx"] * d0, (py - cam["cy"]) / cam["fy"] * d0
    R, t = torch.tensor(cam["R_cw"], device=DEV), torch.tensor(cam["t_cw"], device=DEV)
    out = dict(mean=(torch.stack([xc, yc, d0], 1) - t) @ R, rgb=f["rgb"].double()[:, py, px].T.contiguous(),
               quat=torch.tensor([1.0, 0, 0, 0], device=DEV, dtype=torch.float64).repeat(B, 1))
    X = torch.zeros((B + 127) // 128 * 128, 2048, device=DEV, dtype=torch.float64)
    for k in range(49):
        x, y = px + k % 7 - 3, py + k // 7 - 3
        ok = ((x >= 0) & (y >= 0) & (x < W) & (y < H)).double()[:, None]
        xs, ys = x.clamp(0, W - 1), y.clamp(0, H - 1)
        d = f["depth"].double()[ys, xs]
        ray = torch.stack([(x - cam["cx"]) / cam["fx"], (y - cam["cy"]) / cam["fy"], torch.ones_like(d)], 1)
        ch = torch.cat([f["rgb"].double()[:, ys, xs].T, torch.where(d > 0, d, 0 * d)[:, None],
                        torch.nn.functional.one_hot(f["label"].long()[ys, xs], 32).double(),
                        ray / ray.norm(dim=1, keepdim=True), (d > 0).double()[:, None],
                        torch.full_like(d, 1 / cam["fx"])[:, None]], 1)
        X[:B, 41 * k:41 * (k + 1)] = ch * ok
    Y = _mlp64(X, [w.double() for w in mlp.params])
    y = Y[:B] * mlp.y_std.double() + mlp.y_mean.double()
    out.update(log_scale=y[:, :3].contiguous(), opacity_logit=y[:, 3].contiguous(),
               sem=y[:, 4:4 + case["C"]].contiguous())
    return dict(X=X, Y=Y, out=out)
