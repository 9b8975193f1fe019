"""Performance cases: the work a user of this package has it do, through its public entry
points, over the range of sizes it is used at.

A case is a dict of plain values; its "kind" says which path it takes:

  render    Splatter.forward: all keyframes' Gaussians rendered into all views.
  grad      forward, the loss of Eq. 1 with its image gradients, and the adjoint into the
            learnable keyframes (what a mapping iteration does around its Adam step).
  autograd  the same renderer as a torch.autograd.Function under a loss written in torch.
  stream    mapping.StreamedWindows: iterations, Adam included, on a window in pinned host
            memory, uploaded before and read back after every iteration.
  pose      one iteration of the rendering-based camera initialisation, with the pose
            adjoint and the device pose step, from a frame's first guess.
  infer     the proposal net on new keyframes.
  train     the proposal net's forward, loss and gradients.
  track     GicpTracker.track_sequence on a new sequence of depth frames.

Scenes are box rooms as in synth.py (its rooms, paths and pose perturbations, ray-cast here
on the GPU): depths of 0.5-6 m, one Gaussian per keyframe pixel with scale ~ D / f,
opacity logits ~ N(1, 0.5) and offsets ~ N(0, 3 cm).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2603_21055_gb300 import binding as B
from paper_2603_21055_gb300 import gicp, mapping, proposal, splat, synth


# ----------------------------------------------------------------------------- cases

def _splat(kind, name=None, **kw):
    c = dict(kind=kind, kf_w=640, kf_h=480, kfs=1, view_w=640, view_h=480, views=1, uneven=False, fixed=0,
             depth_weight=0.1, rgb_weight=1.0, ssim_weight=0.0, tile_w=16, tile_h=16, schedule="tiles")
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one tiny keyframe into one view: the latency of a call (a preview, a unit of a test)
        _splat("render", "render_64x48", kf_w=64, kf_h=48, view_w=64, view_h=48),
        # viewing a mapped window: eight VGA keyframes, 2.5 M Gaussians, into eight views
        _splat("render", "render_8x640x480", kfs=8, views=8),
        # a small window into ragged views of three sizes (no size a multiple of a tile)
        _splat("grad", "grad_2x160x120_uneven", kf_w=160, kf_h=120, kfs=2, view_w=300, view_h=170, views=5,
               uneven=True),
        # the headline mapping window, 8 x VGA, colour + depth loss, as one batched pass, with the
        # work split the autotuner picks at this size
        _splat("grad", "grad_8x640x480", kfs=8, views=8, schedule="persistent"),
        # a Replica-sized frame of a sequence: its own Gaussians learnable, its four mapped
        # neighbours fixed, own and neighbour views, all three terms of Eq. 1
        _splat("grad", "grad_5x1200x680_ssim", kf_w=1200, kf_h=680, kfs=5, fixed=4, view_w=1200, view_h=680, views=5,
               rgb_weight=0.8, ssim_weight=0.2, depth_weight=1.0),
        # a quarter-VGA window under a user's own torch loss
        _splat("autograd", "autograd_3x321x243", kf_w=321, kf_h=243, kfs=3, view_w=321, view_h=243, views=2),
        # a window that lives on the host: two iterations and their copies per pass
        _splat("stream", "stream_4x640x480", kfs=4, views=4),
        # camera initialisation of a new VGA frame against the last keyframe
        _splat("pose", "pose_640x480", fixed=1),
        # proposals for the keyframes of one new window
        dict(name="infer_8x640x480", kind="infer", n=8, w=640, h=480),
        # training on small crops of odd size
        dict(name="train_3x315x237", kind="train", n=3, w=315, h=237),
        # depth tracking at TUM size and stride 5, and at Replica size and stride 10
        dict(name="track_4x640x480", kind="track", w=640, h=480, f=600.0, stride=5, frames=4, k_cov=15, k_match=5),
        dict(name="track_6x1200x680", kind="track", w=1200, h=680, f=600.0, stride=10, frames=6, k_cov=10, k_match=5),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["render", "render", "grad", "grad", "grad", "autograd", "stream", "pose", "infer", "train",
                       "track", "track"])
    if kind in ("infer", "train"):
        w = _log_int(rng, 33, 1200)
        h = max(17, int(w * rng.uniform(0.5, 0.9)))
        return dict(kind=kind, n=max(1, min(rng.randint(1, 8), (8 if kind == "infer" else 4) * 640 * 480 // (w * h))),
                    w=w, h=h)
    if kind == "track":
        w = _log_int(rng, 200, 1200)
        h = int(w * rng.uniform(0.55, 0.8))
        stride = rng.randint(max(2, w // 130), max(3, w // 60))
        return dict(kind=kind, w=w, h=h, f=round(w * rng.uniform(0.5, 1.0), 1), stride=stride,
                    frames=rng.randint(3, 6), k_cov=rng.choice([10, 15, 23]), k_match=rng.randint(3, 8))
    lo, hi = {"render": (48, 1200), "grad": (64, 1200), "autograd": (64, 640), "stream": (320, 640),
              "pose": (160, 1200)}[kind]
    w = _log_int(rng, lo, hi)
    h = int(w * rng.uniform(0.55, 0.8))
    vw = max(40, int(w * rng.uniform(0.7, 1.4)))
    vh = max(30, int(vw * rng.uniform(0.55, 0.8)))
    if kind == "stream":
        vw, vh = w, h
    # at most the listed 8 x VGA keyframes into 8 x VGA views, and half of it for the kinds around it
    pairs = (8 * 640 * 480) ** 2 // (1 if kind in ("render", "grad") else 4)
    kfs, views = rng.randint(1, 8), rng.randint(1, 8)
    if kind == "pose":
        kfs, views = rng.randint(1, 2), 1
    if kind == "autograd":
        kfs, views = rng.randint(1, 4), rng.randint(1, 3)
    if kind == "stream":
        kfs, views = rng.randint(2, 4), rng.randint(2, 4)
    while kfs * w * h * views * vw * vh > pairs or kfs * w * h > 2500000:
        if kfs >= views and kfs > 1:
            kfs -= 1
        elif views > 1:
            views -= 1
        else:
            w, h, vw, vh = int(w * 0.8), int(h * 0.8), int(vw * 0.8), int(vh * 0.8)
    ssim = kind in ("grad", "stream") and rng.random() < 0.4
    return _splat(kind, kf_w=w, kf_h=h, kfs=kfs, view_w=vw, view_h=vh, views=views,
                  uneven=kind in ("render", "grad") and rng.random() < 0.3,
                  fixed=kfs if kind == "pose" else (rng.randint(0, kfs - 1) if kind == "grad" else 0),
                  depth_weight=rng.choice([0.0, 0.1, 1.0]) if kind != "pose" else 0.1,
                  rgb_weight=0.8 if ssim else 1.0, ssim_weight=0.2 if ssim else 0.0,
                  tile_w=(t := rng.choice([16, 16, 16, 8, 32])), tile_h=256 // t,
                  schedule=rng.choice(["tiles", "persistent"]))


# ----------------------------------------------------------------------------- rooms on the GPU

def _raycast(room, tex, c2w, w, h, fx, fy, cx, cy):
    """z-depth (h, w) and RGB (3, h, w) of a room, FP32 on the GPU."""
    d64 = dict(dtype=torch.float64, device="cuda")
    R = torch.as_tensor(np.asarray(c2w, np.float64)[:, :3], **d64)
    o = np.asarray(c2w, np.float64)[:, 3]
    u = (torch.arange(w, **d64) - cx) / fx
    v = (torch.arange(h, **d64) - cy) / fy
    rays = torch.stack([u[None, :].expand(h, w), v[:, None].expand(h, w), torch.ones(h, w, **d64)], -1)
    d = rays @ R.T
    d = torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    inv = 1.0 / d
    org = torch.as_tensor(o, **d64)
    hi = torch.as_tensor(room.shell_hi, **d64)
    t_wall = torch.where(d > 0, (hi - org) * inv, -org * inv)
    t, face = t_wall.min(-1)
    face = 2 * face + (torch.gather(d, -1, face[..., None])[..., 0] > 0)
    for b in range(len(room.boxes_lo)):
        t1 = (torch.as_tensor(room.boxes_lo[b], **d64) - org) * inv
        t2 = (torch.as_tensor(room.boxes_hi[b], **d64) - org) * inv
        near, ax = torch.minimum(t1, t2).max(-1)
        far = torch.maximum(t1, t2).min(-1).values
        hit = (near <= far) & (near > 1e-6) & (near < t)
        t = torch.where(hit, near, t)
        face = torch.where(hit, 6 * (b + 1) + 2 * ax, face)
    pts = org + d * t[..., None]
    color = torch.as_tensor(room.face_color, **d64)[face]
    n = torch.zeros_like(color)
    for f, ph, amp in tex:                     # three octaves of smooth texture per channel
        n += amp * torch.sin(pts @ torch.as_tensor(f, **d64) + torch.as_tensor(ph, **d64))
    rgb = (color + 0.3 * n).clamp(0, 1)
    return t.float().contiguous(), rgb.permute(2, 0, 1).float().contiguous()


def _room(seed, n_poses):
    rng = np.random.default_rng(seed)
    centre = np.array([3.0, 2.5, 1.5])
    room = synth.make_room(rng, keep_free=(centre, 1.1))
    tex = [(rng.normal(0, 2.5 * 2 ** k, (3, 3)), rng.uniform(0, 6.28, 3), 0.6 / 2 ** k) for k in range(3)]
    return rng, room, tex, synth.keyframe_path(rng, n_poses, centre)


def _f32(p):
    return np.ascontiguousarray(np.asarray(p, np.float64).astype(np.float32))


def _scene(c, seed):
    """Device keyframes, views and targets of a splatting case."""
    rng, room, tex, poses = _room(seed, c["kfs"])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kw, kh, kf_f = c["kf_w"], c["kf_h"], float(c["kf_w"]) * 600.0 / 640.0
    kfs = []
    for i, p in enumerate(poses):
        cam = synth.Camera(kw, kh, kf_f, kf_f, kw / 2.0, kh / 2.0, _f32(p))
        depth, rgb = _raycast(room, tex, p, kw, kh, cam.fx, cam.fy, cam.cx, cam.cy)
        noise = torch.randn(2, kh, kw, generator=gen, device="cuda")
        scale = depth / kf_f * (0.8 + 0.4 * torch.rand(kh, kw, generator=gen, device="cuda"))
        kfs.append(splat.DeviceKeyframe(cam, depth, 0.03 * noise[0], rgb, 1.0 + 0.5 * noise[1], scale,
                                        i >= c["fixed"]))
    views, trgb, tdep = [], [], []
    for j in range(c["views"]):
        s = (1.0, 0.55, 0.25)[j % 3] if c["uneven"] else 1.0
        w, h = max(24, int(c["view_w"] * s)), max(18, int(c["view_h"] * s))
        p = synth.perturb_pose(rng, poses[j % c["kfs"]], 0.05, 2.0)
        f = w * 600.0 / 640.0
        cam = synth.Camera(w, h, f, f, w / 2.0, h / 2.0, _f32(synth.pose_inverse(p)))
        d, r = _raycast(room, tex, p, w, h, cam.fx, cam.fy, cam.cx, cam.cy)
        hole = torch.rand(h, w, generator=gen, device="cuda") < 0.02         # missing sensor depth
        views.append(cam)
        trgb.append(r)
        tdep.append(torch.where(hole, torch.zeros_like(d), d))
    return kfs, views, trgb, tdep


def _host_scene(c, kfs, views, trgb, tdep):
    n = lambda t: t.cpu().numpy()
    ks = [synth.Keyframe(k.cam, n(k.depth), n(k.offset), n(k.rgb), n(k.logit), n(k.scale), k.learnable) for k in kfs]
    return synth.Scene(ks, views, [n(t) for t in trgb], [n(t) for t in tdep], c["depth_weight"], c["rgb_weight"],
                       "window", c["ssim_weight"])


# ----------------------------------------------------------------------------- the package's calls

SILHOUETTE = 0.99


class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.case = c
    if c["kind"] in ("infer", "train"):
        return _prepare_net(c, seed, s)
    if c["kind"] == "track":
        return _prepare_track(c, seed, s)
    s.kfs, s.views, s.trgb, s.tdep = _scene(c, seed)
    work = dict(fwd_schedule=c["schedule"], bwd_schedule=c["schedule"])
    if c["kind"] == "stream":
        sp = splat.Splatter(tile=(c["tile_w"], c["tile_h"]), **work)
        s.sw = mapping.StreamedWindows(_host_scene(c, s.kfs, s.views, s.trgb, s.tdep), options=sp.options)
        s.kfs = s.trgb = s.tdep = None
        s.sw.capture()
        return s
    s.sp = splat.Splatter(tile=(c["tile_w"], c["tile_h"]), **work)
    if c["kind"] == "pose":
        s.state0 = torch.zeros(B.SGAD_POSE_STATE_FLOATS, device="cuda")
        eye = torch.tensor([1.0, 0, 0, 0, 0, 1.0, 0, 0, 0, 0, 1.0, 0], device="cuda")
        s.state0[0:12] = eye
        s.state0[12:24] = eye
        s.state = s.state0.clone()
        for k in s.kfs:
            k.learnable, k.world_transform = False, s.state[12:24]
        s.W0 = np.asarray(s.views[0].pose, np.float32).reshape(12).copy()
        s.d_pose = torch.zeros(12, device="cuda")
    s.sp.plan(s.kfs, s.views)
    s.images = splat.alloc_images(s.views)
    if c["kind"] in ("grad", "pose"):
        s.d_rgb = [torch.empty_like(im["rgb"]) for im in s.images]
        s.d_dep = [torch.empty_like(im["depth"]) for im in s.images]
        s.loss = torch.zeros(1, device="cuda")
        s.valid = torch.zeros(len(s.views), dtype=torch.int32, device="cuda")
        use_dep = c["depth_weight"] != 0
        s.gin = [dict(rgb=r, depth=d if use_dep else None) for r, d in zip(s.d_rgb, s.d_dep)]
        if c["kind"] == "pose":
            s.gin[0]["pose"] = s.d_pose
        s.grads = [dict(d_offset=torch.empty_like(k.offset), d_rgb=torch.empty_like(k.rgb),
                        d_logit=torch.empty_like(k.logit), d_scale=torch.empty_like(k.scale)) if k.learnable else None
                   for k in s.kfs]
    if c["kind"] == "autograd":
        s.params = [t.clone().requires_grad_() for k in s.kfs for t in (k.offset, k.rgb, k.logit, k.scale)]
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "render":
        s.sp.forward(s.kfs, s.views, s.images)
        return dict(images=s.images)
    if kind == "grad":
        s.sp.forward(s.kfs, s.views, s.images)
        _loss(s)
        if c["ssim_weight"] != 0:
            s.sp.ssim_loss_grad(s.views, s.images, s.trgb, c["ssim_weight"], s.d_rgb, s.loss)
        s.sp.backward(s.kfs, s.views, s.gin, s.grads)
        return dict(images=s.images, loss=s.loss, grads=[g for g in s.grads if g is not None])
    if kind == "autograd":
        out = splat.SplatFn.apply(s.sp, s.kfs, s.views, *s.params)
        loss = 0.0
        for i, (t, d) in enumerate(zip(s.trgb, s.tdep)):
            loss = loss + ((out[3 * i] - t) ** 2).mean() + c["depth_weight"] * ((out[3 * i + 1] - d) ** 2).mean()
        grads = torch.autograd.grad(loss, s.params)
        return dict(loss=loss.detach(), out=[o.detach() for o in out], grads=list(grads))
    if kind == "stream":
        s.sw.replay()
        s.sw.finish()
        # the loss as the host reads it: the last 64-float slot of the state read back
        return [dict(images=m.images, loss=o[-64:-63], grads=m.grads) for m, o in zip(s.sw.mappers, s.sw.host_out)]
    if kind == "pose":
        s.state.copy_(s.state0)                       # a new frame starts from its first guess
        s.sp.forward(s.kfs, s.views, s.images)
        _loss(s, SILHOUETTE)
        s.sp.backward(s.kfs, s.views, s.gin, s.grads)
        B.sgad_pose_adam_step(s.d_pose.data_ptr(), s.W0, s.state.data_ptr(), 2e-3, 2e-3, stream=s.sp.stream())
        return dict(images=s.images, loss=s.loss, d_pose=s.d_pose, state=s.state)
    if kind == "infer":
        s.net.forward(s.rgb, s.depth, s.delta, s.logit)
        return dict(delta=s.delta, logit=s.logit)
    if kind == "train":
        s.net.forward(s.rgb, s.depth, s.delta, s.logit)
        s.net.loss_grad(s.t_delta, s.t_logit)
        s.net.backward()
        return dict(delta=s.delta, logit=s.logit, loss=s.net.loss, dw=s.net.dw, db=s.net.db)
    s.tr.map.count.zero_()                            # a new sequence
    poses = s.tr.track_sequence(s.cam, s.depths, s.first)
    # the poses as the FP32 camera poses that the mapping takes them in
    return dict(poses=np.asarray(poses, np.float32), points=s.tr.map.pos, count=s.tr.map.count)


def _loss(s, min_alpha=-1.0):
    c = s.case
    s.loss.zero_()
    use_dep = c["depth_weight"] != 0
    s.sp.l1_loss_grad(s.views, s.images, s.trgb, s.tdep if use_dep else None, c["rgb_weight"], c["depth_weight"],
                      s.d_rgb, s.d_dep if use_dep else None, s.loss, s.valid if use_dep else None,
                      min_alpha=min_alpha)


def _prepare_net(c, seed, s):
    rng, room, tex, poses = _room(seed, c["n"])
    f = c["w"] * 600.0 / 640.0
    frames = [_raycast(room, tex, p, c["w"], c["h"], f, f, c["w"] / 2.0, c["h"] / 2.0) for p in poses]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s.depth = torch.stack([d for d, _ in frames])
    s.depth = (s.depth + 0.01 * torch.randn(s.depth.shape, generator=gen, device="cuda")).contiguous()
    s.rgb = torch.stack([r for _, r in frames]).contiguous()
    params = [(w, rng.normal(0, 0.05, b.shape).astype(np.float32)) for w, b in proposal.he_init(seed)]
    s.net = proposal.ProposalNet(params)
    s.net.reserve(c["n"], c["h"], c["w"])
    s.delta, s.logit = torch.empty_like(s.depth), torch.empty_like(s.depth)
    s.t_delta = 0.03 * torch.randn(s.depth.shape, generator=gen, device="cuda")
    s.t_logit = 1.0 + torch.randn(s.depth.shape, generator=gen, device="cuda")
    return s


def _prepare_track(c, seed, s):
    rng, room, tex, _ = _room(seed, 1)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pos, yaw, pitch = np.array([3.0, 2.5, 1.5]), rng.uniform(0, 6.28), rng.uniform(-0.1, 0.1)
    step, turn = 0.02 * synth.random_unit(rng), math.radians(rng.uniform(-1.2, 1.2))
    s.cam = synth.Camera(c["w"], c["h"], c["f"], c["f"], c["w"] / 2.0, c["h"] / 2.0, np.eye(3, 4, dtype=np.float32))
    s.depths = []
    for i in range(c["frames"]):
        p = synth.look_pose(pos + i * step, yaw + i * turn, pitch)
        if i == 0:
            s.first = p
        d, _ = _raycast(room, tex, p, c["w"], c["h"], s.cam.fx, s.cam.fy, s.cam.cx, s.cam.cy)
        s.depths.append((d + 0.002 * torch.randn(d.shape, generator=gen, device="cuda")).contiguous())
    cells = (-(-c["w"] // c["stride"])) * (-(-c["h"] // c["stride"]))
    s.tr = gicp.GicpTracker(src_capacity=max(1024, cells), map_capacity=1 << 19, stride=c["stride"], k_cov=c["k_cov"],
                            k_match=c["k_match"])
    return s


# ----------------------------------------------------------------------------- what a pass cannot do without

def _sizes(c):
    g = c["kfs"] * c["kf_w"] * c["kf_h"]
    p = 0
    for j in range(c["views"]):
        s = (1.0, 0.55, 0.25)[j % 3] if c["uneven"] else 1.0
        p += max(24, int(c["view_w"] * s)) * max(18, int(c["view_h"] * s))
    return g, p


def work(case):
    c = case
    if c["kind"] in ("infer", "train"):
        px = c["n"] * c["w"] * c["h"]
        mul = 9 * (4 * 32 + 32 * 32 + 32 * 32 + 32 * 2)
        if c["kind"] == "infer":
            return {"bytes": px * 4 * (4 + 2), "flops": px * 2 * mul}
        # gradients of weights (all layers) and of inputs (all but the first)
        return {"bytes": px * 4 * (4 + 2 + 2), "flops": px * 2 * (3 * mul - 9 * 4 * 32)}
    if c["kind"] == "track":
        n = (-(-c["w"] // c["stride"])) * (-(-c["h"] // c["stride"]))
        # per frame: the selected depths and the source's Gaussians (64 B); per iteration (about 12 from
        # a constant-speed guess) the matched map Gaussians (64 B) and ~600 operations a point
        return {"bytes": c["frames"] * n * (4 + 64 + 64), "flops": (c["frames"] - 1) * n * 12 * 600}
    g, p = _sizes(c)
    # contributing (pixel, Gaussian) pairs: about 7 a pixel for each keyframe that covers it
    pairs = 7.0 * min(c["kfs"], 8) * p
    b, f = 28 * g + 20 * p, 29 * pairs
    if c["kind"] != "render":
        learn = g * (c["kfs"] - c["fixed"]) // c["kfs"]
        b += 24 * learn + 16 * p            # gradients written, targets read
        f += 77 * pairs
        if c["ssim_weight"]:
            f += 3 * p * 360
    if c["kind"] == "stream":
        # two iterations: the window up, its state down, and Adam over six planes
        b, f = 2 * (b + (28 * g + 16 * p) + 24 * g + 6 * 28 * g), 2 * f
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- the same in 64 bits

def exact(case, seed):
    c = case
    if c["kind"] == "track":
        return None          # an iterative estimate that ends by a tolerance, from integer decisions in FP32
    if c["kind"] in ("infer", "train"):
        return _exact_net(c, seed)
    kfs, views, trgb, tdep = _scene(c, seed)
    if c["kind"] == "pose":
        for k in kfs:
            k.learnable = False
    want_pose = c["kind"] == "pose"
    r = _ExactSplat(kfs, views, want_pose, (c["tile_w"], c["tile_h"]))
    images = r.forward()
    if c["kind"] == "render":
        return dict(images=images)
    loss, gi = _exact_loss(c, images, trgb, tdep)
    grads, d_pose = r.backward(gi)
    loss = loss.reshape(1)
    if c["kind"] == "grad":
        return dict(images=images, loss=loss, grads=[g for k, g in zip(kfs, grads) if k.learnable])
    if c["kind"] == "autograd":
        flat = [g[n] for g in grads for n in ("d_offset", "d_rgb", "d_logit", "d_scale")]
        return dict(loss=loss.reshape(()), out=[im[n] for im in images for n in ("rgb", "depth", "alpha")], grads=flat)
    if c["kind"] == "stream":
        return [dict(images=images, loss=loss, grads=grads)] * 2
    return dict(images=images, loss=loss, d_pose=d_pose, state=None)


def _exact_loss(c, images, trgb, tdep):
    """Loss and its gradients by the rendered images."""
    loss, leaves = 0.0, []
    for im, tr, td in zip(images, trgb, tdep):
        x, d = im["rgb"].clone().requires_grad_(), im["depth"].clone().requires_grad_()
        leaves.append((x, d))
        y, td = tr.double(), td.double()
        if c["kind"] == "autograd":
            loss = loss + ((x - y) ** 2).mean() + c["depth_weight"] * ((d - td) ** 2).mean()
            continue
        keep = (im["alpha"] > SILHOUETTE).double() if c["kind"] == "pose" else torch.ones_like(d)
        loss = loss + c["rgb_weight"] * ((x - y).abs() * keep).mean()
        if c["depth_weight"]:
            ok = (td > 0).double()
            loss = loss + c["depth_weight"] * ((d - td).abs() * ok * keep).sum() / ok.sum().clamp(min=1)
        if c["ssim_weight"]:
            loss = loss + c["ssim_weight"] * (1.0 - _ssim(x, y).mean())
    gs = torch.autograd.grad(loss, [t for p in leaves for t in p], allow_unused=True)
    return loss.detach(), [(gs[2 * i], gs[2 * i + 1]) for i in range(len(images))]


def _ssim(x, y):
    k = torch.arange(11, dtype=torch.float64, device="cuda") - 5
    k = torch.exp(-k * k / 4.5)
    k = k / k.sum()
    blur = lambda t: F.conv2d(F.conv2d(t[:, None], k.view(1, 1, 1, 11), padding=(0, 5)), k.view(1, 1, 11, 1),
                              padding=(5, 0))[:, 0]
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    mx, my, xx, yy, xy = blur(x), blur(y), blur(x * x), blur(y * y), blur(x * y)
    return ((2 * mx * my + c1) * (2 * (xy - mx * my) + c2)) / \
        ((mx * mx + my * my + c1) * (xx - mx * mx + yy - my * my + c2))


class _ExactSplat:
    """The renderer in FP64: every tile's list against all of its pixels, dense."""

    BUDGET = 90000                       # (tile, list position) slots handled at once

    def __init__(self, kfs, views, want_pose, tile):
        self.kfs, self.views, self.want_pose, self.tile = kfs, views, want_pose, tile

    def _params(self, grad):
        ps = []
        for k in self.kfs:
            ps.append([t.detach().double().reshape(-1, k.n).clone().requires_grad_(grad)
                       for t in (k.offset, k.rgb, k.logit, k.scale)])
        return ps

    def _gaussians(self, ps):
        """(mu (G, 3), opacity, colour (G, 3), scale)."""
        mus = []
        for k, (off, _, _, _) in zip(self.kfs, ps):
            c = k.cam
            P = torch.as_tensor(np.asarray(c.pose, np.float64), device="cuda")
            j = torch.arange(k.n, device="cuda")
            u, v = (j % c.width).double(), (j // c.width).double()
            d = (k.depth.double().reshape(-1) + off[0]).abs()
            q = torch.stack([d * (u - c.cx) / c.fx, d * (v - c.cy) / c.fy, d], -1)
            mus.append(q @ P[:, :3].T + P[:, 3])
        cat = lambda i, n: torch.cat([p[i].T.reshape(-1, n) for p in ps])
        return torch.cat(mus), torch.sigmoid(cat(2, 1)[:, 0]), cat(1, 3), cat(3, 1)[:, 0]

    @staticmethod
    def _project(mu, o, rgb, s, v, W):
        """(G, 10): mean, conic, opacity, colour, depth; and the covariance."""
        t = mu @ W[:, :3].T + W[:, 3]
        z = torch.where(t[:, 2] > 0.2, t[:, 2], torch.ones_like(t[:, 2]))
        ux, uy = t[:, 0] / z, t[:, 1] / z
        j00, j11 = v.fx / z, v.fy / z
        j02, j12 = -j00 * ux, -j11 * uy
        s2 = s * s
        xx = s2 * (j00 * j00 + j02 * j02) + 0.3
        xy = s2 * j02 * j12
        yy = s2 * (j11 * j11 + j12 * j12) + 0.3
        det = xx * yy - xy * xy
        q = torch.stack([v.fx * ux + v.cx, v.fy * uy + v.cy, yy / det, -xy / det, xx / det, o, rgb[:, 0], rgb[:, 1],
                         rgb[:, 2], z], -1)
        return q, (xx, yy, det, t[:, 2] > 0.2)

    def _lists(self, q, cov, v):
        """Gaussians of every tile, front to back: (tile, Gaussian) pairs and the tiles' offsets."""
        xx, yy, det, front = cov
        tw, th = self.tile
        mid = 0.5 * (xx + yy)
        rho = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        x0, x1 = torch.floor(q[:, 0] - rho), torch.floor(q[:, 0] + rho)
        y0, y1 = torch.floor(q[:, 1] - rho), torch.floor(q[:, 1] + rho)
        ok = front & (x1 >= 0) & (y1 >= 0) & (x0 <= v.width - 1) & (y0 <= v.height - 1)
        g = torch.nonzero(ok)[:, 0]
        g = g[torch.argsort(q[g, 9].float(), stable=True)]
        tile = lambda t, n, size: (t[g].clamp(0, n - 1) / size).long()
        tx0, tx1 = tile(x0, v.width, tw), tile(x1, v.width, tw)
        ty0, ty1 = tile(y0, v.height, th), tile(y1, v.height, th)
        nx, n = tx1 - tx0 + 1, (tx1 - tx0 + 1) * (ty1 - ty0 + 1)
        rep = torch.repeat_interleave(torch.arange(len(g), device="cuda"), n)
        k = torch.arange(len(rep), device="cuda") - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
        tiles_x, tiles_y = -(-v.width // tw), -(-v.height // th)
        t = (ty0[rep] + k // nx[rep]) * tiles_x + tx0[rep] + k % nx[rep]
        order = torch.argsort(t, stable=True)
        counts = torch.bincount(t, minlength=tiles_x * tiles_y)
        return g[rep][order], torch.cumsum(counts, 0) - counts, counts, tiles_x

    def _batches(self, counts):
        order = torch.argsort(counts, descending=True).cpu().tolist()
        n = counts.cpu().tolist()
        i = 0
        while i < len(order) and n[order[i]] > 0:
            take = max(1, self.BUDGET // n[order[i]])
            yield torch.tensor(order[i:i + take], device="cuda"), n[order[i]]
            i += take

    def _tiles(self, q, ids, off, counts, tiles_x, tl, most):
        """Rendered (rgb, depth, alpha) of the tiles tl, dense over `most` list positions."""
        tw, th = self.tile
        j = torch.arange(most, device="cuda")
        valid = j[None] < counts[tl][:, None]
        g = ids[(off[tl][:, None] + j[None]).clamp(max=len(ids) - 1)]
        e = q[g]                                                        # (T, n, 10)
        p = torch.arange(tw * th, device="cuda")
        px = ((tl % tiles_x)[:, None] * tw + p[None] % tw).double()
        py = ((tl // tiles_x)[:, None] * th + p[None] // tw).double()
        dx, dy = e[:, :, 0:1] - px[:, None], e[:, :, 1:2] - py[:, None]
        power = -0.5 * (e[:, :, 2:3] * dx * dx + e[:, :, 4:5] * dy * dy) - e[:, :, 3:4] * dx * dy
        alpha = (e[:, :, 5:6] * torch.exp(power.clamp(max=0))).clamp(max=0.99)
        with torch.no_grad():
            on = valid[:, :, None] & (power <= 0) & (alpha >= 1.0 / 255.0)
            on &= torch.cumprod(torch.where(on, 1 - alpha, torch.ones_like(alpha)), 1) >= 1e-4
        a = torch.where(on, alpha, torch.zeros_like(alpha))
        logt = torch.log1p(-a)
        w = a * torch.exp(torch.cumsum(logt, 1) - logt)
        out = torch.einsum("tnp,tnc->tcp", w, e[:, :, 6:10])
        return torch.cat([out, w.sum(1, keepdim=True)], 1)              # (T, 5, pixels)

    def forward(self):
        with torch.no_grad():
            self.state, images = [], []
            base = self._gaussians(self._params(False))
            for v in self.views:
                W = torch.as_tensor(np.asarray(v.pose, np.float64), device="cuda")
                q, cov = self._project(*base, v, W)
                lists = self._lists(q, cov, v)
                self.state.append((q, lists))
                ids, off, counts, tiles_x = lists
                im = torch.zeros(len(counts), 5, self.tile[0] * self.tile[1], dtype=torch.float64, device="cuda")
                for tl, most in self._batches(counts):
                    im[tl] = self._tiles(q, ids, off, counts, tiles_x, tl, most)
                im = self._untile(im, v, tiles_x)
                images.append(dict(rgb=im[:3].contiguous(), depth=im[3].contiguous(), alpha=im[4].contiguous()))
        return images

    def _untile(self, t, v, tiles_x):
        tw, th = self.tile
        t = t.view(-1, tiles_x, t.shape[1], th, tw).permute(2, 0, 3, 1, 4)
        return t.reshape(t.shape[0], t.shape[1] * th, tiles_x * tw)[:, :v.height, :v.width]

    def _retile(self, im, tiles_x, n_tiles):
        tw, th = self.tile
        h, w = n_tiles // tiles_x * th, tiles_x * tw
        im = F.pad(im, (0, w - im.shape[2], 0, h - im.shape[1]))
        im = im.view(im.shape[0], h // th, th, tiles_x, tw).permute(1, 3, 0, 2, 4)
        return im.reshape(n_tiles, im.shape[2], th * tw)

    def backward(self, image_grads):
        ps = self._params(True)
        d_pose = None
        for v, (q, lists), (gr, gd) in zip(self.views, self.state, image_grads):
            ids, off, counts, tiles_x = lists
            gi = torch.zeros(5, v.height, v.width, dtype=torch.float64, device="cuda")
            gi[:3] = gr
            if gd is not None:
                gi[3] = gd
            gi = self._retile(gi, tiles_x, len(counts))
            dq = torch.zeros_like(q)
            for tl, most in self._batches(counts):
                # a leaf of these tiles' entries alone, so that a batch costs its own lists
                span = (off[tl][:, None] + torch.arange(most, device="cuda")[None]).clamp(max=len(ids) - 1)
                used, at = torch.unique(ids[span], return_inverse=True)
                leaf = q[used].requires_grad_()
                local = at.reshape(len(tl), most)
                out = self._tiles_local(leaf, local, counts, tiles_x, tl, most)
                (d,) = torch.autograd.grad(out, leaf, gi[tl])
                dq[used] += d
            W = torch.as_tensor(np.asarray(v.pose, np.float64), device="cuda").requires_grad_(self.want_pose)
            full, _ = self._project(*self._gaussians(ps), v, W)
            leaves = [t for p in ps for t in p] + ([W] if self.want_pose else [])
            gs = torch.autograd.grad(full, leaves, dq, allow_unused=True)
            if self.want_pose:
                d_pose = gs[-1].reshape(12)
            for t, d in zip([t for p in ps for t in p], gs):
                t.grad = d if t.grad is None else t.grad + d
        names = ("d_offset", "d_rgb", "d_logit", "d_scale")
        grads = []
        for k, p in zip(self.kfs, ps):
            h, w = k.cam.height, k.cam.width
            grads.append({n: t.grad.view(3, h, w) if n == "d_rgb" else t.grad.view(h, w) for n, t in zip(names, p)})
        return grads, d_pose

    def _tiles_local(self, leaf, local, counts, tiles_x, tl, most):
        """_tiles for entries named by their place in `leaf`, one row of `local` per tile."""
        full = torch.zeros_like(counts)
        full[tl] = torch.arange(len(tl), device="cuda") * most
        return self._tiles(leaf, local.reshape(-1), full, counts, tiles_x, tl, most)


def _bf16(t):
    return t.float().bfloat16().double()


def _exact_net(c, seed):
    """The net in FP64 with its bfloat16 storage points (input, weights, activations and the
    gradients between layers)."""
    s = _prepare_net(c, seed, _State())
    real = [(torch.as_tensor(w).cuda().double(), torch.as_tensor(b).cuda().double()) for w, b in s.net.real_params()]
    x = _bf16(torch.cat([s.rgb, s.depth[:, None]], 1))
    acts, ks = [x], []
    for l, (w, b) in enumerate(real):
        k = _bf16(w).permute(3, 2, 0, 1).contiguous()                   # (co, ci, ky, kx)
        ks.append(k)
        x = _conv(x, k) + b[None, :, None, None]
        if l < 3:
            x = _bf16(x.clamp(min=0))
        acts.append(x)
    out = dict(delta=0.01 * acts[4][:, 0], logit=acts[4][:, 1])
    if c["kind"] == "infer":
        return out
    n = s.depth.numel()
    e0, e1 = acts[4][:, 0] - s.t_delta.double() * 100.0, acts[4][:, 1] - s.t_logit.double()
    out["loss"] = ((e0 * e0).sum() + (e1 * e1).sum()).reshape(1) / n
    d = _bf16(torch.stack([2 * e0 / n, 2 * e1 / n], 1))
    dw, db = [None] * 4, [None] * 4
    for l in range(3, -1, -1):
        co, ci = ks[l].shape[:2]
        cin_p, cout_p = s.net.shapes[l][2:]
        xp = F.pad(acts[l], (1, 1, 1, 1))
        h, w = d.shape[2:]
        dw[l] = torch.zeros(9, cin_p, cout_p, dtype=torch.float64, device="cuda")
        df = d.permute(1, 0, 2, 3).reshape(co, -1)
        for t in range(9):
            win = xp[:, :, t // 3:t // 3 + h, t % 3:t % 3 + w].permute(1, 0, 2, 3).reshape(ci, -1)
            dw[l][t, :ci, :co] = win @ df.T
        db[l] = torch.zeros(cout_p, dtype=torch.float64, device="cuda")
        db[l][:co] = d.sum((0, 2, 3))
        if l > 0:
            back = ks[l].flip(2, 3).permute(1, 0, 2, 3)
            d = _bf16(_conv(d, back) * (acts[l] > 0))
    out.update(dw=dw, db=db)
    return out


def _conv(x, k):
    """3 x 3 convolution with zero padding as nine products."""
    xp = F.pad(x, (1, 1, 1, 1))
    h, w = x.shape[2:]
    y = 0.0
    for t in range(9):
        y = y + torch.einsum("oi,nihw->nohw", k[:, :, t // 3, t % 3], xp[:, :, t // 3:t // 3 + h, t % 3:t % 3 + w])
    return y
