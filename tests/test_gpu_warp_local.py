"""The warp-local pair of compositing passes against the block-staged forward and the
warp-reduced backward on the same inputs, where its own parts can go wrong: sets of more
than 2^24 Gaussians (whose list entries carry no block masks), Gaussians whose rectangles
span more than 32 pixel blocks (all blocks marked), lists of one entry, blocks that most of
their tile's entries reach (whose lists carry no pixel masks) and the smallest views; and
image gradients that are not finite. Every keyframe but the first is fixed. Both forwards
walk every pixel's list in the same order with the same arithmetic, so images and pixel
state are equal bit for bit; the gradients differ by the order of FP32 additions alone
(bounds of tests/test_gpu_batching.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cam(w, h, f, cx, cy, t=(0.0, 0.0, 0.0)):
    from paper_2603_21055_gb300.synth import Camera
    p = np.eye(4, dtype=np.float32)[:3].copy()
    p[:, 3] = t
    return Camera(w, h, f, f, cx, cy, p)


def _keyframes(n, w, h, f, scale, logit, seed, z=(2.0, 3.0)):
    import torch
    from paper_2603_21055_gb300 import splat
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    out = []
    for i in range(n):
        depth = z[0] + (z[1] - z[0]) * rnd(h, w)
        out.append(splat.DeviceKeyframe(_cam(w, h, f, w / 2.0, h / 2.0, (0.01 * i, 0.0, 0.0)), depth,
                                        0.02 * (rnd(h, w) - 0.5), rnd(3, h, w), logit + rnd(h, w),
                                        depth / f * (scale * (0.5 + rnd(h, w))), i == 0))
    return out


def _run(kfs, views, grads_in, **opts):
    import torch
    from paper_2603_21055_gb300 import splat
    sp = splat.Splatter(**opts)
    sp.plan(kfs, views)
    images = splat.alloc_images(views)
    grads = [dict(d_offset=torch.empty_like(k.offset), d_rgb=torch.empty_like(k.rgb),
                  d_logit=torch.empty_like(k.logit), d_scale=torch.empty_like(k.scale)) if k.learnable else None
             for k in kfs]
    sp.forward(kfs, views, images)
    sp.backward(kfs, views, grads_in, grads)
    assert sp.check()[0] == 0
    state = [t.cpu().numpy() for t in sp.state(kfs, views)]
    return images, state, grads[0], sp.stats()


@pytest.mark.parametrize("name,n,w,h,f,scale,logit,view,tile", [
    ("more than 2^24 Gaussians", 32, 820, 640, 700.0, 1.0, 0.0, (90, 61), (16, 16)),
    ("rectangles over 32 blocks", 2, 9, 7, 300.0, 60.0, -1.0, (700, 500), (16, 16)),
    ("rectangles over 32 blocks", 2, 9, 7, 300.0, 60.0, -1.0, (700, 500), (8, 32)),
    ("rectangles over 32 blocks", 2, 9, 7, 300.0, 60.0, -1.0, (700, 500), (32, 8)),
    ("lists of one entry", 1, 3, 2, 40.0, 0.02, 2.0, (130, 90), (16, 16)),
    ("opacities below the floor", 2, 40, 30, 40.0, 1.5, -6.2, (40, 30), (16, 16)),
    ("one pixel", 3, 20, 20, 30.0, 2.0, 1.0, (1, 1), (32, 8)),
])
@pytest.mark.parametrize("schedule", ["tiles", "persistent"])
def test_warp_local_passes_match_block_staged(name, n, w, h, f, scale, logit, view, tile, schedule):
    import torch
    kfs = _keyframes(n, w, h, f, scale, logit, seed=len(name))
    vw, vh = view
    views = [_cam(vw, vh, f * (2.0 if w < 50 else 1.0), vw / 2.0, vh / 2.0, (0.01, -0.02, 0.0))]
    g = torch.Generator(device="cuda").manual_seed(3)
    gin = [dict(rgb=torch.randn(3, vh, vw, generator=g, device="cuda"),
                depth=torch.randn(vh, vw, generator=g, device="cuda"))]
    kw = dict(tile=tile, fwd_schedule=schedule, bwd_schedule=schedule)
    a_im, a_st, a_g, a_stats = _run(kfs, views, gin, bwd_algorithm="warp_local", **kw)
    b_im, b_st, b_g, b_stats = _run(kfs, views, gin, bwd_algorithm="warp_reduce", **kw)
    for q in ("rgb", "depth", "alpha"):
        assert torch.equal(a_im[0][q], b_im[0][q]), q
    for x, y in zip(a_st, b_st):
        assert np.array_equal(x, y)
    assert a_stats["n_keys"] == b_stats["n_keys"] > 0 and a_stats["n_pairs"] == b_stats["n_pairs"]
    assert a_stats["n_pairs"] > 0 or logit < -6.0
    for q in ("d_offset", "d_rgb", "d_logit", "d_scale"):
        x, y = a_g[q].double().cpu().numpy(), b_g[q].double().cpu().numpy()
        assert np.all(np.isfinite(x)), q
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y) + 1e-30, q
        assert np.abs(x - y).max() <= 1e-4 * np.abs(y).max() + 1e-30, q


@pytest.mark.parametrize("value", [float("inf"), float("nan"), -3e38])
def test_gradients_that_are_not_finite_stay_with_their_pixels(value):
    """An infinite, undefined or huge image gradient at single pixels reaches the Gaussians
    that contribute there and no others."""
    import torch
    kfs = _keyframes(2, 40, 30, 40.0, 1.5, 0.0, seed=8)
    views = [_cam(40, 30, 40.0, 20.0, 15.0, (0.01, -0.02, 0.0))]
    g = torch.Generator(device="cuda").manual_seed(5)
    rgb, depth = torch.randn(3, 30, 40, generator=g, device="cuda"), torch.randn(30, 40, generator=g, device="cuda")
    rgb[1, 7, 9] = value
    rgb[0, 22, 31] = value
    depth[13, 20] = value
    gin = [dict(rgb=rgb, depth=depth)]
    a = _run(kfs, views, gin, bwd_algorithm="warp_local")[2]
    b = _run(kfs, views, gin, bwd_algorithm="warp_reduce")[2]
    for q in ("d_offset", "d_rgb", "d_logit", "d_scale"):
        x, y = a[q].double().cpu().numpy(), b[q].double().cpu().numpy()
        ok = np.isfinite(y) & (np.abs(y) < 1e30)
        assert np.array_equal(ok, np.isfinite(x) & (np.abs(x) < 1e30)), q
        assert 0 < (~ok).sum() < ok.size // 4
        assert np.abs(x[ok] - y[ok]).max() <= 1e-4 * np.abs(y[ok]).max(), q


@pytest.mark.parametrize("pose", [False, True])
@pytest.mark.parametrize("learnable", [1, 2])
def test_launches_of_few_and_many_units_agree(pose, learnable):
    """Four views of 2,560 work units each, launched view by view (few units each) and together
    (10,240 units): images, pixel state and counters are equal, gradients up to the order of
    FP32 additions (the bounds above), with and without fixed keyframes and pose gradients."""
    import torch
    kfs = _keyframes(2, 160, 128, 80.0, 1.5, 0.0, seed=4)
    kfs[1].learnable = learnable == 2
    views = [_cam(320, 256, 160.0, 160.0, 128.0, (0.02 * i, -0.02, 0.01 * i)) for i in range(4)]
    g = torch.Generator(device="cuda").manual_seed(6)
    gin = [dict(rgb=torch.randn(3, 256, 320, generator=g, device="cuda"),
                depth=torch.randn(256, 320, generator=g, device="cuda")) for _ in views]
    out = {}
    for sched in ("per_view", "tiles"):
        poses = [torch.empty(12, device="cuda") for _ in views]
        gi = [dict(x, pose=p) for x, p in zip(gin, poses)] if pose else gin
        out[sched] = _run(kfs, views, gi, fwd_schedule=sched, bwd_schedule=sched) + (poses,)
    a, b = out["per_view"], out["tiles"]
    for x, y in zip(a[0], b[0]):
        assert all(torch.equal(x[q], y[q]) for q in ("rgb", "depth", "alpha"))
    assert all(np.array_equal(x, y) for x, y in zip(a[1], b[1]))
    assert a[3]["n_pairs"] == b[3]["n_pairs"] and a[3]["n_evals"] == b[3]["n_evals"]
    pairs = [(a[2][q], b[2][q]) for q in ("d_offset", "d_rgb", "d_logit", "d_scale")]
    for x, y in pairs + (list(zip(a[4], b[4])) if pose else []):
        x, y = x.double().cpu().numpy(), y.double().cpu().numpy()
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)
        assert np.abs(x - y).max() <= 1e-4 * np.abs(y).max()
