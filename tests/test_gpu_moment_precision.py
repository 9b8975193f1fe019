"""The colour gradients of the default backward carry FP32's 24 bits. Where no two Gaussians
reach a pixel a Gaussian's blend weights are the alpha image, so its colour gradient is the sum
of the alpha image times the image gradient over its pixels, exactly known in 64 bits. Here a
Gaussian reaches at most six pixel blocks: six FP32 additions, each off by at most half of a
last place (2^-25 relative to a sum of one sign), bound the root mean square error by 6 x 2^-25
= 1.8e-7 of the sums of positive terms, if the sums inside a block add none. (Operands of 22
bits, truncated, leave 4e-7.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fixed", [False, True])
@pytest.mark.parametrize("seed", [1, 2])
def test_colour_gradients_against_64_bits(seed, fixed):
    import torch
    from paper_2603_21055_gb300 import splat
    from paper_2603_21055_gb300.synth import Camera
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    kw, kh, step = 40, 30, 14
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    w, h = kw * step, kh * step
    view = Camera(w, h, 40.0 * step, 40.0 * step, 0.5 * w + 0.3, 0.5 * h - 0.2, eye)
    kfs = []
    for i in range(2 if fixed else 1):             # the fixed keyframe lies behind the camera
        depth = 2.0 + 0.5 * rnd(kh, kw)
        pose = eye.copy()
        pose[2, 3] = 0.0 if i == 0 else -50.0
        kfs.append(splat.DeviceKeyframe(Camera(kw, kh, 40.0, 40.0, kw / 2.0, kh / 2.0, pose), depth,
                                        torch.zeros(kh, kw, device="cuda"), rnd(3, kh, kw), 0.5 + rnd(kh, kw),
                                        depth * (0.1 + 0.1 * rnd(kh, kw)) / (40.0 * step), i == 0))
    gin = [dict(rgb=0.5 + rnd(3, h, w))]
    sp = splat.Splatter()
    sp.plan(kfs, [view])
    im = splat.alloc_images([view])
    grads = [dict(d_offset=torch.empty_like(k.offset), d_rgb=torch.empty_like(k.rgb),
                  d_logit=torch.empty_like(k.logit), d_scale=torch.empty_like(k.scale)) if k.learnable else None
             for k in kfs]
    sp.forward(kfs, [view], im)
    sp.backward(kfs, [view], gin, grads)
    alpha = im[0]["alpha"].double().cpu().numpy()
    assert sp.stats()["n_pairs"] == np.count_nonzero(alpha)          # one Gaussian per pixel
    # the Gaussian nearest to each pixel: means lie at step (u - kw / 2) + cx, unmoved by the depth
    u = np.rint((np.arange(w) - (0.5 * w + 0.3)) / step + kw / 2.0).astype(int)
    v = np.rint((np.arange(h) - (0.5 * h - 0.2)) / step + kh / 2.0).astype(int)
    on = (alpha > 0) & (v >= 0)[:, None] & (v < kh)[:, None] & (u >= 0)[None] & (u < kw)[None]
    assert on.sum() == np.count_nonzero(alpha)
    at = np.where(on, np.clip(v, 0, kh - 1)[:, None] * kw + np.clip(u, 0, kw - 1)[None], 0).ravel()
    got = grads[0]["d_rgb"].double().cpu().numpy()
    for c in range(3):
        g = gin[0]["rgb"][c].double().cpu().numpy()
        want = np.bincount(at, (alpha * g * on).ravel(), kw * kh)
        seen = want > 0
        assert seen.sum() > 0.9 * kw * kh
        rel = got[c].ravel()[seen] / want[seen] - 1.0
        assert np.sqrt(np.mean(rel ** 2)) <= 1.8e-7
