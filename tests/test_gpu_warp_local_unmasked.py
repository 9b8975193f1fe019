"""The warp-local backward where every block's list starts without pixel masks: each entry
reaches every block of its tiles, so the masks give way to list positions, and the first round
of every unit stores positions in the shared memory through which the pixels' image gradients
have just passed. The red gradient, whose place the positions take, is large and of one sign:
a position's bits read in its stead would be a tiny number and show as a missing term.
Compared with the warp-reduced backward (sums of the same FP32 terms in another order: bounds
of tests/test_gpu_batching.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(16, 16), (8, 32), (32, 8)])
@pytest.mark.parametrize("pose,fixed", [(False, False), (False, True), (True, True)])
def test_first_rounds_without_pixel_masks(tile, pose, fixed):
    import torch
    from paper_2603_21055_gb300 import splat
    from paper_2603_21055_gb300.synth import Camera
    gen = torch.Generator(device="cuda").manual_seed(9)
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    cam = Camera(20, 16, 24.0, 24.0, 10.0, 8.0, eye)
    kfs = []
    for i in range(2):
        depth = 2.0 + rnd(16, 20)
        # 320 Gaussians of about 80 pixels' standard deviation each, faint: all reach all pixels
        kfs.append(splat.DeviceKeyframe(cam, depth, 0.02 * rnd(16, 20), rnd(3, 16, 20), -4.4 + 0.3 * rnd(16, 20),
                                        depth * (1.0 + 0.2 * rnd(16, 20)), i == 0 or not fixed))
    views = [Camera(96, 64, 80.0, 80.0, 48.0, 32.0, eye) for _ in range(6)]
    gin = [dict(rgb=1.0 + rnd(3, 64, 96), depth=rnd(64, 96)) for _ in views]
    out = {}
    for algo in ("warp_local", "warp_reduce"):
        poses = [torch.empty(12, device="cuda") for _ in views]
        gi = [dict(x, pose=p) for x, p in zip(gin, poses)] if pose else gin
        sp = splat.Splatter(tile=tile, bwd_algorithm=algo)
        sp.plan(kfs, views)
        im = splat.alloc_images(views)
        grads = [dict(d_offset=torch.empty_like(k.offset), d_rgb=torch.empty_like(k.rgb),
                      d_logit=torch.empty_like(k.logit), d_scale=torch.empty_like(k.scale)) if k.learnable else None
                 for k in kfs]
        sp.forward(kfs, views, im)
        # every entry reaches most pixels of its tile: no room for the masks
        st = sp.stats()
        assert st["n_pairs"] > 0.75 * 256 * st["n_keys"]
        runs = []
        for _ in range(4):
            sp.backward(kfs, views, gi, grads)
            runs.append([g[q].double().cpu().numpy() for g in grads if g for q in sorted(g)] +
                        ([p.double().cpu().numpy() for p in poses] if pose else []))
        assert sp.check()[0] == 0
        out[algo] = runs
    want = out["warp_reduce"][0]
    for run in out["warp_local"]:
        for x, y in zip(run, want):
            assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y)
            assert np.abs(x - y).max() <= 1e-4 * np.abs(y).max()
