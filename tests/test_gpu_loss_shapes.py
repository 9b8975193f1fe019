"""The L1 loss over the block sizes and access widths its launch chooses between: one pixel,
one and one-past-one block of pixels, sizes whose planes do not take 16-byte accesses next to
ones that do, fewer blocks than a cluster and more blocks than SMs; with and without depth
and silhouette mask. The reference is the definition in FP64. Gradients are a sign times one
of two FP32 weights (relative 2e-7: their two roundings); the loss is a sum of nonnegative
FP32 terms in chains of at most 64 per thread, 8 per block tree and 8 + grid / 8 <= 200
additions, 300 roundings of 2^-24 at worst, 2e-5, and of independent signs 1e-6."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(1, 1)], [(32, 32)], [(41, 25)], [(1023, 1), (64, 48), (3, 7)],
                                   [(161, 119), (160, 120)], [(640, 480)] * 9, [(1251, 1001)]])
@pytest.mark.parametrize("depth,mask", [(True, False), (False, False), (True, True)])
def test_l1_loss_and_gradient(sizes, depth, mask):
    import numpy as np
    import torch
    from paper_2603_21055_gb300 import splat
    from paper_2603_21055_gb300.synth import Camera
    gen = torch.Generator(device="cuda").manual_seed(len(sizes))
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    views = [Camera(w, h, 50.0, 50.0, w / 2.0, h / 2.0, eye) for w, h in sizes]
    im = [dict(rgb=rnd(3, h, w), depth=1.0 + rnd(h, w), alpha=rnd(h, w)) for w, h in sizes]
    trgb = [rnd(3, h, w) for w, h in sizes]
    tdep = [torch.where(rnd(h, w) > 0.3, 1.0 + rnd(h, w), torch.zeros(h, w, device="cuda")) for w, h in sizes]
    d_rgb, d_dep = [torch.full_like(t, 7.0) for t in trgb], [torch.full_like(t, 7.0) for t in tdep]
    loss, valid = torch.zeros(1, device="cuda"), torch.zeros(len(sizes), dtype=torch.int32, device="cuda")
    wr, wd, thr = 0.8, 0.5 if depth else 0.0, 0.4 if mask else -1.0
    splat.Splatter().l1_loss_grad(views, im, trgb, tdep, wr, wd, d_rgb, d_dep, loss, valid, min_alpha=thr)
    total = 0.0
    for x, t, td, gr, gd in zip(im, trgb, tdep, d_rgb, d_dep):
        keep = x["alpha"] > thr
        e = (x["rgb"].double() - t.double()) * keep
        ref = torch.sign(e) * (wr / t.numel())
        assert ((gr.double() - ref).abs() <= 2e-7 * ref.abs()).all()
        total += wr * e.abs().sum().item() / t.numel()
        ok, n = td > 0, int((td > 0).sum())
        if depth and n:
            e = (x["depth"].double() - td.double()) * (keep & ok)
            ref = torch.sign(e) * (wd / n)
            total += wd * e.abs().sum().item() / n
        else:
            ref = torch.zeros_like(gd).double()
        assert ((gd.double() - ref).abs() <= 2e-7 * ref.abs()).all()
    assert abs(loss.item() - total) <= 1e-6 * total
