"""Neighbours of frames with few valid pixels against the oracle, bit for bit: so few that every
search passes over all points (by the rule on n^2 against K ncells), and clusters with single
points far from them, whose windows grow until they give way to that pass."""
import numpy as np
import pytest

from oracle import gicp as G

pytestmark = pytest.mark.gpu

W, H, F = 160, 120, 150.0


@pytest.mark.parametrize("kind,frac", [("even", 0.0006), ("even", 0.005), ("even", 0.04), ("even", 0.06), ("pairs", 0.0),
                                       ("cluster", 0.0), ("near", 0.0)])
@pytest.mark.parametrize("k_cov", [3, 10, 32])
def test_neighbours_of_sparse_frames(kind, frac, k_cov):
    import torch
    from paper_2603_21055_gb300 import synth
    from paper_2603_21055_gb300.gicp import GicpTracker
    rng = np.random.default_rng(6)
    v, u = np.mgrid[0:H, 0:W]
    depth = (2.0 + 0.4 * np.sin(0.07 * u) * np.cos(0.05 * v) + 0.002 * rng.normal(size=(H, W))).astype(np.float32)
    if kind == "even":
        on = rng.random((H, W)) < frac
    elif kind == "pairs":
        on = (u % 23 < 2) & (v % 19 == 0)
    else:                                              # a block of 50 x 40 and single points around it
        on = (u >= 20) & (u < 70) & (v >= 30) & (v < 70)
        for x, y in rng.integers(0, (W, H), (12, 2)):
            on[y, x] = True
        if kind == "near":                             # a few of them right before the camera
            for x, y in rng.integers(0, (W, H), (6, 2)):
                depth[y, x], on[y, x] = 0.15, True
    depth = np.where(on, depth, 0).astype(np.float32)
    cam = synth.Camera(W, H, F, F, W / 2.0, H / 2.0, np.eye(4, dtype=np.float32)[:3].copy())
    tr = GicpTracker(src_capacity=W * H, map_capacity=1024, stride=1, k_cov=k_cov)
    knn = torch.full((W * H, k_cov), -7, dtype=torch.int32, device="cuda")
    tr.frame(cam, torch.as_tensor(depth).cuda(), knn_out=knn)
    ref = G.frame_gaussians(depth, F, F, W / 2.0, H / 2.0, 1, k_cov)
    n = tr.src.n()
    assert n == len(ref["points"]) > 3
    k = min(k_cov, n)
    assert np.array_equal(tr.src.host()[0], ref["points"])
    assert np.array_equal(knn[:n, :k].cpu().numpy(), ref["knn"][:, :k])
