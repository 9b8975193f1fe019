"""The tracking library's paths against one another and the oracle, at the sizes where they
part: neighbour searches by windows of the selection grid and by the hash grid, sets cut
off at their capacity, and tracks whose points fit the rows and the kept candidates of the
tracking kernel or go beyond them (a row holds 16 points; 608 rows, then further points
share them; past four points per warp a point's candidates are not kept).

A track is compared with the same Gauss-Newton iterations taken on the host from
sgad_gicp_linearize, which searches the map for every point at every pose: both sum the
same FP32 terms, so the poses differ by FP64 rounding and, where that moves a coordinate
across an FP32 rounding boundary, by its last place (2.4e-7 at 2-4 m): 2e-6 is allowed.
"""
import numpy as np
import pytest

from oracle import gicp as G

pytestmark = pytest.mark.gpu

F = 150.0


def _frames(w, h, seed=17):
    from paper_2603_21055_gb300 import synth
    rng = np.random.default_rng(seed)
    centre = np.array([3.0, 2.5, 1.5])
    room = synth.make_room(rng, keep_free=(centre, 1.1))
    p0 = synth.keyframe_path(rng, 1, centre)[0]
    p1 = np.hstack([synth.rotation_about(np.array([0.0, 0.6, 0.8]), 0.008) @ p0[:, :3], p0[:, 3:] + 0.006])
    out = []
    for p in (p0, p1):
        d, _ = synth.raycast(room, p, w, h, F, F, w / 2.0, h / 2.0)
        d = (d + rng.normal(scale=0.001, size=d.shape)).astype(np.float32)
        d[h // 4:h // 3, w // 2:w // 2 + w // 6] = 0.0
        out.append((p, d))
    cam = synth.Camera(w, h, F, F, w / 2.0, h / 2.0, np.eye(4, dtype=np.float32)[:3].copy())
    return cam, out


def _tracker(**kw):
    from paper_2603_21055_gb300.gicp import GicpTracker
    return GicpTracker(**kw)


@pytest.mark.parametrize("w,h,stride,k_cov,cap", [
    (160, 120, 2, 10, 8192),      # window search (cells <= 3 x capacity)
    (160, 120, 2, 32, 1601),      # window search, the set cut off at its capacity
    (160, 120, 2, 15, 1599),      # hash search, cut off
    (37, 29, 1, 23, 400),         # window search over most of a small grid
    (7, 5, 1, 32, 64),            # fewer points than neighbours
    (90, 1, 1, 10, 128),          # one row of cells
])
def test_neighbours_match_oracle_on_both_searches(w, h, stride, k_cov, cap):
    import torch
    cam, frames = _frames(w, h)
    depth = frames[0][1].copy()
    tr = _tracker(src_capacity=cap, map_capacity=4096, stride=stride, k_cov=k_cov)
    knn = torch.full((cap, k_cov), -7, dtype=torch.int32, device="cuda")
    tr.frame(cam, torch.as_tensor(depth).cuda(), knn_out=knn)
    n = tr.src.n()
    # the oracle on the selected pixels that fit
    sel = np.zeros_like(depth, bool)
    sel[::stride, ::stride] = depth[::stride, ::stride] > 0
    keep = np.flatnonzero(sel.ravel())
    depth.ravel()[keep[cap:]] = 0.0
    ref = G.frame_gaussians(depth, F, F, w / 2.0, h / 2.0, stride, k_cov)
    assert n == min(len(keep), cap) == len(ref["points"])
    pos, cov, _ = tr.src.host()
    assert np.array_equal(pos, ref["points"])
    assert np.array_equal(knn[:n].cpu().numpy(), ref["knn"])
    # entries <= 1 from an FP32 covariance (the bound of tests/test_gpu_gicp.py)
    assert np.abs(cov - ref["cov"]).max() < 2e-3


def _host_track(tr, pose, iters):
    P = np.asarray(pose, np.float64).copy()
    for _ in range(iters):
        s = tr.linearize(P.astype(np.float32))
        H = np.zeros((6, 6))
        H[np.triu_indices(6)] = s[:21]
        H = np.triu(H) + np.triu(H, 1).T
        xi = np.linalg.solve(H, -s[21:27])
        w, th = xi[:3], np.linalg.norm(xi[:3])
        K = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
        E = np.eye(3) + (np.sin(th) / th) * K + ((1 - np.cos(th)) / th ** 2) * (K @ K) if th > 1e-9 else np.eye(3) + K
        P = np.hstack([E @ P[:, :3], E @ P[:, 3:] + xi[3:, None]])
    return P


@pytest.mark.parametrize("w,h,stride,k_match,turn", [
    (28, 21, 7, 8, 0.0),          # 12 points: one row, partly filled
    (160, 120, 5, 5, 0.0),        # 768 points
    (160, 120, 1, 5, 0.0),        # 18,900 points: rows shared by two rounds of points
    (210, 130, 1, 3, 0.0),        # 26,700 points: some without kept candidates
    (160, 120, 3, 1, 0.15),       # a first step of 0.15 rad: large moves between iterations
])
def test_track_matches_iterations_from_linearize(w, h, stride, k_match, turn):
    import torch
    from paper_2603_21055_gb300 import synth
    cam, frames = _frames(w, h)
    cells = -(-w // stride) * -(-h // stride)
    tr = _tracker(src_capacity=cells, map_capacity=1 << 16, stride=stride, k_cov=6, k_match=k_match, tol=0.0,
                  max_iters=8, d_overlap=0.002, r_max=0.3 if cells < 100 or turn else 0.1)
    tr.frame(cam, torch.as_tensor(frames[0][1]).cuda())
    tr.set_pose(frames[0][0])
    tr.insert()
    tr.frame(cam, torch.as_tensor(frames[1][1]).cuda())
    start = np.array(frames[0][0], np.float64)
    start[:, :3] = synth.rotation_about(np.array([0.0, 0.0, 1.0]), turn) @ start[:, :3]
    tr.track(start)
    got, st = tr.result()
    assert st.iterations == 8 and st.status == 0
    want = _host_track(tr, start, 8)
    assert np.abs(got - want).max() < 2e-6
