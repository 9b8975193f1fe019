"""Tracking of frames without a valid depth between frames with one: the terms that a track
leaves in its blocks' shared memory must not reach the sums of an empty set. Its system is
exactly zero, and its track ends before the first step with the pose it was given. (A block
that summed a row of no points took its warps' zeroes without waiting for them.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H, F = 160, 120, 150.0


@pytest.mark.parametrize("stride", [1, 5])          # more rows than blocks, and a few rows
def test_empty_frames_between_tracked_ones(stride):
    import torch
    from paper_2603_21055_gb300 import synth
    from paper_2603_21055_gb300.gicp import GicpTracker
    rng = np.random.default_rng(23)
    centre = np.array([3.0, 2.5, 1.5])
    room = synth.make_room(rng, keep_free=(centre, 1.1))
    pose = synth.keyframe_path(rng, 1, centre)[0]
    d, _ = synth.raycast(room, pose, W, H, F, F, W / 2.0, H / 2.0)
    depth = torch.as_tensor(d.astype(np.float32)).cuda()
    empty = torch.zeros(H, W, device="cuda")
    cam = synth.Camera(W, H, F, F, W / 2.0, H / 2.0, np.eye(4, dtype=np.float32)[:3].copy())
    tr = GicpTracker(src_capacity=W * H, map_capacity=1 << 15, stride=stride, k_cov=6, max_iters=3, tol=0.0)
    tr.frame(cam, depth)
    tr.set_pose(pose)
    tr.insert()
    start = np.array(pose, np.float64)
    start[:, 3] += 0.01
    for _ in range(20):
        tr.frame(cam, depth)
        tr.track(start)
        _, st = tr.result()
        assert st.status == 0 and st.iterations == 3
        tr.frame(cam, empty)
        tr.track(start)
        got, st = tr.result()
        assert st.status == 2 and st.iterations == 0 and st.n_matches == 0 and st.cost == 0.0
        assert np.array_equal(got, start)
        assert not tr.linearize(start.astype(np.float32)).any()
