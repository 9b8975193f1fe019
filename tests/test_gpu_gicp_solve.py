"""The tracking kernel's Gauss-Newton solve and pose update in FP64, against the same step on
the host from the system that sgad_gicp_linearize returns (the two sum the same FP32 terms
exactly, so they solve the same system). A factorisation of a 6 x 6 system with correctly
rounded operations leaves at most about 6^2 roundings, each amplified by the system's
condition: 40 eps cond |xi|, plus the rounding of the pose's elements (below 8 m, a few
products each): 1e-14."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H, F = 160, 120, 150.0


@pytest.mark.parametrize("flat", [False, True])          # flat: a wall alone, whose slides are weakly held
@pytest.mark.parametrize("shift,turn", [(0.0, 0.0), (0.02, 0.01), (0.05, 0.12)])
def test_one_step_matches_the_host(flat, shift, turn):
    import torch
    from paper_2603_21055_gb300 import synth
    from paper_2603_21055_gb300.gicp import GicpTracker
    rng = np.random.default_rng(31)
    centre = np.array([3.0, 2.5, 1.5])
    room = synth.make_room(rng, keep_free=(centre, 1.1))
    pose = synth.keyframe_path(rng, 1, centre)[0]
    d, _ = synth.raycast(room, pose, W, H, F, F, W / 2.0, H / 2.0)
    d = (np.full((H, W), 2.0) if flat else d) + rng.normal(scale=0.002, size=(H, W))
    depth = torch.as_tensor(d.astype(np.float32)).cuda()
    cam = synth.Camera(W, H, F, F, W / 2.0, H / 2.0, np.eye(4, dtype=np.float32)[:3].copy())
    tr = GicpTracker(src_capacity=W * H, map_capacity=1 << 15, stride=2, k_cov=8, max_iters=1, tol=0.0, r_max=0.3)
    tr.frame(cam, depth)
    tr.set_pose(pose)
    tr.insert()
    P = np.array(pose, np.float64)
    P[:, :3] = synth.rotation_about(np.array([0.6, 0.0, 0.8]), turn) @ P[:, :3]
    P[:, 3] += shift
    P = P.astype(np.float32).astype(np.float64)            # the pose that both evaluate the terms at
    s = tr.linearize(P.astype(np.float32))
    A = np.zeros((6, 6))
    A[np.triu_indices(6)] = s[:21]
    A = np.triu(A) + np.triu(A, 1).T
    xi = np.linalg.solve(A, -s[21:27])
    th = np.linalg.norm(xi[:3])
    K = np.array([[0, -xi[2], xi[1]], [xi[2], 0, -xi[0]], [-xi[1], xi[0], 0]])
    # (1 - cos) / th^2 without its cancellation
    a, b = (np.sin(th) / th, 2 * np.sin(th / 2) ** 2 / th ** 2) if th > 0 else (1.0, 0.5)
    E = np.eye(3) + a * K + b * (K @ K)
    want = np.hstack([E @ P[:, :3], E @ P[:, 3:] + xi[3:, None]])
    tr.track(P)
    got, st = tr.result()
    assert st.status == 0 and st.iterations == 1 and st.n_matches == int(s[28])
    eps = np.finfo(np.float64).eps
    tol = 40 * eps * np.linalg.cond(A) * np.linalg.norm(xi) + 1e-14
    assert np.abs(got - want).max() <= tol
    assert abs(st.step - np.linalg.norm(xi)) <= tol
