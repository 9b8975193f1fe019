"""A track whose blocks gave up waiting for one another leaves a pose that is not its result.
The flag is set here by hand, after a track that ended well: it has to outlive the selection
of the next frame, which clears the set's flags, until the next track, and a sequence has to
end with an error instead of going on from such a pose."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H, F = 96, 72, 80.0
GAVE_UP = 204 // 4              # int32 word of the workspace: the last of the state's 208 bytes


def _problem():
    import torch
    from paper_2603_21055_gb300 import synth
    from paper_2603_21055_gb300.gicp import GicpTracker
    rng = np.random.default_rng(4)
    centre = np.array([3.0, 2.5, 1.5])
    room = synth.make_room(rng, keep_free=(centre, 1.1))
    pose = synth.keyframe_path(rng, 1, centre)[0]
    d, _ = synth.raycast(room, pose, W, H, F, F, W / 2.0, H / 2.0)
    cam = synth.Camera(W, H, F, F, W / 2.0, H / 2.0, np.eye(4, dtype=np.float32)[:3].copy())
    tr = GicpTracker(src_capacity=4096, map_capacity=8192, stride=2, k_cov=6, max_iters=4)
    return tr, cam, torch.as_tensor(d.astype(np.float32)).cuda(), pose


def test_flag_outlives_the_next_frame_and_ends_with_the_next_track():
    import torch
    tr, cam, depth, pose = _problem()
    tr.frame(cam, depth)
    tr.set_pose(pose)
    tr.insert()
    tr.track(pose)
    assert tr.result()[1].status == 0
    tr.ws.view(dtype=torch.int32)[GAVE_UP] = 1
    tr.frame(cam, depth)
    assert tr.result()[1].status == 4
    tr.track(pose)
    assert tr.result()[1].status == 0


@pytest.mark.parametrize("bad", [1, 2, 3, None])          # the frame whose track gives up; 3 is the last
def test_sequence_ends_with_an_error(bad):
    import torch
    from paper_2603_21055_gb300 import binding as B
    tr, cam, depth, pose = _problem()
    track, calls = tr.track, []

    def stub(guess):
        track(guess)
        calls.append(guess)
        if len(calls) == bad:
            tr.ws.view(dtype=torch.int32)[GAVE_UP] = 1
    tr.track = stub
    if bad is None:
        assert len(tr.track_sequence(cam, [depth] * 4, pose)) == 4
    else:
        with pytest.raises(B.SgadError) as e:
            tr.track_sequence(cam, [depth] * 4, pose)
        assert e.value.status == B.SGAD_ERR_TIMEOUT and len(calls) == bad
