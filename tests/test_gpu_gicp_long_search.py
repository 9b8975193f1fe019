"""A track whose first iteration takes longer than a second because a single block has all the
work: 16 points whose searches each walk 4.2 million map points of one cell. The other blocks
wait that long and the track ends as any other; it used to give up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_blocks_wait_for_a_long_search():
    import torch
    from paper_2603_21055_gb300.gicp import GicpTracker
    n, k = 1 << 22, 16
    tr = GicpTracker(src_capacity=65536, map_capacity=n, r_max=60.0, max_iters=1, d_overlap=0.0)
    gen = torch.Generator(device="cuda").manual_seed(1)
    for s, m in ((tr.map, n), (tr.src, k)):
        s.pos[:m, :3] = 5.1 + 4.8 * torch.rand(m, 3, generator=gen, device="cuda")      # inside one cell of 10 m
        s.cov[:m, [0, 3, 5]] = 1.0
        s.normal[:m, 2] = 1.0
        s.count.fill_(m)
    tr.index()
    tr.track(np.eye(4)[:3])
    _, st = tr.result()
    assert st.status == 0 and st.iterations == 1 and st.n_matches == k
