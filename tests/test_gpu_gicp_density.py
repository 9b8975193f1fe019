"""Maps of every density the index has cells for: correspondences and the map update against the
oracle, bit for bit, where few points share a cell and where hundreds do (the index then links
smaller cells, of which more rings have to be searched), for points on the map's surface, above
it near the search radius and out of reach. A tracker's index is built for each density in turn,
dense and sparse ones after each other."""
import numpy as np
import pytest

from oracle import gicp as G

pytestmark = pytest.mark.gpu

R_MAX, CELL = 0.2, 0.2 * 1.001 / 2
LEVEL = 208 // 4                    # int32 word of the workspace: the index's cell level


def _surface(rng, n):
    """n points of a rough plane over 10 x 10 cells of half the radius, in one layer of cells of
    every level."""
    p = rng.uniform(0.0005, 10 * CELL - 0.0005, (n, 3))
    p[:, 2] = 20.25 * CELL + rng.uniform(-0.005, 0.005, n)
    nr = np.array([0.0, 0.0, 1.0]) + 0.1 * rng.normal(size=(n, 3))
    return p.astype(np.float32), (nr / np.linalg.norm(nr, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("d_overlap", [0.01, 0.2])            # a fraction of the radius, and all of it
@pytest.mark.parametrize("k_match", [1, 8])
def test_index_of_every_density_matches_the_oracle(k_match, d_overlap):
    import torch
    from paper_2603_21055_gb300.gicp import GicpTracker
    rng = np.random.default_rng(12)
    tr = GicpTracker(src_capacity=1024, map_capacity=1 << 15, k_match=k_match, r_max=R_MAX, d_overlap=d_overlap)
    eye = np.eye(4, dtype=np.float32)[:3].copy()
    seen = set()
    # points per cell of half the radius, and the level of its cells
    for per_cell, level in [(5, 0), (30, 1), (3, 0), (50, 2), (120, 3), (40, 3), (150, 3), (2, 0), (0.01, 0)]:
        n = max(1, int(100 * per_cell))
        pos, nrm = _surface(rng, n)
        tr.map.load(pos, np.tile(np.eye(3), (n, 1, 1)), nrm)
        tr.index()
        assert int(tr.ws.view(torch.int32)[LEVEL]) == level, per_cell
        seen.add(level)
        src, _ = _surface(rng, 240)
        src[60:120, 2] += rng.uniform(0.0, 0.05, 60).astype(np.float32)
        src[120:180, 2] += rng.uniform(0.1, 0.205, 60).astype(np.float32)       # around the radius
        src[180:, 2] += np.float32(0.5)                                          # out of reach
        src[200:220, :2] += np.float32(0.9)                                      # beside the patch
        tr.src.load(src, np.tile(np.eye(3), (240, 1, 1)), np.tile(np.array([0.0, 0.0, 1.0]), (240, 1)))
        idx = torch.full((1024,), -7, dtype=torch.int32, device="cuda")
        tr.correspond(eye, idx)
        want = G.correspond(src, eye, pos, nrm, R_MAX, k_match)
        assert np.array_equal(idx[:240].cpu().numpy(), want), per_cell
        tr.set_pose(eye.astype(np.float64))
        tr.insert()
        ref = G.insert(dict(points=pos, cov=np.tile(np.eye(3), (n, 1, 1)), normal=nrm),
                       dict(points=src, cov=np.tile(np.eye(3), (240, 1, 1)), normal=np.tile([0.0, 0.0, 1.0], (240, 1))),
                       eye, d_overlap)
        assert np.array_equal(tr.map.host()[0], ref["points"]), per_cell
    assert seen == {0, 1, 2, 3}
