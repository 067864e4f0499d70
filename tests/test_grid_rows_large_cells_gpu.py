"""Two neighbouring cells of the eps-grid whose point pairs are more than an int
holds (46,401 x 46,401 > 2^31) go to the warp search's list, not to one lane.

In either cell one point is core, so the search itself is short: a bulk of equal
points, one more point at the cell's other edge, and a group that only this one
reaches.  min_pts lies between what the bulk and what that point sees.
"""
import numpy as np
import pytest

from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BULK, GROUP, PAIRS_SLOT = 46_400, 600, 30


def test_pair_of_large_cells_is_listed():
    from paper_1506_02226_gb300.api import Plan
    # eps 10 units: cells of 8; cells 0 and 2 along y are neighbours, their points 20 apart
    parts = []
    for y in (0, 20):
        parts += [np.tile([0, y], (BULK, 1)), np.array([[6, y]]), np.tile([16, y], (GROUP, 1))]
    u = np.concatenate(parts)
    half = BULK + 1 + GROUP
    want = np.repeat(np.array([BULK, half + BULK], dtype=np.int32), half)
    x = torch.from_numpy((u / 1024).astype(np.float32)).cuda()
    with Plan(max_n=len(u), max_d=2) as p:
        lab, st = p.run(x, 10 / 1024, BULK + GROUP // 2, stats=True)
        assert st["path"] == B.DBSCAN_PATH_GRID and (st["n_core"], st["n_clusters"], st["n_noise"]) == (2, 2, 0)
        np.testing.assert_array_equal(lab.cpu().numpy(), want)
        assert p.counters()[PAIRS_SLOT] & 0xFFFFFFFF == 1
