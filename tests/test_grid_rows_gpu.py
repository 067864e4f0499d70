"""The eps-grid runs above 4,096 points against the oracle, bit for bit: cells in
key order with a direct table (plane), with the occupancy bitmap (space), and
the hashed table where neither fits; and the candidate pairs against the host's
count of the same cells.
"""
import numpy as np
import pytest

import bench
import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def blobs(rng, n, d, sigmas, loose):
    c = rng.integers(50, 970, size=(len(sigmas), d))
    k = rng.integers(0, len(sigmas), size=n)
    u = c[k] + np.rint(np.array(sigmas)[k, None] * rng.standard_normal((n, d))).astype(int)
    out = rng.random(n) < loose
    u[out] = rng.integers(0, 1024, size=(int(out.sum()), d))
    return u


CASES = {
    "plane": (2, 6.3, 5, lambda r, n: blobs(r, n, 2, [2, 5, 12, 30], 0.2)),
    "plane wide": (2, 40.0, 60, lambda r, n: blobs(r, n, 2, [2, 20, 60], 0.3)),
    "space": (3, 11.0, 6, lambda r, n: blobs(r, n, 3, [2, 6, 15, 25], 0.3)),
    "space tiny eps": (3, 1.5, 2, lambda r, n: blobs(r, n, 3, [1, 4, 9], 0.2)),  # 1024^3 cells: hashed
    "line": (1, 0.5, 4, lambda r, n: r.integers(0, 1024, size=(n, 1))),
    "line wide": (1, 3.0, 3, lambda r, n: 7 * r.integers(0, 146, size=(n, 1)) % 1024),
    "strips": (2, 8.9, 4, lambda r, n: np.stack([r.integers(0, 1024, n), 9 * r.integers(0, 100, n)], 1)),
    "edges": (3, 30.0, 5, lambda r, n: np.where(r.random((n, 3)) < 0.5, r.integers(0, 20, (n, 3)),
                                                r.integers(1000, 1024, (n, 3)))),
    "one cell": (2, 900.0, 3, lambda r, n: r.integers(0, 300, size=(n, 2))),
}


@pytest.mark.parametrize("name", list(CASES))
def test_grid_run(name):
    from paper_1506_02226_gb300.api import Plan
    d, eps_units, min_pts, make = CASES[name]
    rng = np.random.default_rng(len(name) + d)
    for n in (4097, 20011):
        x = np.ascontiguousarray(np.clip(make(rng, n), 0, 1023).astype(np.float32) / np.float32(1024))
        xt = torch.from_numpy(x).cuda()
        eps = float(np.float32(eps_units / 1024))
        for mode in (0, 1):
            want, cnt, core = oracle.dbscan(x, eps, min_pts, label_mode=mode)
            with Plan(max_n=n, max_d=d, label_mode=mode) as p:
                lab, c, k, st = p.run_detail(xt, eps, min_pts)
                np.testing.assert_array_equal(c.cpu().numpy(), cnt)
                np.testing.assert_array_equal(k.cpu().numpy().astype(bool), core)
                np.testing.assert_array_equal(lab.cpu().numpy(), want, err_msg=f"n={n} mode={mode}")
                assert st["path"] == B.DBSCAN_PATH_GRID
                assert st["n_core"] == int(core.sum()) and st["n_core"] + st["n_border"] + st["n_noise"] == n
                assert st["n_clusters"] == len(set(want[core].tolist()))
                assert st["candidate_pairs"] == bench.grid_candidate_pairs(x, eps)
                assert p.pair_tests()[0] <= st["candidate_pairs"] and st["pair_tests"] == sum(p.pair_tests())
                np.testing.assert_array_equal(p.run(xt, eps, min_pts).cpu().numpy(), want)  # counts stop early
    bad = xt.clone()
    bad[n - 1, d - 1] = 0.3
    with Plan(max_n=n, max_d=3, synchronous=False) as p:  # an error stays until it is asked for
        p.run(bad, eps, min_pts)
        lab = p.run(xt, eps, min_pts)
        assert p.sync() == B.DBSCAN_ERR_NOT_QUANTISED
        np.testing.assert_array_equal(lab.cpu().numpy(), oracle.dbscan(x, eps, min_pts)[0])
