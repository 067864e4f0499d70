"""The eps-grid kernels that serve any size (grid.cu), at small sizes, against the
oracle, bit for bit: cells in a direct table, hashed with the occupancy bitmap
and without, in one to three dimensions; sizes around blocks and the other grid
kernels' limits; dense cells and lattices; an error that outlasts a good run.
"""
import numpy as np
import pytest

import bench
import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def blobs(rng, n, d, sigma, loose=0.2):
    c = rng.integers(60, 960, size=(5, d))
    u = c[rng.integers(0, 5, size=n)] + np.rint(sigma * rng.standard_normal((n, d))).astype(int)
    out = rng.random(n) < loose
    u[out] = rng.integers(0, 1024, size=(int(out.sum()), d))
    return u


# d, eps in units, min_pts, points, max_n (which sizes the cell table and the bitmap)
CASES = {
    "line direct": (1, 3.0, 3, lambda r, n: blobs(r, n, 1, 20), 9001),
    "plane direct": (2, 25.0, 8, lambda r, n: blobs(r, n, 2, 25), 9001),
    "plane bitmap": (2, 3.1, 4, lambda r, n: blobs(r, n, 2, 8), 9001),
    "plane finest": (2, 1.2, 2, lambda r, n: blobs(r, n, 2, 5), 4000),  # 2^20 cells, 2^15 words of bits: just fit
    "space direct": (3, 90.0, 9, lambda r, n: blobs(r, n, 3, 40), 9001),
    "space bitmap": (3, 16.5, 5, lambda r, n: blobs(r, n, 3, 12), 9001),
    "space hashed": (3, 9.0, 5, lambda r, n: blobs(r, n, 3, 9), 9001),
    "space finest": (3, 1.5, 2, lambda r, n: blobs(r, n, 3, 3), 9001),
    "dense cells": (2, 7.0, 40, lambda r, n: np.array([[100, 100], [112, 100], [900, 20]])[r.integers(0, 3, n)]
                    + r.integers(-2, 3, size=(n, 2)), 9001),
    "lattice": (3, 19.9, 3, lambda r, n: r.integers(0, 12, size=(n, 3)) * 21 + r.integers(0, 2, size=(n, 3)), 9001),
}


@pytest.mark.parametrize("name", list(CASES))
def test_general_grid_run(name):
    from paper_1506_02226_gb300.api import Plan
    d, eps_units, min_pts, make, max_n = CASES[name]
    rng = np.random.default_rng(len(name) + 10 * d)
    eps = float(np.float32(eps_units / 1024))
    for n in (1, 33, 257, 2048, 2049, 4096, 9001):
        if n > max_n:
            continue
        x = np.ascontiguousarray(np.clip(make(rng, n), 0, 1023).astype(np.float32) / np.float32(1024))
        xt = torch.from_numpy(x).cuda()
        for mode in (0, 1):
            want, cnt, core = oracle.dbscan(x, eps, min_pts, label_mode=mode)
            with Plan(max_n=max_n, max_d=d, label_mode=mode, profile=True) as p:
                B.dbscan_plan_test_hook(p.handle, B.DBSCAN_HOOK_GRID_GENERAL)
                lab, c, flags, st = p.run_detail(xt, eps, min_pts)
                assert "grid_nbrs" in {k for k, _ in p.phase_times()}  # only this chain lists neighbours
                assert st["path"] == B.DBSCAN_PATH_GRID
                np.testing.assert_array_equal(c.cpu().numpy(), cnt)
                np.testing.assert_array_equal(flags.cpu().numpy().astype(bool), core)
                np.testing.assert_array_equal(lab.cpu().numpy(), want, err_msg=f"n={n} mode={mode}")
                assert st["n_core"] == int(core.sum()) and st["n_core"] + st["n_border"] + st["n_noise"] == n
                assert st["n_clusters"] == len(set(want[core].tolist()))
                assert st["candidate_pairs"] == bench.grid_candidate_pairs(x, eps)
                B.dbscan_plan_test_hook(p.handle, B.DBSCAN_HOOK_GRID_GENERAL)
                np.testing.assert_array_equal(p.run(xt, eps, min_pts).cpu().numpy(), want)  # counts stop early
                np.testing.assert_array_equal(p.run(xt, eps, min_pts).cpu().numpy(), want)  # the hook is consumed
                if n <= 2048:  # (above, the finest grids have no other kernels)
                    assert "grid_nbrs" not in {k for k, _ in p.phase_times()}
    bad = xt.clone()
    bad[len(x) - 1, d - 1] = 0.3
    with Plan(max_n=len(x), max_d=d) as p:
        B.dbscan_plan_test_hook(p.handle, B.DBSCAN_HOOK_GRID_GENERAL)
        with pytest.raises(B.DbscanError) as err:
            p.run(bad, eps, min_pts)
        assert err.value.status == B.DBSCAN_ERR_NOT_QUANTISED
    with Plan(max_n=len(x), max_d=d, synchronous=False) as p:
        for pts in (bad, xt):
            B.dbscan_plan_test_hook(p.handle, B.DBSCAN_HOOK_GRID_GENERAL)
            lab = p.run(pts, eps, min_pts)
        assert p.sync() == B.DBSCAN_ERR_NOT_QUANTISED
        np.testing.assert_array_equal(lab.cpu().numpy(), oracle.dbscan(x, eps, min_pts)[0])
        assert p.sync() == 0
