"""The arrays of paths that a run does not take cost no memory of their own, and
runs of all paths on one plan, one after the other, do not read what is left of
one another."""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def workspace(**kw):
    from paper_1506_02226_gb300.api import Plan
    with Plan(**kw) as p:
        return B.dbscan_plan_workspace_bytes(p.handle)


@pytest.mark.parametrize("n", [3000, 100_000])
def test_warp_tiles_share_the_other_paths_memory(n):
    for max_d in (4, 8, 12, 16, 64):  # a plan of the CUDA-core test has no warp tiles
        assert workspace(max_n=n, max_d=max_d) == workspace(max_n=n, max_d=max_d, precision=B.DBSCAN_PREC_EXACT_SIMT)
    for max_d in (8, 16):  # without the grid's arrays: packed rows, counts, flags and parents, 45 or 77 bytes a point
        rest = workspace(max_n=n, max_d=max_d, grid=B.DBSCAN_GRID_OFF, precision=B.DBSCAN_PREC_EXACT_SIMT)
        assert workspace(max_n=n, max_d=max_d, grid=B.DBSCAN_GRID_OFF) <= rest + 45 * n + 65536


def test_served_jobs(n=50_000):
    sizes = {}
    for prec in (B.DBSCAN_PREC_AUTO, B.DBSCAN_PREC_EXACT_SIMT):
        o = B.dbscan_serve_opts_default()
        o.precision, o.max_n, o.slots = prec, n, 1
        s = B.dbscan_serve_create(o)
        try:
            sizes[prec] = {d: B.dbscan_serve_job_bytes(s, n, d) for d in (2, 3, 5, 8, 12, 16, 32)}
        finally:
            B.dbscan_serve_destroy(s)
    auto, simt = sizes[B.DBSCAN_PREC_AUTO], sizes[B.DBSCAN_PREC_EXACT_SIMT]
    for d in (2, 3, 5, 8, 16, 32):
        assert auto[d] == simt[d], d
    assert auto[12] <= simt[12] + 16 * n


def test_one_plan_all_paths():
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(9)

    def points(n, d, spread):
        c = rng.integers(80, 940, size=(6, d))
        u = c[rng.integers(0, 6, size=n)] + rng.integers(-spread, spread + 1, size=(n, d))
        loose = rng.random(n) < 0.1
        u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
        return (np.clip(u, 0, 1023) / 1024).astype(np.float32)

    #        n, d, spread, eps, min_pts, path
    runs = [(6000, 12, 30, 90, 6, B.DBSCAN_PATH_ALLPAIRS_SIMT),
            (7000, 3, 40, 6, 5, B.DBSCAN_PATH_GRID),            # ranks by the bitmap
            (6500, 2, 40, 12, 5, B.DBSCAN_PATH_GRID),           # direct ranks
            (1500, 3, 30, 12, 5, B.DBSCAN_PATH_GRID),           # one launch
            (6000, 5, 20, 14, 5, B.DBSCAN_PATH_GRID_PROJECTED),
            (5000, 20, 30, 130, 6, B.DBSCAN_PATH_ALLPAIRS_TC),
            (7000, 3, 60, 1.4, 2, B.DBSCAN_PATH_GRID)]          # hashed cells
    runs = [(points(n, d, s), float(np.float32(e / 1024)), m, path) for n, d, s, e, m, path in runs]
    order = [a for k in range(len(runs)) for a in (0, k, k, 0, (3 * k + 1) % len(runs))]
    for mode in (0, 1):
        want = [oracle.dbscan(x, eps, m, label_mode=mode) for x, eps, m, _ in runs]
        with Plan(max_n=7000, max_d=20, label_mode=mode) as p:
            for k in order:
                x, eps, m, path = runs[k]
                lab, cnt, core, st = p.run_detail(torch.from_numpy(x).cuda(), eps, m)
                assert st["path"] == path
                np.testing.assert_array_equal(lab.cpu().numpy(), want[k][0], err_msg=f"run {k} mode {mode}")
                np.testing.assert_array_equal(cnt.cpu().numpy(), want[k][1])
                assert st["n_core"] == int(want[k][2].sum())
