"""The one-launch eps-grid run (d <= 3, up to 2,048 points) against the oracle, bit for bit.

Sizes around a block's share of the points and the limit, sparse points (one a
cell), dense cells whose pairs go to whole warps, lattices whose cell pairs
mostly hold no neighbours, thresholds at pair distances, exact counts, both
label modes, statistics, asynchronous plans and off-grid input.
"""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def points(kind, n, d, rng):
    if kind == "sparse":
        return rng.integers(0, 1024, size=(n, d)), 30.0, 2
    if kind == "dense":  # a few hundred points a cell, blobs that nearly touch
        c = np.array([[200, 300, 100], [212, 300, 100], [600, 700, 900]])[:, :d]
        return c[rng.integers(0, 3, size=n)] + rng.integers(-3, 4, size=(n, d)), 6.5, 20
    if kind == "lattice":  # small groups on a lattice just over eps apart
        g = rng.integers(0, 12, size=(n, d)) * 21
        return g + rng.integers(0, 2, size=(n, d)), 19.9, 3
    c = rng.integers(40, 980, size=(6, d))
    u = c[rng.integers(0, 6, size=n)] + np.rint(15 * rng.standard_normal((n, d))).astype(int)
    loose = rng.random(n) < 0.15
    u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
    return u, 12.0, 5


@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("kind", ["sparse", "dense", "lattice", "blobs"])
def test_small_grid_run(kind, d):
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(40 * d + len(kind))
    for n in (1, 2, 7, 8, 9, 511, 513, 2000, 2047, 2048, 2049, 4096):
        u, eps_units, min_pts = points(kind, n, d, rng)
        x = np.ascontiguousarray(np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024))
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
                assert (st["kernels"] == 1) == (n <= 2048)
                assert st["n_core"] == int(core.sum()) and st["n_core"] + st["n_border"] + st["n_noise"] == n
                assert st["n_clusters"] == len(set(want[core].tolist()))
                assert st["candidate_pairs"] >= int(cnt.sum()) and st["pair_tests"] == sum(p.pair_tests())
                np.testing.assert_array_equal(p.run(xt, eps, min_pts).cpu().numpy(), want)


def test_errors_and_asynchronous_plans():
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(1)
    u, eps_units, min_pts = points("blobs", 3000, 2, rng)
    x = np.ascontiguousarray(np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024))
    eps = float(np.float32(eps_units / 1024))
    want = oracle.dbscan(x, eps, min_pts)[0]
    good, bad = torch.from_numpy(x).cuda(), torch.from_numpy(x).cuda()
    bad[2999, 1] = 0.3
    with Plan(max_n=3000, max_d=2) as p:
        with pytest.raises(B.DbscanError) as err:
            p.run(bad, eps, min_pts)
        assert err.value.status == B.DBSCAN_ERR_NOT_QUANTISED
        np.testing.assert_array_equal(p.run(good, eps, min_pts).cpu().numpy(), want)
    with Plan(max_n=3000, max_d=2, synchronous=False) as p:
        p.run(bad, eps, min_pts)
        lab = p.run(good, eps, min_pts)  # the first run's error stays until it is asked for
        assert p.sync() == B.DBSCAN_ERR_NOT_QUANTISED
        np.testing.assert_array_equal(lab.cpu().numpy(), want)
        assert p.sync() == 0
