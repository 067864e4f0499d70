"""The warp-tile all-pairs path (d <= 16, default precision) against the oracle, bit for bit.

Sizes around the 64-row tiles and the column chunks, every dimension class with
the grid off or absent, thresholds at pair distances of coordinates at the
grid's ends, early leave against exact counts, equal points, no core point at
all, and one plan used for several sizes and dimensions.
"""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def blobs(seed, n, d, spread, k):
    rng = np.random.default_rng(seed)
    c = rng.integers(spread, 1024 - spread, size=(k, d))
    u = c[rng.integers(0, k, size=n)] + rng.integers(-spread, spread + 1, size=(n, d))
    loose = rng.random(n) < 0.12
    u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
    return u


def check(plan, u, eps_units, min_pts, mode=0):
    x = np.ascontiguousarray(np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024))
    eps = float(np.float32(eps_units / 1024))
    want, cnt, core = oracle.dbscan(x, eps, min_pts, label_mode=mode)
    xt = torch.from_numpy(x).cuda()
    lab, c, k, st = plan.run_detail(xt, eps, min_pts)
    assert st["path"] == B.DBSCAN_PATH_ALLPAIRS_SIMT
    np.testing.assert_array_equal(c.cpu().numpy(), cnt)
    np.testing.assert_array_equal(k.cpu().numpy().astype(bool), core)
    np.testing.assert_array_equal(lab.cpu().numpy(), want)
    assert st["n_core"] == int(core.sum()) and st["n_core"] + st["n_border"] + st["n_noise"] == len(x)
    assert st["n_clusters"] == len(set(want[core].tolist()))
    np.testing.assert_array_equal(plan.run(xt, eps, min_pts).cpu().numpy(), want)  # rows left early


@pytest.mark.parametrize("d", [1, 2, 3, 5, 9, 12, 16])
@pytest.mark.parametrize("mode", [0, 1])
def test_sizes(d, mode):
    from paper_1506_02226_gb300.api import Plan
    with Plan(max_n=3000, max_d=16, grid=B.DBSCAN_GRID_OFF, label_mode=mode) as p:
        for n in (1, 2, 31, 33, 63, 64, 65, 129, 513, 3000, 700):
            check(p, blobs(10 * n + d, n, d, 10 + 4 * d, 4), 13 * np.sqrt(d), 4, mode)


def test_many_chunks():
    from paper_1506_02226_gb300.api import Plan
    with Plan(max_n=20011, max_d=12) as p:
        check(p, blobs(5, 20011, 12, 60, 9), 150, 12)
        check(p, blobs(6, 20011, 12, 60, 9), 60, 12)  # hardly any core point
        check(p, blobs(7, 9000, 9, 15, 40), 45, 6)


def test_extremes_and_degenerate():
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(8)
    with Plan(max_n=2000, max_d=16, grid=B.DBSCAN_GRID_OFF) as p:
        for d in (9, 16):
            u = rng.choice([0, 1, 511, 512, 1022, 1023], size=(1500, d))
            D = np.unique(((u[:, None, :] - u[None, :30, :]) ** 2).sum(2))
            for v in (D[1], D[len(D) // 2], D[-1]):
                for off in (-0.25, 0.25):
                    check(p, u, np.sqrt(v + off), 5)
        check(p, rng.integers(0, 1024, size=(900, 4)), 0.4, 2)  # duplicates only
        check(p, np.full((1000, 7), 1023), 0.5, 1000)
        check(p, np.full((1000, 7), 0), 0.5, 1001)
        x = torch.full((100, 3), 0.3, device="cuda")
        with pytest.raises(B.DbscanError) as err:
            p.run(x, 0.1, 3)
        assert err.value.status == B.DBSCAN_ERR_NOT_QUANTISED
