"""The eps-grid kernels on either side of the one-launch kernel's limit (2,048
points), against the oracle and the host's count of candidate pairs: the largest
and ragged sizes of the one launch with an error that outlasts a good run on an
asynchronous plan, and the smallest sizes of the key-ordered cells."""
import numpy as np
import pytest

import bench
import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def points(rng, n, d):
    c = rng.integers(60, 960, size=(6, d))
    u = c[rng.integers(0, 6, size=n)] + np.rint(14 * rng.standard_normal((n, d))).astype(int)
    loose = rng.random(n) < 0.2
    u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
    return np.ascontiguousarray(np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024))


@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("n", [7, 1025, 2047, 2048, 2049, 2050, 3000])
def test_errors_of_asynchronous_plans(n, d):
    from paper_1506_02226_gb300.api import Plan
    x, eps, min_pts = points(np.random.default_rng(n + d), n, d), 9 / 1024, 4
    good, bad = torch.from_numpy(x).cuda(), torch.from_numpy(x).cuda()
    bad[n - 1, d - 1] = 0.3
    for mode in (0, 1):
        want = oracle.dbscan(x, eps, min_pts, label_mode=mode)[0]
        with Plan(max_n=n, max_d=d, label_mode=mode, synchronous=False) as p:
            first = p.run(good, eps, min_pts)
            p.run(bad, eps, min_pts)
            lab = p.run(good, eps, min_pts)  # the error stays until it is asked for
            assert p.sync() == B.DBSCAN_ERR_NOT_QUANTISED
            np.testing.assert_array_equal(first.cpu().numpy(), want)
            np.testing.assert_array_equal(lab.cpu().numpy(), want)
            assert p.sync() == 0
            np.testing.assert_array_equal(p.run(good, eps, min_pts).cpu().numpy(), want)
            assert p.sync() == 0


@pytest.mark.parametrize("d", [1, 2, 3])
def test_key_ordered_cells_at_their_smallest(d):
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(90 + d)
    for n in (2049, 2050, 2111, 2559, 3000, 4095, 4096):
        for eps_units in (2.5, 9.0, 40.0):
            x, eps = points(rng, n, d), float(np.float32(eps_units / 1024))
            xt = torch.from_numpy(x).cuda()
            want, cnt, core = oracle.dbscan(x, eps, 5)
            with Plan(max_n=n, max_d=d) as p:
                lab, c, flags, st = p.run_detail(xt, eps, 5)
                assert st["path"] == B.DBSCAN_PATH_GRID and st["kernels"] > 1
                np.testing.assert_array_equal(lab.cpu().numpy(), want, err_msg=f"n={n} eps={eps_units}")
                np.testing.assert_array_equal(c.cpu().numpy(), cnt)
                np.testing.assert_array_equal(flags.cpu().numpy().astype(bool), core)
                assert st["candidate_pairs"] == bench.grid_candidate_pairs(x, eps)
                np.testing.assert_array_equal(p.run(xt, eps, 5).cpu().numpy(), want)
