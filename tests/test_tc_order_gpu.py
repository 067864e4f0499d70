"""The tensor-core path's ordering and tile-pair cull against the oracle, bit for bit.

From 32,768 points on, points are grouped by sampled pivots and tile pairs that
the triangle inequality proves empty are skipped; row units leave the count
early and merged tile pairs are skipped.  None of it may change a count, a core
flag or a label: inputs with well separated groups (most tile pairs skipped),
with none at all (nothing skipped), one dense group (every unit leaves early),
chains of touching groups and many equal points, at sizes around the limit, the
256-point tiles and the pivot counts.
"""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PRECS = [("fp16", B.DBSCAN_PREC_FP16_GRAM), ("bf16", B.DBSCAN_PREC_BF16_GRAM)]


def points(kind, n, d, seed):
    rng = np.random.default_rng(seed)
    if kind == "groups":  # one group per 1,500 points, 15% scattered
        c = rng.integers(80, 944, size=(max(2, n // 1500), d))
        u = c[rng.integers(0, len(c), size=n)] + np.rint(20 * rng.standard_normal((n, d))).astype(int)
        loose = rng.random(n) < 0.15
        u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
        return u, 20 * np.sqrt(2 * d) * 0.92, 8
    if kind == "scattered":  # no structure; eps reaches a few points
        u = rng.integers(0, 1024, size=(n, d))
        D = ((u[1:3000] - u[0]) ** 2).sum(1)
        return u, float(np.sqrt(np.quantile(D, 0.002))), 6
    if kind == "dense":  # almost every pair of one group are neighbours
        u = 500 + np.rint(9 * rng.standard_normal((n, d))).astype(int)
        u[rng.integers(0, n, size=n // 50)] = rng.integers(0, 1024, size=(n // 50, d))
        return u, 9 * np.sqrt(2 * d) * 1.1, 12
    if kind == "chain":  # groups a little over eps long, end to end, in random order
        t = rng.integers(0, 900, size=n)
        u = 60 + t[:, None] + rng.integers(-3, 4, size=(n, d))
        return u, 14 * np.sqrt(d), 5
    u = rng.integers(0, 1024, size=(40, d))[rng.integers(0, 40, size=n)]  # 40 distinct points
    return u, 3.0, 700


@pytest.mark.parametrize("name,prec", PRECS)
@pytest.mark.parametrize("kind,n,d", [("groups", 32767, 32), ("groups", 32768, 64), ("groups", 65600, 17),
                                      ("scattered", 33025, 16), ("dense", 40001, 32), ("chain", 33111, 48),
                                      ("equal", 32769, 24)])
def test_ordered_path_matches_oracle(name, prec, kind, n, d):
    from paper_1506_02226_gb300.api import Plan
    u, eps_units, min_pts = points(kind, n, d, 900 + n + d)
    x = np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024)
    x = np.ascontiguousarray(x[np.random.default_rng(n).permutation(n)])
    eps = float(np.float32(eps_units / 1024))
    want_lab, want_cnt, want_core = oracle.dbscan(x, eps, min_pts)
    xt = torch.from_numpy(x).cuda()
    with Plan(max_n=n, max_d=d, precision=prec) as p:
        lab, cnt, core, st = p.run_detail(xt, eps, min_pts)
        assert st["path"] == B.DBSCAN_PATH_ALLPAIRS_TC
        np.testing.assert_array_equal(cnt.cpu().numpy(), want_cnt)
        np.testing.assert_array_equal(core.cpu().numpy().astype(bool), want_core)
        np.testing.assert_array_equal(lab.cpu().numpy(), want_lab)
        assert st["n_core"] == int(want_core.sum())
        assert st["n_core"] + st["n_border"] + st["n_noise"] == n
        assert st["n_clusters"] == len(set(want_lab[want_core].tolist()))
        np.testing.assert_array_equal(p.run(xt, eps, min_pts).cpu().numpy(), want_lab)  # early exits
        few = p.run(xt[:5001].contiguous(), eps, min_pts).cpu().numpy()  # the plan again, below the limit
        np.testing.assert_array_equal(few, oracle.dbscan(x[:5001], eps, min_pts)[0])
