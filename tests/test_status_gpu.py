"""A run's status on every path: reported by the label kernel, or copied behind
the run, it names off-grid input once and not for the next run."""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,opts", [
    (300, 2, {}),                                                # one launch
    (5000, 3, {}),                                               # cells in key order
    (3000, 5, {}),                                               # projected grid
    (2000, 12, {}),                                              # warp tiles
    (2000, 12, {"precision": B.DBSCAN_PREC_EXACT_SIMT}),         # CUDA-core tiles
    (4500, 20, {}),                                              # tensor cores
    (5000, 3, {"label_mode": B.DBSCAN_LABEL_COMPACT}),           # kernels after the labels
])
@pytest.mark.parametrize("stats", [False, True])
def test_status_of_a_run(n, d, opts, stats):
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(n + d)
    u = np.clip(rng.integers(100, 900, size=(8, d))[rng.integers(0, 8, size=n)] + rng.integers(-9, 10, size=(n, d)), 0, 1023)
    x = (u / 1024).astype(np.float32)
    eps, min_pts = 8 * d / 1024, 5
    want = oracle.dbscan(x, eps, min_pts, label_mode=opts.get("label_mode", 0))[0]
    good = torch.from_numpy(x).cuda()
    bad = good.clone()
    bad[n - 1, d - 1] = 0.3
    with Plan(max_n=n, max_d=d, **opts) as p:
        for _ in range(2):
            with pytest.raises(B.DbscanError) as err:
                p.run(bad, eps, min_pts, stats=stats)
            assert err.value.status == B.DBSCAN_ERR_NOT_QUANTISED
            lab = p.run(good, eps, min_pts, stats=stats)
            lab = lab[0] if stats else lab
            np.testing.assert_array_equal(lab.cpu().numpy(), want)
