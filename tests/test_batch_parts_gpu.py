"""A batch of more tiles than one part takes (2^20): every instance of every part
gets its labels and statistics."""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

INSTANCE = np.dtype({"names": ["points", "n", "d", "eps", "min_pts", "labels"],
                     "formats": ["<u8", "<i8", "<i4", "<f4", "<i4", "<u8"],
                     "offsets": [0, 8, 16, 20, 24, 32], "itemsize": 40})


def test_more_than_a_part():
    from paper_1506_02226_gb300.api import Plan
    rng = np.random.default_rng(5)
    sizes = np.array([3, 1, 0, 5, 2], dtype=np.int64)
    pool = [(rng.integers(0, 60, size=(s, 2)) / 1024).astype(np.float32) for s in sizes]
    eps, min_pts, count = 25 / 1024, 2, 1_400_003
    want = [oracle.dbscan(p, eps, min_pts)[0] if len(p) else np.zeros(0, np.int32) for p in pool]
    kind = np.arange(count) % len(pool)
    n = sizes[kind]
    first = np.concatenate([[0], np.cumsum(n)[:-1]])
    x = torch.from_numpy(np.concatenate(pool)).cuda()
    at = np.concatenate([[0], np.cumsum(sizes)[:-1]])[kind]
    labels = torch.full((int(n.sum()),), -9, dtype=torch.int32, device="cuda")
    assert (n > 0).sum() > 1 << 20
    t = np.zeros(count, INSTANCE)
    t["points"], t["n"], t["d"], t["eps"] = x.data_ptr() + 8 * at, n, 2, eps
    t["min_pts"], t["labels"] = min_pts, labels.data_ptr() + 4 * first
    insts = (B.dbscan_instance * count).from_buffer(t)
    st = (B.dbscan_stats * count)()
    with Plan(max_n=16, max_d=2) as p:
        assert B.dbscan_batch(p.handle, insts, st) == B.DBSCAN_OK
        # an off-grid instance in the first part: the call fails, the other parts' labels are as before
        good = labels.clone()
        bad = torch.full((3, 2), 0.3, device="cuda")
        t["points"][0] = bad.data_ptr()
        labels.fill_(-9)
        assert B.dbscan_batch(p.handle, insts) == B.DBSCAN_ERR_NOT_QUANTISED
        assert torch.equal(labels[-1000:], good[-1000:])
        t["points"][0] = x.data_ptr() + 8 * at[0]
        labels.fill_(-9)
        assert B.dbscan_batch(p.handle, insts) == B.DBSCAN_OK and torch.equal(labels, good)
    whole = np.concatenate(want)
    reps = -(-count // len(pool))
    np.testing.assert_array_equal(labels.cpu().numpy(), np.tile(whole, reps)[:len(labels)])
    got = np.frombuffer(st, dtype=np.dtype({"names": ["n_core"], "formats": ["<i8"],
                                            "offsets": [B.dbscan_stats.n_core.offset], "itemsize": 96}))["n_core"]
    cores = np.array([oracle.dbscan(p, eps, min_pts)[2].sum() if len(p) else 0 for p in pool])
    np.testing.assert_array_equal(got, cores[kind])
