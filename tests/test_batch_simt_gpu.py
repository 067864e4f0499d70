"""A batch on a plan that asks for the CUDA-core pair test runs it, with the
results of the default: against the oracle, at sizes around tiles and chunks,
every dimension class, and the grid's end units."""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B
from paper_1506_02226_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def instances():
    rng = np.random.default_rng(12)
    out = []
    for k, n in enumerate((1, 2, 31, 33, 64, 65, 129, 700, 4100)):
        for d in (1, 2, 3, 4, 8, 9, 16)[k % 2::2]:
            c = rng.integers(60, 960, size=(4, d))
            u = c[rng.integers(0, 4, size=n)] + rng.integers(-25, 26, size=(n, d))
            out.append((u, 14 * np.sqrt(d), 4))
    ends = rng.choice([0, 1, 511, 512, 1022, 1023], size=(600, 16))
    D = np.unique(((ends[:, None, :] - ends[None, :30, :]) ** 2).sum(2))
    out += [(ends, np.sqrt(v + off), 5) for v in (D[1], D[len(D) // 2], D[-1]) for off in (-0.25, 0.25)]
    return [inputs.Instance((u / 1024).astype(np.float32), float(np.float32(e / 1024)), m) for u, e, m in out]


@pytest.mark.parametrize("mode", [0, 1])
def test_cuda_core_batch(mode):
    from paper_1506_02226_gb300.api import Plan, make_instances
    insts = instances()
    names, stats = {}, {}
    for prec in (B.DBSCAN_PREC_AUTO, B.DBSCAN_PREC_EXACT_SIMT):
        for profile in (False, True):
            items = [(torch.from_numpy(i.points).cuda(), i.eps, i.min_pts,
                      torch.full((i.n,), -9, dtype=torch.int32, device="cuda")) for i in insts]
            st = (B.dbscan_stats * len(insts))()
            with Plan(max_n=16, max_d=16, precision=prec, label_mode=mode, profile=profile) as p:
                assert B.dbscan_batch(p.handle, make_instances(items), st) == B.DBSCAN_OK
                if profile:
                    names[prec] = {n for n, _ in p.phase_times()}
            for k, (inst, it) in enumerate(zip(insts, items)):
                want = oracle.dbscan(inst.points, inst.eps, inst.min_pts, label_mode=mode)[0]
                np.testing.assert_array_equal(it[3].cpu().numpy(), want, err_msg=f"instance {k} n={inst.n} d={inst.d}")
        stats[prec] = [(s.n_core, s.n_border, s.n_noise, s.n_clusters) for s in st]
    assert stats[B.DBSCAN_PREC_AUTO] == stats[B.DBSCAN_PREC_EXACT_SIMT]
    passes = {"batch_count", "batch_core", "batch_union_near", "batch_union", "batch_border"}
    assert passes <= names[B.DBSCAN_PREC_AUTO]
    assert {n + "_simt" for n in passes} <= names[B.DBSCAN_PREC_EXACT_SIMT]
    assert not passes & names[B.DBSCAN_PREC_EXACT_SIMT]
