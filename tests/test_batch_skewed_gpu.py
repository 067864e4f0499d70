"""A batch of a few large instances among many small ones, whose tiles are laid
out in another order than the instances: labels, per-instance statistics and pair
counts against the oracle and against each instance alone."""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B
from paper_1506_02226_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def instance(rng, n, d):
    c = rng.integers(100, 900, size=(4, d))
    u = c[rng.integers(0, 4, size=n)] + rng.integers(-40, 41, size=(n, d)) if n else np.zeros((0, d), int)
    return inputs.Instance((np.clip(u, 0, 1023) / 1024).astype(np.float32), float(np.float32(9 * np.sqrt(d) / 1024)), 4)


@pytest.mark.parametrize("mode", [0, 1])
def test_large_among_small(mode):
    from paper_1506_02226_gb300.api import Plan, make_instances
    rng = np.random.default_rng(31 + mode)
    sizes = [64] * 150 + [17_001, 0, 4096, 4097, 1] + [63, 65] * 40 + [20_480, 9000] + [3] * 60
    insts = [instance(rng, n, (2, 3, 9)[k % 3]) for k, n in enumerate(sizes)]

    def run(batch, p):
        items = [(torch.from_numpy(i.points).cuda(), i.eps, i.min_pts,
                  torch.full((i.n,), -9, dtype=torch.int32, device="cuda")) for i in batch]
        st = (B.dbscan_stats * len(batch))()
        assert B.dbscan_batch(p.handle, make_instances(items), st) == B.DBSCAN_OK
        return [it[3].cpu().numpy() for it in items], st

    with Plan(max_n=16, max_d=16, label_mode=mode) as p:
        for _ in range(2):
            labs, st = run(insts, p)
            for k, (inst, lab) in enumerate(zip(insts, labs)):
                if not inst.n:
                    continue
                want, _, core = oracle.dbscan(inst.points, inst.eps, inst.min_pts, label_mode=mode)
                np.testing.assert_array_equal(lab, want, err_msg=f"instance {k} n={inst.n}")
                noise = int((want < 0).sum())
                assert (st[k].n_core, st[k].n_noise) == (int(core.sum()), noise)
                assert st[k].n_border == inst.n - int(core.sum()) - noise
                assert st[k].n_clusters == len(set(want[core].tolist()))
        alone, st1 = run(insts[150:151], p)  # a smaller batch on the same plan
        np.testing.assert_array_equal(alone[0], labs[150])
        assert st1[0].n_core == st[150].n_core
