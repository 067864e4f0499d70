"""The batch's warp tiles against the oracle, bit for bit.

Rows run 64 to a tile and 32 to a warp, on FP16 matrix instructions whose sums
stay exact integers.  Sizes around the tiles, the warps and the largest sorted
instance, every dimension class, coordinates at the grid's ends (dot products
up to 16 * 2^18) with thresholds on and next to pair distances, thresholds
beyond every distance, equal points, and groups that touch, alone and together
in one batch.
"""
import numpy as np
import pytest

import oracle
from paper_1506_02226_gb300 import binding as B
from paper_1506_02226_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def instance(u, eps_units, min_pts):
    x = np.ascontiguousarray(np.clip(u, 0, 1023).astype(np.float32) / np.float32(1024))
    return inputs.Instance(x, float(np.float32(eps_units / 1024)), min_pts)


def blobs(rng, n, d, spread):
    c = rng.integers(spread, 1024 - spread, size=(5, d))
    u = c[rng.integers(0, 5, size=n)] + rng.integers(-spread, spread + 1, size=(n, d))
    loose = rng.random(n) < 0.1
    u[loose] = rng.integers(0, 1024, size=(int(loose.sum()), d))
    return u


def run(insts, mode=0):
    from paper_1506_02226_gb300.api import Plan, make_instances
    items = [(torch.from_numpy(i.points).cuda(), i.eps, i.min_pts,
              torch.full((i.n,), -9, dtype=torch.int32, device="cuda")) for i in insts]
    with Plan(max_n=16, max_d=16, label_mode=mode) as p:
        st = (B.dbscan_stats * len(insts))()
        assert B.dbscan_batch(p.handle, make_instances(items), st) == B.DBSCAN_OK
        with_stats = [it[3].cpu().numpy() for it in items]
        for it in items:
            it[3].fill_(-9)
        assert B.dbscan_batch(p.handle, make_instances(items)) == B.DBSCAN_OK
        for a, it in zip(with_stats, items):
            np.testing.assert_array_equal(a, it[3].cpu().numpy())
    return with_stats, st


def check(insts, mode=0):
    labs, st = run(insts, mode)
    for k, (inst, lab) in enumerate(zip(insts, labs)):
        want, _, core = oracle.dbscan(inst.points, inst.eps, inst.min_pts, label_mode=mode)
        np.testing.assert_array_equal(lab, want, err_msg=f"instance {k} n={inst.n} d={inst.d}")
        assert st[k].n_core == int(core.sum())


@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 8, 9, 16])
def test_sizes_around_tiles(d):
    rng = np.random.default_rng(700 + d)
    sizes = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 193, 1000, 2049]
    check([instance(blobs(rng, n, d, 12 + 4 * d), 14 * np.sqrt(d), 4) for n in sizes], mode=d & 1)


@pytest.mark.parametrize("d", [2, 16])
def test_largest_sorted_instance(d):
    rng = np.random.default_rng(d)
    check([instance(blobs(rng, n, d, 30), 11 * np.sqrt(d), 9) for n in (16384, 16385, 300)])


def test_extreme_units():
    rng = np.random.default_rng(77)
    insts = []
    for d in (9, 16):
        ends = rng.choice([0, 1, 511, 512, 1022, 1023], size=(700, d))
        ends[:40] = 0
        ends[40:80] = 1023
        D = np.unique(((ends[:, None, :] - ends[None, :50, :]) ** 2).sum(2))
        for v in (0, D[1], D[len(D) // 2], D[-2], D[-1]):
            for off in (-0.25, 0.25):  # just below and just above the distance
                insts.append(instance(ends, max(np.sqrt(max(v + off, 0.0)), 0.4), 5))
        insts.append(instance(ends, 1023 * np.sqrt(d) + 2, 3))  # beyond every distance: one cluster
        insts.append(instance(np.full((200, d), 1023), 0.5, 200))  # equal points
    check(insts)


def test_touching_groups_and_mixed_tiles():
    rng = np.random.default_rng(3)
    chain = 40 + rng.permutation(900)[:, None] + rng.integers(-2, 3, size=(900, 3))
    strips = np.concatenate([np.stack([rng.integers(0, 1024, 600), np.full(600, 100 + 9 * k)], 1) for k in range(6)])
    check([instance(chain, 9, 3), instance(strips, 8, 4), instance(strips, 9, 4), instance(strips, 40, 700)])
