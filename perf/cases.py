"""The calls that users of this library make, as measurable cases.

A case names a point recipe, its sizes and the entry point that clusters it:
``Plan.run`` (device tensors), ``Plan.run_host`` (host tensors, copies
included), ``Plan.run_detail`` (exact counts and core flags beside the labels),
``dbscan_batch`` (many small instances at once) and a ``dbscan_serve_*`` server
fed a burst of jobs.  Points are drawn on the GPU from a seed and lie on the
2^-10 grid that the library takes.

Recipes (the seeded generators of ``paper_1506_02226_gb300.inputs``, drawn with
torch): ``field`` is 50 blobs of very different widths plus 20% noise (5 blobs
and 10% for the smallest), ``groups`` is about 2,000 points per blob of equal
width plus 15% noise with some tens of neighbours a point, ``mixture`` is the
served and batched jobs' 1 to 8 blobs plus 10% noise.
"""
import math

import numpy as np
import torch

from paper_1506_02226_gb300 import binding as B
from paper_1506_02226_gb300.api import Plan, make_instances

UNIT = 1024  # grid units per coordinate


# ---- cases ------------------------------------------------------------------

def _run(name, recipe, n, d, eps, min_pts, **more):
    case = {"name": name, "kind": "run", "recipe": recipe, "n": n, "d": d, "eps": eps, "min_pts": min_pts,
            "call": "run", "precision": B.DBSCAN_PREC_AUTO, "compact": False, "sync": True}
    case.update(more)
    return case


def listed():
    return [
        # An interactive call on a small 2-D set: launches and the wait decide.
        _run("small_2d", "field", 2000, 2, 0.02, 5, blobs=5, noise=0.1, sigma_lo=0.03, sigma_hi=0.03),
        # The paper's largest 3-D size, from and to host memory, with dense cluster numbers.
        _run("host_3d_60k", "field", 60032, 3, 0.0144, 10, call="host", compact=True),
        # Large spatial data: half a million points in the plane, one blocking call.
        _run("plane_500k", "field", 500000, 2, 0.005, 10),
        # The same in space, enqueued without waiting, as a pipeline of frames does.
        _run("space_500k", "field", 500000, 3, 0.005, 10, sync=False),
        # Exact neighbour counts and core flags beside the labels, a ragged size.
        _run("detail_5d_50k", "field", 50001, 5, 0.0079, 10, call="detail"),
        # Feature vectors of middling dimension.
        _run("features_8d_200k", "field", 200000, 8, 0.01, 10),
        # Between the grids (d <= 8) and the tensor cores (d >= 16): CUDA-core pair tests.
        _run("pairs_12d_30k", "groups", 30011, 12, 0.1975, 20),
        # Embeddings, a small ragged set: few tiles for the tensor cores.
        _run("embed_32d_6k", "groups", 6007, 32, 0.3229, 12),
        # Embeddings at size, in FP16 (the default).
        _run("embed_64d_200k", "groups", 200000, 64, 0.45665, 20),
        # Embeddings in the BF16 form, a ragged size and dimension.
        _run("embed_bf16_48d_100k", "groups", 100003, 48, 0.39547, 20, precision=B.DBSCAN_PREC_BF16_GRAM),
        # Thousands of uneven instances at once.
        {"name": "batch_4096", "kind": "batch", "count": 4096, "n_lo": 64, "n_hi": 8192, "dims": "2,3,16", "mix": 4,
         "compact": False},
        # A burst of uneven jobs to the server.
        {"name": "serve_40", "kind": "serve", "count": 40, "n_lo": 1000, "n_hi": 500000, "dims": "2,3,32", "mix": 5,
         "slots": 8},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    case = _draw(rng)
    case.pop("name", None)
    return case


def _draw(rng):
    kind = rng.choice(["low", "low", "mid", "pairs", "embed", "embed", "job", "batch", "serve"])
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 4, 2048), "n_lo": 64, "n_hi": _log_int(rng, 512, 8192),
                "dims": rng.choice(["2,3,16", "2,3", "3,8,12", "2"]), "mix": rng.randrange(1 << 20),
                "compact": rng.random() < 0.3}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(4, 24), "n_lo": 1000, "n_hi": _log_int(rng, 10000, 250000),
                "dims": rng.choice(["2,3,32", "2,3", "3,8,24"]), "mix": rng.randrange(1 << 20), "slots": 8}
    more = {"call": rng.choice(["run", "run", "run", "detail", "host"]), "compact": rng.random() < 0.3,
            "sync": rng.random() < 0.7}
    if kind == "low":
        d, n = rng.randint(2, 3), _log_int(rng, 1000, 500000)
        eps = min(0.02, 0.005 * math.sqrt(500000 / n))
        return _run("", "field", n, d, eps, rng.randint(4, 16), blobs=max(5, min(50, n // 1000)), **more)
    if kind == "mid":
        d, n = rng.randint(4, 8), _log_int(rng, 1000, 200000)
        return _run("", "field", n, d, 0.005 * math.sqrt(d / 2), rng.randint(4, 16),
                    blobs=max(5, min(50, n // 1000)), **more)
    if kind == "pairs":
        d, n = rng.randint(9, 15), _log_int(rng, 1000, 40000)
        return _run("", "groups", n, d, 0.45665 * math.sqrt(d / 64), rng.randint(8, 24), **more)
    if kind == "embed":
        d, n = rng.randint(16, 64), _log_int(rng, 4096, 120000)
        more["precision"] = rng.choice([B.DBSCAN_PREC_AUTO, B.DBSCAN_PREC_AUTO, B.DBSCAN_PREC_BF16_GRAM])
        return _run("", "groups", n, d, 0.45665 * math.sqrt(d / 64), rng.randint(8, 24), **more)
    n, d = _log_int(rng, 1000, 150000), rng.choice([2, 3, 16, 32])
    return _run("", "mixture", n, d, rng.uniform(0.01, 0.05), rng.randint(4, 16), blobs=rng.randint(1, 8),
                mix=rng.randrange(1 << 20), **more)


def _jobs(case):
    """Sizes and parameters of a batch's or a server's jobs (fixed by the case): n, d, eps, min_pts, sigmas."""
    rng = np.random.default_rng(case["mix"])
    dims = [int(t) for t in case["dims"].split(",")]
    jobs = []
    for _ in range(case["count"]):
        n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"] + 1))))
        d = int(rng.choice(dims))
        jobs.append((n, d, float(np.float32(rng.uniform(0.01, 0.05))), int(rng.integers(4, 17)),
                     _mixture_sigmas(rng, int(rng.integers(1, 9)), d)))
    return jobs


def _mixture_sigmas(rng, blobs, d):
    return [float(s) for s in np.exp(rng.uniform(math.log(0.005), math.log(0.03), size=blobs)) * math.sqrt(2 / d)]


def _sigmas(case):
    if case["recipe"] == "field":
        lo, hi, k = case.get("sigma_lo", 0.002), case.get("sigma_hi", 0.02), case.get("blobs", 50)
        return [lo * (hi / lo) ** ((b + 0.5) / k) for b in range(k)], case.get("noise", 0.2)
    if case["recipe"] == "groups":
        return [0.05] * max(2, round(case["n"] / 2000)), 0.15
    return _mixture_sigmas(np.random.default_rng(case["mix"]), case["blobs"], case["d"]), 0.1


# ---- inputs -----------------------------------------------------------------

def _points(gen, sizes, d, sigmas, noise):
    """Points of several sets of one dimension, one after the other: float32 [sum(sizes), d] on the grid.
    Set i has a blob of each width of sigmas[i] at a uniform centre, and uniform noise."""
    dev = gen.device
    reps = torch.tensor(sizes, device=dev)
    n = int(sum(sizes))
    first = torch.tensor(np.cumsum([0] + [len(s) for s in sigmas])[:-1], device=dev)
    blobs = torch.tensor([len(s) for s in sigmas], device=dev)
    width = torch.tensor([w for s in sigmas for w in s], dtype=torch.float32, device=dev)
    centre = torch.rand((width.numel(), d), generator=gen, device=dev)
    k = torch.repeat_interleave(blobs, reps, output_size=n)
    pick = (torch.rand(n, generator=gen, device=dev) * k).long().clamp_(max=k - 1)
    pick += torch.repeat_interleave(first, reps, output_size=n)
    x = centre[pick] + width[pick, None] * torch.randn((n, d), generator=gen, device=dev)
    bad = ((x < 0) | (x >= 1)).nonzero(as_tuple=True)
    while bad[0].numel():  # coordinates outside [0, 1) are drawn again
        b = pick[bad[0]]
        v = centre[b, bad[1]] + width[b] * torch.randn(b.numel(), generator=gen, device=dev)
        x[bad] = v
        out = (v < 0) | (v >= 1)
        bad = (bad[0][out], bad[1][out])
    loose = torch.rand(n, generator=gen, device=dev) < noise
    x = torch.where(loose[:, None], torch.rand((n, d), generator=gen, device=dev), x)
    return x.mul_(UNIT).floor_().clamp_(0, UNIT - 1).div_(UNIT).contiguous()


def _sets(gen, jobs, noise):
    """One point tensor per job (the jobs of one dimension share an allocation)."""
    out = [None] * len(jobs)
    for d in sorted({j[1] for j in jobs}):
        at = [i for i, j in enumerate(jobs) if j[1] == d]
        x = _points(gen, [jobs[i][0] for i in at], d, [jobs[i][4] for i in at], noise)
        for i, part in zip(at, torch.split(x, [jobs[i][0] for i in at])):
            out[i] = part
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


class _Server:
    """A running server and the jobs in hand; destroyed with the state that holds it."""

    def __init__(self, case, jobs, points, labels):
        o = B.dbscan_serve_opts_default()
        o.slots = case["slots"]
        o.max_n = max(j[0] for j in jobs)
        self.handle = B.dbscan_serve_create(o)
        self.points, self.labels = points, labels
        self.jobs = make_instances([(x, j[2], j[3], lab) for j, x, lab in zip(jobs, points, labels)])

    def __del__(self):
        if getattr(self, "handle", 0):
            B.dbscan_serve_destroy(self.handle)
            self.handle = 0


def prepare(case, seed):
    gen = _generator(seed)
    if case["kind"] == "run":
        sigmas, noise = _sigmas(case)
        x = _points(gen, [case["n"]], case["d"], [sigmas], noise)
        plan = Plan(max_n=case["n"], max_d=case["d"], precision=case["precision"],
                    label_mode=B.DBSCAN_LABEL_COMPACT if case["compact"] else B.DBSCAN_LABEL_ROOT_INDEX,
                    synchronous=case["sync"])
        if case["call"] == "host":
            x = x.cpu().pin_memory()
        return {"case": case, "plan": plan, "points": x}
    jobs = _jobs(case)
    points = _sets(gen, jobs, 0.1)
    total = sum(j[0] for j in jobs)
    flat = torch.empty(total, dtype=torch.int32, device="cuda")
    labels = torch.split(flat, [j[0] for j in jobs])
    if case["kind"] == "serve":
        torch.cuda.synchronize()  # the server's streams do not wait for the one that drew the points
        return {"case": case, "server": _Server(case, jobs, points, labels), "labels": flat}
    plan = Plan(max_n=1, max_d=16, label_mode=B.DBSCAN_LABEL_COMPACT if case["compact"] else B.DBSCAN_LABEL_ROOT_INDEX)
    items = make_instances([(x, j[2], j[3], lab) for j, x, lab in zip(jobs, points, labels)])
    return {"case": case, "plan": plan, "points": points, "items": items, "labels": flat}


# ---- one pass ---------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        srv = state["server"]
        ids = [B.dbscan_serve_submit(srv.handle, job) for job in srv.jobs]
        for i in ids:
            status, _ = B.dbscan_serve_wait(srv.handle, i)
            if status != B.DBSCAN_OK:
                raise B.DbscanError(status, "dbscan_serve_wait")
        return state["labels"]
    if case["kind"] == "batch":
        status = B.dbscan_batch(state["plan"].handle, state["items"])
        if status != B.DBSCAN_OK:
            raise B.DbscanError(status, "dbscan_batch")
        return state["labels"]
    plan, x = state["plan"], state["points"]
    if case["call"] == "host":
        return plan.run_host(x, case["eps"], case["min_pts"])
    if case["call"] == "detail":
        return plan.run_detail(x, case["eps"], case["min_pts"])[:3]
    return plan.run(x, case["eps"], case["min_pts"])


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Bytes: every coordinate read once, every output written once.  Flops: min_pts neighbours of
    every point shown to be near (a multiply and an add per coordinate of each pair)."""
    if case["kind"] == "run":
        jobs = [(case["n"], case["d"], case["eps"], case["min_pts"])]
    else:
        jobs = _jobs(case)
    per_point = 9 if case.get("call") == "detail" else 4  # labels (counts, core flags)
    return {"bytes": sum(4 * j[0] * j[1] + per_point * j[0] for j in jobs),
            "flops": sum(2 * j[0] * j[1] * j[3] for j in jobs)}


# ---- the same by brute force in 64 bits --------------------------------------

_EXACT_MAX_N = 65536  # more points than this take too long


def _brute(x, eps, min_pts, compact):
    """(labels, counts, core flags) of the definitions: float64 squared distances of grid units (exact)."""
    n = x.shape[0]
    u = x.double() * UNIT
    sq = (u * u).sum(1)
    limit = math.floor(float(np.float32(eps)) ** 2 * 2 ** 20)
    step = max(1, (1 << 26) // n)

    def near(a, cols):
        return (sq[a:a + step, None] + sq[cols][None, :] - 2.0 * (u[a:a + step] @ u[cols].T)) <= limit

    everyone = torch.arange(n, device=u.device)
    count = torch.cat([near(a, everyone).sum(1) for a in range(0, n, step)])
    core = count >= min_pts
    cores = core.nonzero().squeeze(1)
    big = n  # no label
    label = torch.where(core, everyone, torch.full_like(everyone, big))
    link = torch.cat([everyone, everyone.new_tensor([big])])
    if cores.numel():
        while True:  # hook every component on its smallest neighbour, then flatten
            least = torch.cat([torch.where(near(a, cores), label[cores][None, :], big).amin(1)
                               for a in range(0, n, step)])
            best = torch.minimum(label, torch.where(core, least, torch.full_like(least, big)))
            if torch.equal(best, label):
                break
            link.scatter_reduce_(0, label[cores], best[cores], "amin")
            while True:
                further = link[link]
                if torch.equal(further, link):
                    break
                link = further
            label = torch.where(core, link[label], label)
        owner = torch.cat([torch.where(near(a, cores), cores[None, :], big).amin(1) for a in range(0, n, step)])
        label = torch.where(core, label, torch.cat([label, label.new_tensor([big])])[owner])
    noise = label == big
    if compact:
        roots = torch.zeros(n + 1, dtype=torch.long, device=u.device)
        roots[label] = 1
        roots[big] = 0
        label = (torch.cumsum(roots, 0) - roots)[label]
    label = torch.where(noise, torch.full_like(label, -1), label)
    return label.int(), count.int(), core.to(torch.uint8)


def exact(case, seed):
    if case["kind"] == "run":
        if case["n"] > _EXACT_MAX_N:
            return None
        sigmas, noise = _sigmas(case)
        x = _points(_generator(seed), [case["n"]], case["d"], [sigmas], noise)
        label, count, core = _brute(x, case["eps"], case["min_pts"], case["compact"])
        if case["call"] == "detail":
            return label, count, core
        return label.cpu() if case["call"] == "host" else label
    jobs = _jobs(case)
    if len(jobs) > 256 or max(j[0] for j in jobs) > _EXACT_MAX_N:
        return None
    points = _sets(_generator(seed), jobs, 0.1)
    return torch.cat([_brute(x, j[2], j[3], case.get("compact", False))[0] for j, x in zip(jobs, points)])
