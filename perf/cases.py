"""What a user of the library has it do, as cases that can be timed one by one.

Every case goes through the public entry points (``Colony``, ``Batch``,
``Server``, ``faco_lists_noalloc``).  Instances are the seeded synthetic ones
of ``paper_2203_02228_gb300.inputs``: uniform squares and the stippled stand-in
of the large-instance study.  Sizes are those of the repository's own
workloads (1,000, 100,000 and 200,000 nodes, the 512-instance batch, the
served stream), smaller ones that are bound by launches and latency, and odd
ones.  Results of the method are tours, lengths and pheromone; they follow
from the instance and the seed alone, whatever ran before.
"""
import math

import numpy as np
import torch

from paper_2203_02228_gb300 import Batch, Colony, Server, inputs, load

BACKUP = 64          # backup list length of the default parameters
NEW_EDGES = 8        # and their least number of new edges per ant


def listed():
    return [
        # candidate lists for a caller that owns the device's memory: one small
        # instance (the smallest call: launches and one synchronisation), and
        # one of the size of the large-instance study
        dict(name="lists_2k", kind="lists", points="uniform", n=2_000, k=16),
        dict(name="lists_100k", kind="lists", points="stippled", n=100_003, k=16),
        # set-up of a colony (lists, nearest-neighbour tour, its local search):
        # what every solve and every request pays before its first iteration
        dict(name="setup_5k", kind="setup", points="uniform", n=5_003, k=16, three_opt=False, device=False),
        dict(name="setup_100k", kind="setup", points="stippled", n=100_000, k=16, three_opt=False, device=True),
        # the 1,000-node workload in full: set-up, 200 iterations of 32 ants
        dict(name="solve_1k", kind="solve", points="uniform", n=1_000, k=16, ants=32, iters=200),
        # iterations of a colony in its steady state: a served request's size,
        # the two large workloads at their own ant counts, wide candidate lists
        # on an odd size, and the walk without the per-ant search
        dict(name="iterate_20k", kind="iterate", points="uniform", n=20_011, k=16, ants=256, iters=8, ls=True, warm=16),
        dict(name="iterate_100k", kind="iterate", points="stippled", n=100_000, k=16, ants=1024, iters=6, ls=True,
             warm=16),
        dict(name="iterate_200k", kind="iterate", points="stippled", n=200_000, k=16, ants=2048, iters=4, ls=True,
             warm=8),
        dict(name="iterate_30k_k32", kind="iterate", points="uniform", n=30_011, k=32, ants=256, iters=8, ls=True,
             warm=16),
        dict(name="iterate_50k_nols", kind="iterate", points="stippled", n=50_000, k=16, ants=512, iters=8, ls=False,
             warm=16),
        # many uneven instances through the same launches, from host
        # coordinates to host tours
        dict(name="batch_64", kind="batch", count=64, lo=200, hi=20_000, sizes=4000, k=16, ants=64, iters=10),
        # a burst of requests to a running server, until the last is answered
        dict(name="serve_6", kind="serve", count=6, lo=1_000, hi=30_000, sizes=5000, k=16, ants=256, iters=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lists", "setup", "solve", "iterate", "iterate", "batch", "serve"])
    points = rng.choice(["uniform", "stippled"])
    k = rng.choice([8, 12, 16, 16, 16, 24, 32])
    if kind == "lists":
        return dict(kind=kind, points=points, n=_log_int(rng, 500, 110_000), k=k)
    if kind == "setup":
        return dict(kind=kind, points=points, n=_log_int(rng, 500, 90_000), k=k, three_opt=rng.random() < 0.2,
                    device=rng.random() < 0.5)
    if kind == "solve":
        return dict(kind=kind, points=points, n=_log_int(rng, 200, 5_000), k=k, ants=_log_int(rng, 8, 128),
                    iters=rng.randint(10, 100))
    if kind == "iterate":
        n = _log_int(rng, 2_000, 180_000)
        return dict(kind=kind, points=points, n=n, k=k, ants=_log_int(rng, 32, 1_536), iters=rng.randint(1, 4),
                    ls=rng.random() < 0.8, warm=8)
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 4, 64), lo=200, hi=_log_int(rng, 1_000, 20_000),
                    sizes=rng.randint(1, 9_999), k=k, ants=_log_int(rng, 16, 64), iters=rng.randint(2, 10))
    return dict(kind=kind, count=rng.randint(1, 6), lo=1_000, hi=_log_int(rng, 2_000, 30_000),
                sizes=rng.randint(1, 9_999), k=k, ants=_log_int(rng, 32, 256), iters=rng.randint(5, 20))


def _points(case, seed):
    n = case["n"]
    if case["points"] == "uniform":
        return inputs.uniform(n, seed=seed)
    if n >= 150_000:  # the densities of the 200,000- and the 100,000-node workload
        return inputs.stippled(n, seed=seed, blobs=256, ridges=16)
    return inputs.stippled(n, seed=seed)


def prepare(case, seed):
    kind, k = case["kind"], case["k"]
    s = dict(case)
    if kind == "lists":
        n = case["n"]
        s["xy"] = torch.from_numpy(_points(case, seed)).cuda()
        s["cand"] = torch.empty((n, k), dtype=torch.int32, device="cuda")
        s["backup"] = torch.empty((n, BACKUP), dtype=torch.int32, device="cuda")
        s["eta"] = torch.empty((n, k), dtype=torch.float32, device="cuda")
    elif kind == "setup":
        xy = _points(case, seed)
        s["xy"] = torch.from_numpy(xy).cuda() if case["device"] else xy
    elif kind == "solve":
        s["xy"] = _points(case, seed)
    elif kind == "iterate":
        # a colony some iterations into its run; without the per-ant search
        # the study keeps rho = 0.9
        more = {} if case["ls"] else dict(local_search=0, rho=0.9)
        s["colony"] = Colony(_points(case, seed), k, seed=seed, **more)
        s["colony"].iterate(case["ants"], case["warm"])
        s["colony"].sync()
    else:  # batch, serve: instances of uneven sizes, log-uniform (the case's), of points of their own (the seed's)
        ns = inputs.batch_sizes(case["count"], case["sizes"], case["lo"], case["hi"])
        s["xs"] = [inputs.uniform(int(n), seed=seed * 1000 + i) for i, n in enumerate(ns)]
        s["seeds"] = [seed + i for i in range(case["count"])]
        if kind == "serve":
            s["server"] = Server(2 << 30)
    return s


def run(s):
    kind, k = s["kind"], s["k"]
    if kind == "lists":
        rc = load().faco_lists_noalloc(s["xy"].data_ptr(), s["n"], k, BACKUP, s["cand"].data_ptr(),
                                       s["backup"].data_ptr(), s["eta"].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise RuntimeError("faco_lists_noalloc: %d" % rc)
        return {"cand": s["cand"], "backup": s["backup"], "eta": s["eta"]}
    if kind == "setup":
        with Colony(s["xy"], k, device=s["device"], init_3opt=int(s["three_opt"])) as col:
            tour, length = col.initial()
            return {"tour": tour, "length": length, "limits": col.limits()}
    if kind == "solve":
        with Colony(s["xy"], k, seed=1) as col:
            col.iterate(s["ants"], s["iters"])
            tour, length = col.best()
            return {"tour": tour, "length": length, "tau": col.tau()}
    if kind == "iterate":
        col = s["colony"]
        col.iterate(s["ants"], s["iters"])
        tour, length = col.best()
        return {"tour": tour, "length": length, "tau": col.tau()}
    if kind == "batch":
        with Batch(s["xs"], k, seeds=s["seeds"]) as b:
            b.iterate(s["ants"], s["iters"])
            tours, lengths = b.tours()
            return {"tours": np.concatenate(tours), "lengths": lengths}
    server = s["server"]
    tickets = [server.submit(x, k, s["ants"], s["iters"], seed) for x, seed in zip(s["xs"], s["seeds"])]
    done = [server.wait(t) for t in tickets]
    for t in tickets:
        server.release(t)
    return {"tours": np.concatenate([d[0] for d in done]), "lengths": np.array([d[1] for d in done])}


def _list_work(n, k):
    # coordinates in; candidates, backups and 1/d out; a distance per entry
    return 8 * n + 4 * n * (2 * k + BACKUP), 5 * n * (k + BACKUP)


def _setup_work(n, k):
    # beside the lists: pheromone, the tour, and every node's 2-opt and Or-opt
    # scan once (both neighbours of k candidates, eight distances each)
    b, f = _list_work(n, k)
    return b + 4 * n * k + 4 * n, f + n * 2 * k * 8 * 5


def _iter_work(n, k, ants, ls):
    # the update of Eq. 2 (pheromone both ways, candidates, 1/d), the best
    # tour, and per ant the roulette rows of its new edges and, with the
    # search, the scan of each of their heads
    b = 16 * n * k + 4 * n + ants * NEW_EDGES * 8 * k
    f = 3 * n * k + ants * NEW_EDGES * 4 * k
    if ls:
        b += ants * NEW_EDGES * 2 * k * 20
        f += ants * NEW_EDGES * 2 * k * 8 * 5
    return b, f


def work(case):
    kind, k = case["kind"], case["k"]
    if kind == "lists":
        b, f = _list_work(case["n"], k)
    elif kind == "setup":
        b, f = _setup_work(case["n"], k)
    elif kind == "iterate":
        b, f = (case["iters"] * v for v in _iter_work(case["n"], k, case["ants"], case["ls"]))
    else:
        count = case.get("count", 1)
        if kind == "solve":
            n = case["n"]
        else:  # the mean of the log-uniform sizes
            lo, hi = case["lo"], case["hi"]
            n = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        b, f = (count * (u + case["iters"] * v)
                for u, v in zip(_setup_work(n, k), _iter_work(n, k, case["ants"], True)))
    return {"bytes": int(b), "flops": int(f)}


def exact(case, seed):
    """The lists by full distance rows in 64-bit integers and 1/d in 64-bit
    floats.  A search's outcome has no value but the sequential one."""
    if case["kind"] != "lists":
        return None
    n, k = case["n"], case["k"]
    xy = torch.from_numpy(_points(case, seed)).cuda().to(torch.int64)
    ids = torch.arange(n, device="cuda")
    rows = max(1, (1 << 27) // n)
    near, dist = [], []
    for at in range(0, n, rows):
        p = xy[at:at + rows]
        m = (p[:, None, 0] - xy[None, :, 0]) ** 2 + (p[:, None, 1] - xy[None, :, 1]) ** 2
        key = m * (1 << 18) + ids  # (squared distance, node id)
        key[torch.arange(p.shape[0], device="cuda"), ids[at:at + rows]] = torch.iinfo(torch.int64).max
        key = torch.topk(key, k + BACKUP, dim=1, largest=False, sorted=True).values
        near.append(key % (1 << 18))
        dist.append(torch.floor(torch.sqrt((key[:, :k] // (1 << 18)).double()) + 0.5))
    near, dist = torch.cat(near), torch.cat(dist)
    return {"cand": near[:, :k], "backup": near[:, k:], "eta": torch.where(dist > 0, 1.0 / dist, 1.0)}
