"""The decoding work that is timed: what a user of this library has it do.

Every case is one call sequence through the public entry points, host buffers
in and tours out (the decoder's inputs and results live on the host: a
heatmap comes from a predictor's output file or process, a tour goes back to
the caller), preparation included:

    solve    one instance by the one-shot call with its defaults
    batch    a batch of instances in the persistent cluster kernel, the layout
             chosen by the library (symmetric or ATSP, with or without the
             restart schedule)
    step     a batch on the per-step kernels with the lookup lists (large
             instances; every kind of local search)
    serve    a request mix through the continuous-batching server, which the
             program keeps

The instances follow the recipe of the repository's synthetic workloads: points
(uniform, 8 Gaussian clusters or a perturbed grid) or an asymmetric cost
matrix, and a row-normalised kNN heatmap exp(-d/dbar) * LogNormal(0, 0.5).
"""
import numpy as np
import torch

from paper_2601_19041_gb300 import heataco, synth


# ------------------------------------------------------------------ cases

def listed():
    return [
        # an interactive decode of a small instance: launch and call overheads count
        dict(name="solve_n100", kind="solve", n=100, knn=50, m=32, k=20, iters=50, rho=0.8, family="uniform", fp16=False),
        # the single-instance workload of the benchmark (n=500, m=50, 100 iterations)
        dict(name="solve_n500", kind="solve", n=500, knn=50, m=50, k=20, iters=100, rho=0.2, family="uniform", fp16=False),
        # one larger instance alone, with an odd size and a binary16 heatmap
        dict(name="solve_n1999", kind="solve", n=1999, knn=50, m=32, k=20, iters=40, rho=0.8, family="gmm", fp16=True),
        # the benchmark's batched workload: 128 uneven instances in one call
        dict(name="batch128_n500_2000", kind="batch", count=128, n_lo=500, n_hi=2000, knn=50, m=64, k=20, iters=200,
             rho=0.2, schedule=0, family="uniform", fp16=False, atsp=False),
        # the benchmark's ATSP workload: cost matrices, directed heatmaps
        dict(name="atsp64_n1000", kind="batch", count=64, n_lo=1000, n_hi=1000, knn=50, m=50, k=20, iters=200, rho=0.2,
             schedule=0, family="uniform", fp16=False, atsp=True),
        # the paper's setting (m=32, rho=0.8, restarts), shortened to 600 of its 5000 iterations
        dict(name="paper128_n500", kind="batch", count=128, n_lo=500, n_hi=500, knn=50, m=32, k=20, iters=600, rho=0.8,
             schedule=1, family="uniform", fp16=False, atsp=False),
        # one mid-size instance decoded alone in the cluster kernel: its critical path
        dict(name="batch1_n1000_k32", kind="batch", count=1, n_lo=1000, n_hi=1000, knn=50, m=64, k=32, iters=100, rho=0.2,
             schedule=0, family="grid", fp16=False, atsp=False),
        # the paper's setting with 2-opt on every ant
        dict(name="step_2opt_every_ant_n500", kind="step", count=64, n=500, knn=50, m=32, k=20, iters=100, rho=0.8,
             schedule=1, local_search=2, ls_k=20, family="uniform", fp16=False),
        # 3-opt on the iteration-best tour
        dict(name="step_3opt_n500", kind="step", count=32, n=500, knn=10, m=32, k=10, iters=8, rho=0.2, schedule=0,
             local_search=3, ls_k=10, family="gmm", fp16=False),
        # large instances without local search: rows from L2, nearest-unvisited steps over 5000 nodes
        dict(name="step_n5000", kind="step", count=16, n=5000, knn=50, m=64, k=20, iters=20, rho=0.2, schedule=0,
             local_search=0, ls_k=20, family="uniform", fp16=True),
        # the large workload of the benchmark (n=10000, k=10, 2-opt on the iteration-best tour), shortened
        dict(name="step_2opt_n10000", kind="step", count=8, n=10000, knn=10, m=64, k=10, iters=15, rho=0.2, schedule=0,
             local_search=1, ls_k=20, family="uniform", fp16=False),
        # a burst of requests of mixed sizes through the server
        dict(name="serve_mix24", kind="serve", count=24, n_hi=5000, knn=50, m=64, k=20, it_lo=20, it_hi=60, rho=0.2),
    ]


def _log(rng, lo, hi):
    return int(round(float(lo) * (float(hi) / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["solve", "batch", "batch", "step", "serve"])
    family = rng.choice(["uniform", "gmm", "grid"])
    fp16 = rng.random() < 0.3
    k = rng.choice([8, 10, 16, 20, 20, 20, 27, 32])
    if kind == "solve":
        return dict(kind=kind, n=_log(rng, 60, 2000), knn=rng.choice([10, 50]), m=rng.randint(8, 64), k=k,
                    iters=_log(rng, 10, 100), rho=rng.choice([0.2, 0.8]), family=family, fp16=fp16)
    if kind == "batch":
        lo, hi = _log(rng, 100, 1000), _log(rng, 1000, 2000)
        return dict(kind=kind, count=_log(rng, 2, 128), n_lo=lo, n_hi=hi, knn=rng.choice([10, 50]), m=rng.choice([20, 32, 50, 64]),
                    k=min(k, 20), iters=_log(rng, 20, 150), rho=rng.choice([0.2, 0.8]), schedule=rng.choice([0, 1]),
                    family=family, fp16=fp16, atsp=rng.random() < 0.25 and hi <= 1400)
    if kind == "step":
        ls = rng.choice([0, 0, 1, 2, 3])
        n = _log(rng, 2000, 10000) if ls == 0 else _log(rng, 200, 5000) if ls == 1 else _log(rng, 100, 800 if ls == 2 else 500)
        return dict(kind=kind, count=_log(rng, 1, 16 if n > 1000 else 64), n=n, knn=rng.choice([10, 20]), m=rng.choice([32, 50, 64]),
                    k=min(k, 20), iters=_log(rng, 5, 20 if ls < 3 else 8), rho=rng.choice([0.2, 0.8]), schedule=rng.choice([0, 1]),
                    local_search=ls, ls_k=rng.choice([8, 10, 20]), family=family, fp16=fp16)
    return dict(kind=kind, count=_log(rng, 4, 24), n_hi=_log(rng, 1000, 5000), knn=rng.choice([20, 50]), m=rng.choice([32, 64]), k=min(k, 20),
                it_lo=10, it_hi=_log(rng, 20, 60), rho=0.2)


# ------------------------------------------------------------------ inputs

def _points(rng, n, family):
    return {"uniform": synth.uniform_points, "gmm": synth.gaussian_mixture_points,
            "grid": synth.perturbed_grid_points}[family](rng, n)


def _knn(rows_of, n, K):
    """K nearest of each row of an n x n distance matrix given in blocks of rows, on the GPU."""
    idx, dist = [], []
    for s in range(0, n, 2048):
        d = rows_of(s, min(n, s + 2048))
        d[torch.arange(d.shape[0], device="cuda"), torch.arange(s, s + d.shape[0], device="cuda")] = float("inf")
        v, i = torch.topk(d, K, dim=1, largest=False)
        idx.append(i.cpu().numpy())
        dist.append(v.cpu().numpy())
    return np.concatenate(idx), np.concatenate(dist)


def _euclid(seed, n, knn, family, fp16):
    rng = np.random.default_rng(seed)
    pts = _points(rng, n, family)
    p = torch.from_numpy(pts).cuda().double()

    def rows_of(s, e):
        dx, dy = p[s:e, 0:1] - p[None, :, 0], p[s:e, 1:2] - p[None, :, 1]
        return torch.sqrt(dx * dx + dy * dy)

    nbr, nd = _knn(rows_of, n, min(knn, n - 1))
    rowptr, col, val = synth.knn_heatmap(rng, nbr, nd, np.float16 if fp16 else np.float32)
    return synth.Instance(n=n, kind=0, coords=pts, cost=None, rowptr=rowptr, col=col, val=val, symmetrize=1, seed=seed)


def _atsp(seed, n, knn):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.from_numpy(rng.random((n, 2))).cuda()
    dx, dy = p[:, 0:1] - p[None, :, 0], p[:, 1:2] - p[None, :, 1]
    c = torch.sqrt(dx * dx + dy * dy) + 0.5 * torch.rand((n, n), generator=gen, device="cuda", dtype=torch.float64)
    c.fill_diagonal_(0.0)
    c = c.float()
    nbr, nd = _knn(lambda s, e: c[s:e].double(), n, min(knn, n - 1))
    rowptr, col, val = synth.knn_heatmap(rng, nbr, nd, np.float32)
    return synth.Instance(n=n, kind=1, coords=None, cost=c.cpu().numpy(), rowptr=rowptr, col=col, val=val, symmetrize=0, seed=seed)


def _instances(case, seed):
    """The case's instances and parameters, from the seed alone."""
    kind, ins, ps = case["kind"], [], []
    count = case.get("count", 1)
    rng = np.random.default_rng([count, case.get("n_hi", 0)])   # sizes and budgets belong to the case, not to the seed
    if kind == "batch":
        sizes = rng.integers(case["n_lo"], case["n_hi"] + 1, size=count)
    elif kind == "serve":
        sizes = [s for s in (500, 1000, 2000, 5000) if s < case["n_hi"]] + [case["n_hi"]]
        sizes = [sizes[q % len(sizes)] for q in range(count)]
    else:
        sizes = [case["n"]] * count
    fams = ("uniform", "gmm", "grid")
    for q in range(count):
        n, s = int(sizes[q]), 1000 * (seed % 1000003) + q
        if case.get("atsp"):
            ins.append(_atsp(s, n, case["knn"]))
        else:
            ins.append(_euclid(s, n, case["knn"], case.get("family", fams[q % 3]), case.get("fp16", True)))
        iters = int(rng.integers(case["it_lo"], case["it_hi"] + 1)) if kind == "serve" else case["iters"]
        ps.append(synth.Params(m=case["m"], k=case["k"], iterations=iters, rho=case["rho"], seed=s,
                               degree_target=1 if case.get("atsp") else 2, schedule=case.get("schedule", 0),
                               local_search=case.get("local_search", 0), ls_k=case.get("ls_k", 20)))
    return ins, ps


def prepare(case, seed):
    ins, ps = _instances(case, seed)
    state = dict(kind=case["kind"], ins=ins, ps=ps)
    if case["kind"] == "batch":
        state["exec"] = heataco.make_exec(fused=1, fallback_list=32)
    elif case["kind"] == "step":
        state["exec"] = heataco.make_exec(fallback_list=32, parts=min(4, len(ins)))
    elif case["kind"] == "serve":
        need = sum(heataco.hac_server_request_bytes(i, p) for i, p in zip(ins, ps))
        state["server"] = heataco.Server(need + (64 << 20), max_slots=64, iters_per_tick=10, max_n=10000,
                                         steps_per_tick=4000, step_min_n=3000,
                                         exec_=heataco.make_exec(fused=1, fallback_list=32))
    return state


# ------------------------------------------------------------------ the calls

def run(state):
    ins, ps = state["ins"], state["ps"]
    if state["kind"] == "solve":
        tour, length, stats = heataco.hac_solve(ins[0], ps[0])
        return {"tour": tour, "length": length, "ant_steps": stats["ant_steps"], "fallback_steps": stats["fallback_steps"],
                "restarts": stats["restarts"], "kappa": stats["kappa"], "edges_per_n": stats["edges_per_n"],
                "L_nn": stats["L_nn"]}
    if state["kind"] == "serve":
        return _serve(state["server"], ins, ps)
    tours, lens = heataco.solve_batch(ins, ps, state["exec"])
    return {"tours": np.concatenate(tours), "lengths": lens}


def _serve(server, ins, ps):
    """All requests are there at once; each is submitted as soon as the server takes it."""
    tickets, waiting, done = {}, list(range(len(ins))), {}
    while waiting or tickets:
        while waiting:
            t = server.submit(ins[waiting[0]], ps[waiting[0]])
            if t is None:
                break
            tickets[t] = waiting.pop(0)
        server.tick()
        for t in list(tickets):
            r = server.poll(t)
            if r is not None:
                done[tickets.pop(t)] = r
    return {"tours": np.concatenate([done[q][0] for q in range(len(ins))]),
            "lengths": np.array([done[q][1] for q in range(len(ins))])}


# ------------------------------------------------------------------ its size

def work(case):
    """Inputs read and tours written once; per ant-step the weighing of k candidates (mask, sum, compare)
    and per iteration the evaporation of n*k pheromone values."""
    count = case.get("count", 1)
    if case["kind"] == "batch":
        n = (case["n_lo"] + case["n_hi"]) / 2
    elif case["kind"] == "serve":
        sizes = [s for s in (500, 1000, 2000, 5000) if s < case["n_hi"]] + [case["n_hi"]]
        n = sum(sizes) / len(sizes)
    else:
        n = case["n"]
    iters = (case["it_lo"] + case["it_hi"]) / 2 if case["kind"] == "serve" else case["iters"]
    nnz = n * min(case["knn"], n - 1)
    fp16 = case.get("fp16", True)
    geometry = 4 * n * n if case.get("atsp") else 8 * n
    return {"bytes": int(count * (geometry + 4 * (n + 1) + nnz * (6 if fp16 else 8) + 4 * n + 8)),
            "flops": int(count * iters * n * case["k"] * (3 * case["m"] + 3))}


# ------------------------------------------------------------------ exact values

def exact(case, seed):
    """The scalars of the preparation in 64 bits; a tour found by the random search has no such value."""
    if case["kind"] != "solve":
        return None
    ins, ps = _instances(case, seed)
    I, p = ins[0], ps[0]
    n, K = I.n, min(p.k, I.n - 1)
    H = np.zeros((n, n))
    rows = np.repeat(np.arange(n), np.diff(I.rowptr))
    H[rows, I.col] = I.val.astype(np.float64)
    H = (H + H.T) / 2
    member = H > p.theta_h
    x = I.coords.astype(np.float64)
    lam = []
    for i in range(n):
        js = np.flatnonzero(member[i])
        d = np.hypot(x[js, 0] - x[i, 0], x[js, 1] - x[i, 1])
        c = H[i, js[np.lexsort((js, d))[:K]]]
        s = np.sort(c)[::-1]
        b = max(p.eps, s[p.degree_target] if len(s) > p.degree_target else 0.0)
        e = np.maximum(c, p.eps) / b
        lam.append(np.log(e[e > 1.0]))
    lam = np.concatenate(lam)
    q = float(np.quantile(lam[lam > 0], p.q_level)) if len(lam) else 0.0
    px = p.p_best ** (1.0 / n)
    R = (K - 1) / 2 * px / (1 - px)
    kappa = p.c_cap * p.alpha * np.log(R) / q if q > 0 and R > 1 else 0.0
    # the initial tour takes the unvisited node of the smallest squared distance in 32 bits (the library's definition)
    f, cur, left, L = I.coords, 0, np.ones(n, bool), 0.0
    left[0] = False
    for _ in range(n - 1):
        dx, dy = f[:, 0] - f[cur, 0], f[:, 1] - f[cur, 1]
        nxt = int(np.argmin(np.where(left, dx * dx + dy * dy, np.float32(np.inf))))
        L += float(np.hypot(x[nxt, 0] - x[cur, 0], x[nxt, 1] - x[cur, 1]))
        left[nxt], cur = False, nxt
    L += float(np.hypot(x[0, 0] - x[cur, 0], x[0, 1] - x[cur, 1]))
    return {"tour": None, "length": None, "ant_steps": None, "fallback_steps": None, "restarts": None,
            "kappa": float(kappa), "edges_per_n": float(member.sum()) / (2 * n), "L_nn": L}
