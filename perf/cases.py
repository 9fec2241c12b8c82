"""The work a user of the library has it do, as measurable cases.

Every case goes through the public binding (``paper_1610_10061_gb300.pm``).
The instance families and sizes are those of the repository's inputs,
configurations and benchmark: graph instances (all-pairs shortest paths of a
connected random graph), uniform Euclidean points and clustered points, from
100 to 10000 clients and facilities.  Inputs are made on the GPU from the seed
alone, with the recipes of ``paper_1610_10061_gb300.inputs`` restated in torch.

A case's ``kind`` says which part of the library it drives:

* ``eval``    one fitness evaluation of a population of random p-subsets.
* ``tables``  the instance build (ordering and increment tables), read back.
* ``job``     distances in host memory -> instance -> GA -> result.
* ``ga``      a plain GA on an instance that exists already.
* ``batch``   a GA over many uneven instances at once (``gens`` > 0), or one
              batched evaluation (``gens`` = 0).
* ``learned`` a GA with the learned swap proposal.
* ``stats``   the swap statistics that the learned proposal reads.
* ``forward`` the perceptron's predictions for candidate moves.
* ``train``   one epoch of training of the perceptron.
"""

import math
import random

import numpy as np
import torch

from paper_1610_10061_gb300 import pm

DEV = "cuda"


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------

def _eval(name, family, n, m, p, pop, cumulative=False, host=False):
    return {"name": name, "kind": "eval", "family": family, "n": n, "m": m, "p": p, "pop": pop,
            "cumulative": cumulative, "host": host}


def listed():
    return [
        # one evaluation of the 100-node graph's population: a small call, where launches count
        _eval("eval_graph100", "graph", 100, 100, 5, 64),
        # one evaluation of the 900-node graph's GA population: the ordinary call
        _eval("eval_graph900", "graph", 900, 900, 90, 1024),
        # the fitness passes of the 10000-point Euclidean instance, few to many open facilities: the largest calls
        _eval("eval_euclid10000_p10", "euclid", 10000, 10000, 10, 4096),
        _eval("eval_euclid10000_p100", "euclid", 10000, 10000, 100, 4096),
        _eval("eval_euclid10000_p1000", "euclid", 10000, 10000, 1000, 4096),
        # odd sizes, more clients than facilities, cumulative tables, population in host memory
        _eval("eval_ragged_cumulative", "euclid", 3001, 2011, 37, 777, cumulative=True, host=True),
        # instance build of the clustered 5000-point instance: sort, truncation, increments, tables read back
        {"name": "tables_gmm5000", "kind": "tables", "family": "gmm", "n": 5000, "m": 5000, "p": 50,
         "cumulative": False},
        # the whole job of a small instance: distances in host memory to the best facilities, 200 generations
        {"name": "job_graph100", "kind": "job", "family": "graph", "n": 100, "m": 100, "p": 5, "pop": 64, "gens": 200,
         "init": "floyd", "migration": "deme"},
        # generations of the 900-node graph's GA, the library's main use
        {"name": "ga_graph900", "kind": "ga", "family": "graph", "n": 900, "m": 900, "p": 90, "pop": 1024, "gens": 100,
         "init": "floyd", "migration": "deme"},
        # many uneven instances evolved together, half graphs and half Euclidean
        {"name": "batch_ga48", "kind": "batch", "count": 48, "shapes": 3, "nmax": 5000, "pop": 256, "gens": 4},
        # generations with the learned swap proposal on the clustered 5000-point instance
        {"name": "learned_gmm5000_p500", "kind": "learned", "family": "gmm", "n": 5000, "m": 5000, "p": 500,
         "pop": 1024, "gens": 10},
        # training of the proposal's perceptron: one epoch in mini-batches, forward, backward and Adam
        {"name": "train_65536", "kind": "train", "rows": 65536, "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _open_count(rng, m):
    """Open facilities from 5 to a tenth of them, as the batched configuration, over their logarithm."""
    return _log_int(rng, 5, max(6, m // 10))


def draw(rng):
    kind = rng.choice(["eval"] * 4 + ["ga"] * 3 + ["batch"] * 2 + ["tables", "job", "learned", "stats", "forward",
                                                                 "train"])
    family = rng.choice(["euclid", "gmm", "graph"])
    cap = 1500 if family == "graph" else 10000
    if kind == "eval":
        m = _log_int(rng, 100, cap)
        n = m if family == "graph" or rng.random() < 0.5 else _log_int(rng, 100, cap)
        p = max(_open_count(rng, m), m // 1000)
        return dict(kind=kind, family=family, n=n, m=m, p=p, pop=_log_int(rng, 32, 4096),
                    cumulative=rng.random() < 0.3, host=rng.random() < 0.2)
    if kind == "tables":
        m = _log_int(rng, 100, min(cap, 5000))
        return dict(kind=kind, family=family, n=m, m=m, p=_open_count(rng, m), cumulative=rng.random() < 0.3)
    if kind in ("ga", "job"):
        m = _log_int(rng, 100, min(cap, 2500))
        return dict(kind=kind, family=family, n=m, m=m, p=_open_count(rng, m), pop=rng.choice([64, 256, 512, 1024]),
                    gens=_log_int(rng, 5, 60), init=rng.choice(["floyd", "floyd", "combinadic"]) if m <= 1000
                    else "floyd", migration=rng.choice(["deme", "deme", "team"]))
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 4, 32), shapes=rng.randrange(1 << 16), nmax=2500,
                    pop=rng.choice([64, 128, 256]), gens=rng.choice([0, 1, 2]))
    if kind == "learned":
        m = _log_int(rng, 200, 3000)
        return dict(kind=kind, family=rng.choice(["euclid", "gmm"]), n=m, m=m, p=_open_count(rng, m),
                    pop=rng.choice([64, 256, 512]), gens=_log_int(rng, 2, 8))
    if kind == "stats":
        m = _log_int(rng, 200, 5000)
        return dict(kind=kind, family=rng.choice(["euclid", "gmm"]), n=m, m=m, p=max(_open_count(rng, m), m // 100),
                    pop=_log_int(rng, 32, 512))
    if kind == "forward":
        return dict(kind=kind, rows=_log_int(rng, 1000, 2_000_000))
    return dict(kind="train", rows=_log_int(rng, 2000, 65536), batch=rng.choice([1024, 2048, 4096]))


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _points(family, n, seed, salt):
    g = _gen(seed, salt)
    if family == "euclid":
        return torch.rand(n, 2, generator=g, device=DEV, dtype=torch.float64)
    # 50 equal-weight Gaussian components, sigma 0.02, points redrawn until inside the unit square
    centres = torch.rand(50, 2, generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
    which = torch.randint(0, 50, (n,), generator=g, device=DEV)
    pts = torch.full((n, 2), -1.0, device=DEV, dtype=torch.float64)
    for _ in range(64):
        fresh = centres[which] + 0.02 * torch.randn(n, 2, generator=g, device=DEV, dtype=torch.float64)
        out = ((pts < 0) | (pts > 1)).any(1, keepdim=True)
        pts = torch.where(out, fresh, pts)
    return pts.clamp_(0.0, 1.0)


def _points_distance(a, b):
    d = torch.empty(a.shape[0], b.shape[0], dtype=torch.int32, device=DEV)
    for r in range(0, a.shape[0], 1024):
        d[r:r + 1024] = torch.floor(1e4 * torch.hypot(a[r:r + 1024, 0:1] - b[:, 0], a[r:r + 1024, 1:2] - b[:, 1]) + 0.5)
    return d


def _graph_distance(n, edges, seed):
    """All-pairs shortest paths of a random recursive tree plus random edges, weights 1..100."""
    rng = np.random.default_rng(int(seed))
    v = np.arange(1, n)
    u = (rng.random(n - 1) * v).astype(np.int64)
    extra = max(0, edges - (n - 1))
    a, b = rng.integers(0, n, extra), rng.integers(0, n, extra)
    us, vs = np.concatenate([u, a]), np.concatenate([v, b])
    w = rng.integers(1, 101, us.size).astype(np.int32)
    big = 1 << 28
    adj = np.full((n, n), big, dtype=np.int32)
    np.minimum.at(adj, (us, vs), w)
    np.minimum.at(adj, (vs, us), w)
    np.fill_diagonal(adj, 0)
    d = torch.from_numpy(adj).to(DEV)
    tmp = torch.empty_like(d)
    for k in range(n):
        torch.add(d[:, k:k + 1], d[k:k + 1, :], out=tmp)
        torch.minimum(d, tmp, out=d)
    return d


def _distances(family, n, m, seed):
    if family == "graph":
        return _graph_distance(n, 18 * n if n >= 500 else 2 * n, seed)
    clients = _points(family, n, seed, 2)
    return _points_distance(clients, clients if m == n else _points(family, m, seed, 3))


def _masks(pop, m, p, seed):
    """Uniformly random p-subsets as bitsets of ceil(m / 32) words (int32 views of the uint32 words)."""
    W = (m + 31) // 32
    g = _gen(seed, 4)
    out = torch.empty(pop, W, dtype=torch.int32, device=DEV)
    bit = (torch.ones(32, dtype=torch.int64, device=DEV) << torch.arange(32, device=DEV))
    for r in range(0, pop, 512):
        k = min(512, pop - r)
        sel = torch.rand(k, m, generator=g, device=DEV).topk(p, dim=1).indices
        on = torch.zeros(k, W * 32, dtype=torch.int64, device=DEV)
        on.scatter_(1, sel, 1)
        out[r:r + k] = (on.view(k, W, 32) * bit).sum(2).to(torch.int32)
    return out


def _batch_sizes(case):
    """n = m log-uniform in [100, nmax], p uniform in [5, n/10]; even entries graphs, odd ones Euclidean."""
    rng = random.Random(case["shapes"])
    sizes = []
    for _ in range(case["count"]):
        n = _log_int(rng, 100, case["nmax"])
        sizes.append((n, rng.randint(5, max(6, n // 10))))
    return sizes


def _batch_instance(k, n, p, seed):
    d = _graph_distance(n, 4 * n, seed + k) if k % 2 == 0 else _distances("euclid", n, n, seed + k)
    return pm.Instance(d, p)


def _params(seed):
    """Weights of a perceptron in the state training leaves it in: He-sized, small biases."""
    rng = np.random.default_rng([int(seed), 5])
    parts = [rng.normal(0, math.sqrt(2 / 16), 16 * 128), rng.normal(0, 0.05, 128),
             rng.normal(0, math.sqrt(2 / 128), 128 * 128), rng.normal(0, 0.05, 128),
             rng.normal(0, math.sqrt(1 / 128), 128), rng.normal(0, 0.05, 1)]
    return np.concatenate(parts).astype(np.float32)


def _rows(rows, seed):
    """Input rows shaped like the move features (8 of them, then zeros) as bf16, and the targets of those moves."""
    g = _gen(seed, 6)
    e = -torch.log(torch.rand(rows, 4, generator=g, device=DEV).clamp_min(1e-6))
    loss, gain = 0.6 * e[:, 0], 0.4 * e[:, 1]
    x = torch.zeros(rows, 16, device=DEV)
    x[:, 0], x[:, 1], x[:, 2], x[:, 3] = loss, gain, e[:, 2], e[:, 3]
    x[:, 4], x[:, 5], x[:, 6], x[:, 7] = loss - gain, torch.log1p(loss), torch.log1p(gain), 0.1
    t = (loss - gain + 0.2 * loss * gain + 0.02 * torch.randn(rows, generator=g, device=DEV)).contiguous()
    return x.to(torch.bfloat16).contiguous(), t


def _model(seed):
    md = pm.Model(seed=int(seed) & 0xFFFF)
    md.set_params(_params(seed))
    return md


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case, "seed": int(seed)}
    if k == "batch":
        sizes = _batch_sizes(case)
        s["insts"] = [_batch_instance(i, n, p, int(seed) * 1000) for i, (n, p) in enumerate(sizes)]
        s["batch"] = pm.Batch(s["insts"])
        if case["gens"] == 0:
            s["pops"] = [case["pop"]] * len(sizes)
            s["masks"] = torch.cat([_masks(case["pop"], n, p, int(seed) * 1000 + i).reshape(-1)
                                    for i, (n, p) in enumerate(sizes)])
        return s
    if k in ("forward", "train"):
        s["x"], s["t"] = _rows(case["rows"], seed)
        s["model"], s["params"] = _model(seed), _params(seed)
        return s
    d = _distances(case["family"], case["n"], case["m"], seed)
    if k == "job":
        s["d"] = d.cpu().numpy()
        return s
    if k == "tables":
        L = case["m"] - case["p"] + 1
        s["d"] = d
        s["pi"] = torch.empty(case["n"], L, dtype=torch.int16, device=DEV)
        s["delta"] = torch.empty(case["n"], L, dtype=torch.int32, device=DEV)
        return s
    s["inst"] = pm.Instance(d, case["p"], cumulative=case.get("cumulative", False))
    if k == "learned":
        s["model"] = _model(seed)
    if k in ("eval", "stats"):
        s["masks"] = _masks(case["pop"], case["m"], case["p"], seed)
        if case.get("host"):
            s["masks"] = s["masks"].cpu().numpy().view(np.uint32)
    return s


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------

def _run_ga(ga, gens):
    trace = ga.step(gens)
    best, ran, evals, mask = ga.result()
    masks, costs = ga.population()
    ga.close()
    return {"trace": trace, "best": best, "gens": ran, "evals": evals, "mask": mask.view(np.int32),
            "masks": masks.view(np.int32), "costs": costs}


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "eval":
        return s["inst"].eval(s["masks"])
    if k == "tables":
        inst = pm.Instance(s["d"], c["p"], cumulative=c["cumulative"])
        pm.pm_instance_tables(inst.handle, s["pi"], s["delta"])
        inst.close()
        return {"pi": s["pi"], "delta": s["delta"]}
    if k == "job":
        inst = pm.Instance(s["d"], c["p"])
        out = _run_ga(pm.GA(inst, seed=s["seed"], pop=c["pop"], init=c["init"], migration=c["migration"]), c["gens"])
        inst.close()
        return out
    if k == "ga":
        return _run_ga(pm.GA(s["inst"], seed=s["seed"], pop=c["pop"], init=c["init"], migration=c["migration"]),
                       c["gens"])
    if k == "learned":
        return _run_ga(pm.GA(s["inst"], seed=s["seed"], pop=c["pop"], model=s["model"]), c["gens"])
    if k == "batch":
        if c["gens"] == 0:
            return s["batch"].eval(s["masks"], s["pops"])
        ga = s["batch"].ga(seed=s["seed"], pop=c["pop"])
        out = {"trace": ga.step(c["gens"]), "best": [], "evals": [], "costs": []}
        masks = []
        for i in range(ga.K):
            best, _, evals, _ = ga.result(i)
            m, costs = ga.population(i)
            out["best"].append(best)
            out["evals"].append(evals)
            out["costs"].append(costs)
            masks.append(m.reshape(-1))
        ga.close()
        out["best"], out["evals"] = np.array(out["best"]), np.array(out["evals"])
        out["costs"], out["masks"] = np.concatenate(out["costs"]), np.concatenate(masks).view(np.int32)
        return out
    if k == "stats":
        n = (c["pop"], c["m"])
        gain, loss = (torch.empty(n, dtype=torch.int64, device=DEV) for _ in range(2))
        cap, assign = (torch.empty(n, dtype=torch.int32, device=DEV) for _ in range(2))
        pm.pm_swap_stats(s["inst"].handle, s["masks"], c["pop"], gain, cap, loss, assign)
        return {"gain": gain, "cap": cap, "loss": loss, "assign": assign}
    if k == "forward":
        return s["model"].forward(s["x"])
    s["model"].set_params(s["params"])
    losses = s["model"].train(s["x"], s["t"], epochs=1, batch=c["batch"], lr=2e-3, seed=s["seed"])
    return {"losses": losses, "params": s["model"].params()}


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------

def _scan_work(n, m, p, pop, evals):
    """Bytes: the part of every client's ordering (2 + 4 bytes a rank) that some individual of the population reaches
    (the largest of `pop` first open ranks, each about (m + 1) / (p + 1)), the bitsets once and the costs once.
    Operations: one addition per (individual evaluated, client)."""
    ranks = min(m - p + 1, (m + 1) / (p + 1) * (math.log(pop) + 1))
    return {"bytes": n * ranks * 6 + pop * ((m + 31) // 32 * 4 + 8), "flops": float(evals) * n}


def _ga_work(n, m, p, pop, gens):
    lg = int(math.log2(min(pop, 256)))
    w = _scan_work(n, m, p, pop, gens * pop * (1 + lg + lg))
    return w


def work(case):
    k = case["kind"]
    if k in ("forward", "train"):
        macs = 16 * 128 + 128 * 128 + 128
        times = 2 if k == "forward" else 6
        return {"bytes": case["rows"] * 36.0 + 4 * 18817, "flops": float(case["rows"]) * macs * times}
    if k == "batch":
        parts = [_ga_work(n, n, p, case["pop"], case["gens"]) if case["gens"] else
                 _scan_work(n, n, p, case["pop"], case["pop"]) for n, p in _batch_sizes(case)]
        return {"bytes": sum(w["bytes"] for w in parts), "flops": sum(w["flops"] for w in parts)}
    n, m, p = case["n"], case["m"], case["p"]
    if k == "eval":
        return _scan_work(n, m, p, case["pop"], case["pop"])
    if k == "tables":
        return {"bytes": n * m * 4.0 + n * (m - p + 1) * 6.0, "flops": float(n) * m}
    if k == "stats":
        w = _scan_work(n, m, p, case["pop"], 2 * case["pop"])
        return {"bytes": w["bytes"] + case["pop"] * m * 24.0, "flops": w["flops"]}
    w = _ga_work(n, m, p, case["pop"], case["gens"])
    if k == "job":
        w["bytes"] += n * m * 4.0
    if k == "learned":
        rows = case["gens"] * case["pop"] * p * 4
        w["flops"] += rows * 2.0 * (16 * 128 + 128 * 128 + 128)
    return w


def exact(case, seed):
    """Predictions in 64 bits.  Costs, tables, populations and statistics are whole numbers, which have to be equal; a
    training run's weights depend on the rounding of every step before."""
    if case["kind"] != "forward":
        return None
    x, _ = _rows(case["rows"], seed)
    v = torch.from_numpy(_params(seed)).to(DEV).double()
    w1, b1, w2, b2, w3, b3 = torch.split(v, [16 * 128, 128, 128 * 128, 128, 128, 1])
    y = torch.empty(case["rows"], dtype=torch.float64, device=DEV)
    for r in range(0, case["rows"], 1 << 16):
        h = torch.relu(x[r:r + (1 << 16)].double() @ w1.view(16, 128) + b1)
        y[r:r + (1 << 16)] = torch.relu(h @ w2.view(128, 128) + b2) @ w3 + b3
    return y
