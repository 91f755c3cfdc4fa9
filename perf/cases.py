"""Performance cases: the calls a program built on dagrt makes, through its Python binding.

Three groups, as the library is used: scheduling batches of task graphs (`Context.load` +
`LoadedBatch.schedule`: the paper's schedule and its bound), judging other SM allocations on
a schedule's structure (`LoadedBatch.bound`, `LoadedBatch.search`), and the learned proposer
(`Model.logits`, `Model.propose`, `Model.train_step`). Graph shapes, loads, SM counts and
levels are those of this repository's workload configurations, sweeps and training driver.
"""
from __future__ import annotations

import heapq
import math

import numpy as np
import torch

from paper_2602_20826_gb300.dagrt import (SEARCH_EXHAUSTIVE, SEARCH_PERTURB, SEARCH_RANDOM, Context, Model)
from paper_2602_20826_gb300.workloads import Batch

# SM levels of the proposer at M = 148, and the perturbation codes of the plain search
LEVELS = (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 148)
CODES = (0,) * 12 + (1, 2, 3, 4)
MODES = {"random": SEARCH_RANDOM, "perturb": SEARCH_PERTURB, "exhaustive": SEARCH_EXHAUSTIVE}
HIDDEN, FEAT, MAX_LEVELS = 128, 16, 16  # the network's fixed sizes (include/dagrt.h)

# what a caller asks a schedule for: the bound alone; the bound beside the baselines of the
# evaluation sweeps; the whole schedule, to launch it
FIELDS = {
    "bound": {"bound": "d8", "status": "d4"},
    "sweep": {"bound": "d8", "status": "d4", "greedy": "d8", "greedy_unaware": "d8", "graham_para": "d8"},
    "plan": {"bound": "d8", "status": "d4", "n_groups": "d4", "n_rows": "d4", "n_extra": "d8", "crit_path": "d8",
             "level": "n4", "wanc": "n8", "block_of": "n4", "group_of": "n4", "exec_group": "n4", "m": "n4",
             "group_R": "n8", "row_id": "r4", "row_group": "r4", "row_m0": "r4", "row_load": "r8"},
}


def _er(n, lo, hi, p, M=148, loads="log", frac=0.3):
    return {"graph": "er", "n_dags": n, "v_lo": lo, "v_hi": hi, "p": p, "M": M, "loads": loads, "frac": frac}


def listed():
    return [
        # one task admitted on its own, host arrays in and the bound out: latency only
        {"name": "schedule_one_task", "kind": "schedule", "host": True, "fields": "bound", "variant": 0,
         **_er(1, 20, 20, 0.2, 8, "uniform100", 0.5)},
        # a sweep point of the evaluation: 1,000 fork-join tasks from host arrays, baselines beside the bound
        {"name": "schedule_sweep_point", "kind": "schedule", "host": True, "fields": "sweep", "variant": 0,
         "graph": "forkjoin", "n_dags": 1000, "width": 16, "depth_lo": 5, "depth_hi": 8, "M": 32,
         "loads": "uniform39", "frac": 1.0},
        # the headline: 10,000 device-resident tasks of 20-200 kernels, bound only
        {"name": "schedule_10k", "kind": "schedule", "host": False, "fields": "bound", "variant": 0,
         **_er(10000, 20, 200, 0.1)},
        # mid-size tasks with the whole schedule written out
        {"name": "schedule_mid_plan", "kind": "schedule", "host": False, "fields": "plan", "variant": 0,
         **_er(1000, 50, 500, 0.05)},
        # compiler-style graphs of 2,000-20,000 kernels
        {"name": "schedule_large", "kind": "schedule", "host": False, "fields": "bound", "variant": 0,
         "graph": "layered", "n_dags": 200, "v_lo": 2000, "v_hi": 20000, "depth_lo": 20, "depth_hi": 60, "M": 148,
         "loads": "lognormal", "frac": 0.3},
        # candidate allocations held in memory, powers of two, 4 structures x 64
        {"name": "bound_blocks_of_64", "kind": "bound", "n_variants": 4, "n_alloc": 64, "alloc": "pow2",
         **_er(1000, 50, 500, 0.05)},
        # a few hand-made allocations of any SM count, an odd number of them
        {"name": "bound_any_sms", "kind": "bound", "n_variants": 2, "n_alloc": 37, "alloc": "any",
         **_er(1000, 20, 200, 0.1)},
        # the plain search of the learning set-up: sparse perturbations of 4 schedules
        {"name": "search_perturb", "kind": "search", "mode": "perturb", "n_variants": 4, "n_alloc": 64,
         **_er(500, 100, 1000, 0.05)},
        # the exhaustive search that labels small tasks on a small GPU
        {"name": "search_exhaustive", "kind": "search", "mode": "exhaustive", "n_variants": 1, "n_alloc": 9 ** 6,
         **_er(2000, 3, 6, 0.35, 8, "uniform40", 0.5)},
        # the network alone on a batch that is kept: the scores of every kernel
        {"name": "logits", "kind": "logits", "n_levels": 15, **_er(300, 100, 1000, 0.05)},
        # the learned proposer on a new batch: schedule, network, top-16, exact check
        {"name": "propose", "kind": "propose", "k": 16, "n_levels": 15, **_er(300, 100, 1000, 0.05)},
        # one training step: forward, backward, Adam
        {"name": "train_step", "kind": "train", "n_levels": 15, **_er(1000, 20, 200, 0.1)},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("schedule", "schedule", "schedule", "bound", "search", "logits", "propose", "train"))
    hi = _log_int(rng, 5, 1000)
    c = {"kind": kind, **_er(1, max(1, int(hi * rng.uniform(0.1, 1.0))), hi, rng.choice((0.05, 0.1, 0.2, 0.35)),
                             rng.choice((8, 30, 32, 64, 128, 148, 148, 256)), rng.choice(("log", "uniform100")),
                             rng.choice((0.3, 0.5, 1.0)))}
    if kind == "schedule":
        fields = rng.choice(("bound", "bound", "sweep", "plan"))
        c.update(host=fields != "plan" and rng.random() < 0.5, fields=fields, variant=rng.choice((0, 0, 0, 1, 2, 3, 4)))
        shape = rng.random()
        if shape < 0.2:
            vh = _log_int(rng, 500, 20000)
            c.update(graph="layered", v_lo=max(2, int(vh * rng.uniform(0.2, 1.0))), v_hi=vh, depth_lo=20, depth_hi=60,
                     loads="lognormal")
            c["n_dags"] = _log_int(rng, 1, max(1, min(200, 1500000 // vh)))
        elif shape < 0.4:
            c.update(graph="forkjoin", width=rng.randint(2, 64), depth_lo=4, depth_hi=rng.randint(4, 64),
                     loads="uniform39", n_dags=_log_int(rng, 1, 1000))
        else:
            c["n_dags"] = _log_int(rng, 1, max(1, min(10000, int(4e8 / hi ** 2))))
    elif kind == "bound":
        c.update(n_variants=rng.randint(1, 4), n_alloc=rng.choice((1, 7, 16, 30, 37, 64, 64, 100, 128)),
                 alloc=rng.choice(("pow2", "any")))
        cap = 2e8 / (2 * hi * c["n_variants"] * c["n_alloc"])
        c["n_dags"] = _log_int(rng, 1, max(1, min(2000, int(cap), int(1e8 / hi ** 2))))
    elif kind == "search":
        c["mode"] = rng.choice(("random", "perturb", "exhaustive"))
        if c["mode"] == "exhaustive":
            c.update(_er(_log_int(rng, 1, 1500), 2, rng.randint(3, 5), 0.35, 8, "uniform40", 0.5), n_variants=1,
                     n_alloc=9 ** 5)
        else:
            c.update(n_variants=rng.randint(1, 4), n_alloc=rng.choice((15, 64, 100, 256)))
            cap = 1e8 / (hi * c["n_variants"] * c["n_alloc"])
            c["n_dags"] = _log_int(rng, 1, max(1, min(1000, int(cap), int(1e8 / hi ** 2))))
    else:
        c["n_dags"] = _log_int(rng, 1, max(1, min(2000, int(1e5 / hi), int(8e7 / hi ** 2))))
        c["n_levels"] = rng.choice((5, 8, 15))
        if kind == "propose":
            c["k"] = rng.choice((1, 8, 16))
    return c


# ---------------------------------------------------------------- inputs

def _loads(kind, u, gauss):
    if kind == "log":  # floor(10^(4U)): 1 .. 9,999 ticks
        w = torch.floor(10.0 ** (4.0 * u))
    elif kind == "lognormal":
        w = torch.floor(torch.exp(4.0 + 1.5 * gauss) + 0.5)
    else:  # "uniformH": 1 .. H ticks
        w = 1 + torch.floor(int(kind[len("uniform"):]) * u)
    return w.clamp(1, 2 ** 32 - 1).to(torch.int64)


def _er_edges(case, gen, V, node_off):
    """Each pair i < j of a DAG is an edge with probability p: geometric gaps over all pairs."""
    dev = V.device
    pairs = V * (V - 1) // 2
    poff = torch.cat([pairs.new_zeros(1), pairs.cumsum(0)])
    total = int(poff[-1])
    want = int(total * case["p"] + 8 * math.sqrt(total * case["p"] + 1) + 16)
    u = torch.rand(want, generator=gen, device=dev, dtype=torch.float64)
    t = (1 + torch.floor(torch.log1p(-u) / math.log1p(-case["p"]))).to(torch.int64).cumsum(0) - 1
    t = t[t < total]
    d = torch.searchsorted(poff, t, right=True) - 1
    q, v = t - poff[d], V[d]
    b = (2 * v - 1).double()
    i = torch.floor((b - torch.sqrt(b * b - 8.0 * q.double())) / 2).to(torch.int64)
    i -= (i * v - i * (i + 1) // 2 > q).long()
    i += ((i + 1) * v - (i + 1) * (i + 2) // 2 <= q).long()
    j = q - (i * v - i * (i + 1) // 2) + i + 1
    return node_off[d] + i, node_off[d] + j


def _layer_widths(case, rng):
    """Layer widths of every DAG: raw widths scaled to a node count, or a source, `depth`
    layers and a sink."""
    out = []
    for _ in range(case["n_dags"]):
        depth = int(rng.integers(case["depth_lo"], case["depth_hi"] + 1))
        if case["graph"] == "forkjoin":
            out.append(np.concatenate([[1], rng.integers(2, case["width"] + 1, depth), [1]]))
            continue
        V = int(rng.integers(case["v_lo"], case["v_hi"] + 1))
        depth = min(depth, V)
        raw = rng.integers(1, 65, depth).astype(np.float64)
        w = np.maximum(1, np.floor(raw * V / raw.sum())).astype(np.int64)
        while w.sum() > V:
            w[np.argmax(w)] -= 1
        w[-1] += V - w.sum()
        out.append(w)
    return out


def _layered_edges(case, gen, widths, V, node_off, dev):
    """1-3 predecessors from the layer before; layered graphs add skip edges (2%), fork-join
    graphs a sink that waits for its whole layer and a successor for every node."""
    w = torch.from_numpy(np.concatenate(widths).astype(np.int64)).to(dev)          # per layer
    depth = torch.tensor([len(x) for x in widths], device=dev)
    ldag = torch.repeat_interleave(torch.arange(len(widths), device=dev), depth)
    first = torch.cat([depth.new_zeros(1), depth.cumsum(0)])[:-1]                  # a DAG's first layer
    lidx = torch.arange(len(w), device=dev) - first[ldag]
    lstart = torch.cat([w.new_zeros(1), w.cumsum(0)])                              # first node, batch-wide
    layer = torch.repeat_interleave(torch.arange(len(w), device=dev), w)           # layer of each node
    N = int(lstart[-1])
    node = torch.arange(N, device=dev)
    fork = case["graph"] == "forkjoin"
    last = (torch.cat([ldag[1:], ldag.new_full((1,), -1)]) != ldag)[layer]         # in its DAG's last layer

    def rand():
        return torch.rand(N, generator=gen, device=dev, dtype=torch.float64)

    inner = lidx[layer] >= 1
    npred = 1 + torch.floor(3 * rand()).long()
    src, dst = [], []
    for k in range(3):
        ok = inner & (npred > k) & ~(last if fork else torch.zeros_like(last))
        pl = (layer - 1).clamp(min=0)
        s = lstart[pl] + torch.floor(rand() * w[pl]).long()
        src.append(s[ok])
        dst.append(node[ok])
    if fork:  # nodes without a successor, and the sink's predecessors
        has = torch.zeros(N, dtype=torch.bool, device=dev)
        has[torch.cat(src)] = True
        nxt = lstart[(layer + 1).clamp(max=len(w) - 1)]
        ok = ~has & ~last
        src.append(node[ok])
        dst.append(nxt[ok])
        pen = (~last) & last[nxt.clamp(max=N - 1)]
        src.append(node[pen])
        dst.append(nxt[pen])
    else:
        ok = (lidx[layer] >= 2) & (rand() < 0.02)
        lo = node_off[ldag[layer]]
        s = lo + torch.floor(rand() * (lstart[(layer - 1).clamp(min=0)] - lo)).long()
        src.append(s[ok])
        dst.append(node[ok])
    key = torch.unique(torch.cat(src) * N + torch.cat(dst))
    return key // N, key % N


def _graphs(case, seed):
    """The batch as torch CUDA tensors in the layout of `Context.load`."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    n = case["n_dags"]
    # the sizes belong to the case (its outputs then have one shape), their order to the seed
    rng = np.random.default_rng(20260226)
    order = np.random.default_rng(int(seed)).permutation(n)
    if case["graph"] == "er":
        sizes = rng.integers(case["v_lo"], case["v_hi"] + 1, n)[order]
        widths = None
    else:
        widths = _layer_widths(case, rng)
        widths = [widths[d] for d in order]
        sizes = np.array([x.sum() for x in widths])
    V = torch.from_numpy(sizes.astype(np.int64)).to(dev)
    node_off = torch.cat([V.new_zeros(1), V.cumsum(0)])
    N = int(node_off[-1])
    if widths is None:
        src, dst = _er_edges(case, gen, V, node_off)
    else:
        src, dst = _layered_edges(case, gen, widths, V, node_off, dev)
    dag = torch.repeat_interleave(torch.arange(n, device=dev), V)
    deg = torch.cat([V.new_zeros(1), torch.bincount(src, minlength=N).cumsum(0)])
    edge_off = deg[node_off]
    entry_dag = torch.repeat_interleave(torch.arange(n, device=dev), V + 1)
    row_ptr = deg[torch.arange(N + n, device=dev) - entry_dag] - edge_off[entry_dag]
    u = torch.rand(N, generator=gen, device=dev, dtype=torch.float64)
    gauss = torch.randn(N, generator=gen, device=dev, dtype=torch.float64)
    k64 = torch.randint(round(64 * case["frac"]), 65, (N,), generator=gen, device=dev)
    return {"node_off": node_off, "edge_off": edge_off, "row_ptr": row_ptr.to(torch.int32),
            "col": (dst - node_off[dag[dst]]).to(torch.int32), "wcet": _loads(case["loads"], u, gauss),
            "k64": k64.to(torch.uint8)}, gen


def _params(seed):
    """He-uniform weights in the model's flat layout, zero biases."""
    rng = np.random.default_rng([int(seed), 3])
    out = []
    for fan in (3 * FEAT, 3 * HIDDEN, 3 * HIDDEN):
        out += [rng.uniform(-1, 1, fan * HIDDEN) * math.sqrt(6 / fan), np.zeros(HIDDEN)]
    out += [rng.uniform(-1, 1, HIDDEN * MAX_LEVELS) * math.sqrt(6 / HIDDEN), np.zeros(MAX_LEVELS)]
    return np.concatenate(out).astype(np.float32)


def _labels(g, n_levels):
    """Heavier kernels get more SMs: the level index a bucket of log2 of the load."""
    return (torch.log2(g["wcet"].double()) * n_levels / 13.3).long().clamp(0, n_levels - 1).to(torch.int8)


LR = 2e-3


def prepare(case, seed):
    dev, kind = torch.device("cuda"), case["kind"]
    g, gen = _graphs(case, seed)
    n, N, M = case["n_dags"], int(g["node_off"][-1]), case["M"]
    ctx = Context(0, torch.cuda.current_stream().cuda_stream)
    s = {"kind": kind, "case": case, "ctx": ctx, "dev": g, "M": M}
    size = {"d": n, "n": N, "r": 2 * N}

    def zeros(spec):
        t = {"1": torch.uint8, "4": torch.int32, "8": torch.int64}[spec[1]]
        return torch.zeros(max(1, size[spec[0]]), dtype=t, device=dev)

    if kind == "schedule":
        s["fields"] = tuple(FIELDS[case["fields"]])
        if case["host"]:
            s["host"] = Batch(*(g[k].cpu().numpy() for k in ("node_off", "edge_off", "row_ptr", "col", "wcet", "k64")), M)
        else:
            s["out"] = {f: zeros(t) for f, t in FIELDS[case["fields"]].items()}
        return s
    if kind in ("bound", "search"):
        s["batch"] = ctx.load(g, M)
        s["variants"] = list(range(case["n_variants"]))
        for v in s["variants"]:
            s["batch"].schedule(v, out={"status": torch.zeros(n, dtype=torch.int32, device=dev)})
        s["out"] = {"best_bound": zeros("d8"), "best_cand": zeros("d4")}
        if kind == "search":
            s["levels"] = CODES if case["mode"] == "perturb" else tuple(range(1, 9)) if case["mode"] == "exhaustive" else LEVELS
            s["out"]["best_m"] = zeros("r1")
            s["seed"] = int(seed)
            return s
        nv, na = case["n_variants"], case["n_alloc"]
        s["stride"] = (nv * na + 15) // 16 * 16
        levels = (1, 2, 4, 8, 16, 32) if case["alloc"] == "pow2" else tuple(range(1, min(M, 255) + 1))
        pick = torch.randint(len(levels), (2 * N, s["stride"]), generator=gen, device=dev, dtype=torch.int16)
        s["cand"] = torch.tensor(levels, dtype=torch.uint8, device=dev)[pick.int()]
        s["cand"][:, 0:nv * na:na] = 0  # allocation 0 of each structure keeps the schedule's own SMs
        s["out"]["out_bound"] = torch.zeros(n * nv * na, dtype=torch.int64, device=dev)
        return s
    s["model"] = Model(ctx, LEVELS[:case["n_levels"]], seed=0)
    s["model"].params(set_to=_params(seed))
    s["logits"] = torch.zeros(N * case["n_levels"], dtype=torch.float32, device=dev)
    if kind == "propose":
        nc = case["k"] + 1
        s["out"] = {"out_bound": torch.zeros(n * nc, dtype=torch.int64, device=dev), "best_bound": zeros("d8"),
                    "best_cand": zeros("d4"), "best_m": zeros("r1")}
        return s
    s["batch"] = ctx.load(g, M)
    if kind == "train":
        s["labels"] = _labels(g, case["n_levels"]).cpu().numpy()
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "schedule":
        if case["host"]:
            b = s["ctx"].load(s["host"])
            r = b.schedule(case["variant"], fields=s["fields"])
            r.pop("rc")
        else:
            b = s["ctx"].load(s["dev"], s["M"])
            r = b.schedule(case["variant"], out=s["out"])
        b.free()
        return r
    if kind == "bound":
        o = s["out"]
        s["batch"].bound(s["variants"], case["n_alloc"], s["cand"], s["stride"], o["out_bound"], o["best_bound"], o["best_cand"])
        return o
    if kind == "search":
        return s["batch"].search(s["variants"], case["n_alloc"], s["levels"], s["seed"], out=s["out"], mode=MODES[case["mode"]])
    if kind == "logits":
        return s["model"].logits(s["batch"], out=s["logits"])
    if kind == "propose":
        b = s["ctx"].load(s["dev"], s["M"])
        z = s["model"].logits(b, out=s["logits"])
        o = s["model"].propose(b, case["k"], out=s["out"])
        b.free()
        return {"logits": z, **o}
    loss = s["model"].train_step(s["batch"], s["labels"], LR)
    return {"loss": loss, "params": s["model"].params()}


# ---------------------------------------------------------------- what a pass cannot do without

def _mean_size(case):
    """Expected (nodes, edges) of one DAG."""
    if case["graph"] == "er":
        v = np.arange(case["v_lo"], case["v_hi"] + 1, dtype=np.float64)
        return float(v.mean()), float((v * (v - 1) / 2).mean() * case["p"])
    if case["graph"] == "forkjoin":
        depth, w = (case["depth_lo"] + case["depth_hi"]) / 2, (2 + case["width"]) / 2
        return 2 + depth * w, 2 * depth * w
    v = (case["v_lo"] + case["v_hi"]) / 2
    return v, 2 * v


def work(case):
    n, kind = case["n_dags"], case["kind"]
    v, e = _mean_size(case)
    N, E = n * v, n * e
    graph = 16 * (n + 1) + 4 * (N + n) + 4 * E + 9 * N  # CSR, loads, fractions
    if kind == "schedule":
        size = {"d": n, "n": N, "r": N}  # at least one plan row per node
        return {"bytes": graph + sum(size[t[0]] * int(t[1]) for t in FIELDS[case["fields"]].values()), "flops": 0}
    if kind == "bound":  # a byte per candidate and row, the rows, the bounds; an addition per candidate and row
        c = case["n_variants"] * case["n_alloc"]
        return {"bytes": N * c + 13 * N * case["n_variants"] + n * (8 * c + 12), "flops": N * c}
    if kind == "search":
        c = case["n_variants"] * case["n_alloc"]
        rows = N * c
        if case["mode"] == "exhaustive":  # distinct assignments only
            rows = n * float(np.mean([x * min(case["n_alloc"], 9 ** x) for x in range(case["v_lo"], case["v_hi"] + 1)]))
        return {"bytes": 13 * N * case["n_variants"] + 12 * n + N, "flops": rows}
    # the network's products; its inputs, parameters and logits
    mul = 2 * N * HIDDEN * (3 * FEAT + 6 * HIDDEN + case["n_levels"])
    add = 4 * E * (FEAT + 2 * HIDDEN)
    params = 4 * len(_params(0))
    if kind == "logits":
        return {"bytes": N * (2 * FEAT + 4 * case["n_levels"]) + 8 * E + params, "flops": mul + add}
    if kind == "propose":
        return {"bytes": graph + params + 4 * N * case["n_levels"] + n * (8 * case["k"] + 20) + N, "flops": mul + add}
    return {"bytes": N * (2 * FEAT + 1) + 8 * E + 6 * params, "flops": 3 * mul + 2 * add}


# ---------------------------------------------------------------- 64-bit values of the network's outputs

def _time(x, k, m, M):
    return max(1, -(-(-(-m // M) * x * (64 * m - k * (m - 1))) // (64 * m)))


def _schedule(succ, x, k, M):
    """Level, W^anc and SM count of every node of one DAG (Kahn levels, Eq.2, Alg.1, Alg.2),
    in whole numbers."""
    V = len(succ)
    indeg, pred = [0] * V, [[] for _ in range(V)]
    for u in range(V):
        for t in succ[u]:
            indeg[t] += 1
            pred[t].append(u)
    level, left, order = [0] * V, indeg[:], [u for u in range(V) if not indeg[u]]
    reach = np.zeros((V, V), bool)  # reach[v]: the ancestors of v
    for u in order:
        if pred[u]:
            reach[u] = reach[pred[u]].any(axis=0)
            reach[u, pred[u]] = True
        for t in succ[u]:
            level[t] = max(level[t], level[u] + 1)
            left[t] -= 1
            if not left[t]:
                order.append(t)
    wanc = reach.astype(np.int64) @ np.array(x, np.int64) + np.array(x, np.int64)
    # blocks: ancestors of each join, joins by (W^anc, id), less the earlier blocks
    joins = sorted((u for u in range(V) if indeg[u] >= 2), key=lambda u: (wanc[u], u))
    block = np.full(V, len(joins))
    for b in reversed(range(len(joins))):
        block[reach[joins[b]]] = b
    block = block.tolist()
    rank = {u: i for i, u in enumerate(sorted(range(V), key=lambda u: (-wanc[u], u)))}
    heads = [[] for _ in range(len(joins) + 1)]
    for u in range(V):
        if not any(block[p] == block[u] for p in pred[u]):
            heads[block[u]].append(u)
    groups = []
    for b, hs in enumerate(heads):
        while hs:
            top = sorted(hs, key=rank.get)[:M]
            big = [u for u in top if x[u] >= M]
            if big:
                top = [max(big, key=lambda u: (x[u], -rank[u]))]
            groups.append(sorted(top))
            gone = set(top)
            hs = [u for u in hs if u not in gone] + [t for u in top for t in succ[u] if block[t] == b]
    # Alg.2 with SMs taken by each parallel launch and one segmentation per group
    rem, m, done, left = list(x), [0] * V, [False] * V, indeg[:]
    ready = [rank[u] for u in range(V) if not indeg[u]]
    heapq.heapify(ready)
    node = sorted(range(V), key=rank.get)
    for g in groups:
        live = [u for u in g if not done[u]]
        if not live:
            continue
        tot = sum(rem[u] for u in live)
        for u in live:
            m[u] = min(rem[u], max(1, (2 * rem[u] * M + tot) // (2 * tot)))
        S = M - sum(m[u] for u in live)
        while S < 0:
            u = max(live, key=lambda u: (m[u], u))
            m[u] -= 1
            S += 1
        R = max(_time(rem[u], k[u], m[u], M) for u in live)
        mine, back, fin = set(live), [], live
        while S > 0 and ready:
            u = node[heapq.heappop(ready)]
            if done[u] or u in mine:
                if not done[u]:
                    back.append(rank[u])
                continue
            mu = min(rem[u], S)
            if _time(rem[u], k[u], mu, M) > R:  # segmentation: the largest part that fits
                lo, hi = 1, rem[u] - 1
                while lo < hi:
                    mid = (lo + hi + 1) // 2
                    if _time(mid, k[u], min(mid, S), M) <= R:
                        lo = mid
                    else:
                        hi = mid - 1
                rem[u] -= lo
                back.append(rank[u])
                break
            m[u] = mu
            S -= mu
            fin = fin + [u]
        for r in back:
            heapq.heappush(ready, r)
        for u in fin:
            done[u] = True
            for t in succ[u]:
                left[t] -= 1
                if not left[t]:
                    heapq.heappush(ready, rank[t])
    return level, wanc, m


def _features(g, M):
    off, eoff = g["node_off"].tolist(), g["edge_off"].tolist()
    rp, col, x, k = (g[n].tolist() for n in ("row_ptr", "col", "wcet", "k64"))
    rows = []
    for d in range(len(off) - 1):
        a, V = off[d], off[d + 1] - off[d]
        r = rp[a + d:a + d + V + 1]
        succ = [col[eoff[d] + r[u]:eoff[d] + r[u + 1]] for u in range(V)]
        level, wanc, m = _schedule(succ, x[a:a + V], k[a:a + V], M)
        depth, tot = max(level), float(sum(x[a:a + V]))
        rows += [[level[u] / depth if depth else 0.0, wanc[u] / tot, math.log2(max(m[u], 1)) / 12] for u in range(V)]
    return torch.tensor(rows, dtype=torch.float64, device="cuda")


def _network(case, seed):
    """Features, edges and parameters (as leaves) of the network in 64 bits."""
    g, _ = _graphs(case, seed)
    dev, N, n = g["wcet"].device, len(g["wcet"]), case["n_dags"]
    dag = torch.repeat_interleave(torch.arange(n, device=dev), g["node_off"].diff())
    entry_dag = torch.repeat_interleave(torch.arange(n, device=dev), g["node_off"].diff() + 1)
    deg = g["row_ptr"].long().diff()[entry_dag[1:] == entry_dag[:-1]]
    src = torch.repeat_interleave(torch.arange(N, device=dev), deg)
    dst = g["col"].long() + g["node_off"][dag[src]]
    s = _features(g, case["M"])
    indeg = torch.bincount(dst, minlength=N).double()
    f = torch.zeros(N, FEAT, dtype=torch.float64, device=dev)
    f[:, 0] = torch.log2(g["wcet"].double()) / 32
    f[:, 1] = g["k64"].double() / 64
    f[:, 2] = torch.log2(1 + indeg) / 8
    f[:, 3] = torch.log2(1 + deg.double()) / 8
    f[:, 4:7] = s
    f[:, 7] = 1
    p = torch.from_numpy(_params(seed)).to(dev).double().requires_grad_()
    return g, f, src, dst, indeg.clamp(min=1)[:, None], deg.double().clamp(min=1)[:, None], p


def _logits(f, src, dst, indeg, outdeg, p, n_levels):
    h, at = f, 0
    for width in (FEAT, HIDDEN, HIDDEN):
        W = p[at:at + 3 * width * HIDDEN].view(3 * width, HIDDEN)
        at += 3 * width * HIDDEN
        mp = torch.zeros_like(h).index_add(0, dst, h[src]) / indeg
        ms = torch.zeros_like(h).index_add(0, src, h[dst]) / outdeg
        h = torch.relu(torch.cat([h, mp, ms], 1) @ W + p[at:at + HIDDEN])
        at += HIDDEN
    W = p[at:at + HIDDEN * MAX_LEVELS].view(HIDDEN, MAX_LEVELS)
    return h @ W[:, :n_levels] + p[at + HIDDEN * MAX_LEVELS:][:n_levels]


def exact(case, seed):
    """The network's outputs in 64 bits; the library's other outputs are whole numbers."""
    if case["kind"] not in ("logits", "propose", "train") or case["n_dags"] * _mean_size(case)[0] > 2e5:
        return None
    g, f, src, dst, indeg, outdeg, p = _network(case, seed)
    z = _logits(f, src, dst, indeg, outdeg, p, case["n_levels"])
    if case["kind"] == "logits":
        return z.detach().reshape(-1)
    if case["kind"] == "propose":
        return {"logits": z.detach().reshape(-1), **{k: None for k in ("out_bound", "best_bound", "best_cand", "best_m")}}
    loss = torch.nn.functional.cross_entropy(z, _labels(g, case["n_levels"]).long())
    (d,) = torch.autograd.grad(loss, p)
    # Adam's first step: bias-corrected moments are the gradient and its square
    return {"loss": float(loss.detach()), "params": (p - LR * d / (d.abs() + 1e-8)).detach()}
