"""Performance cases: what a user of this library has it do, timed as whole calls.

A case is a dict of plain values.  `prepare` makes what the user's program has
in hand before the call (graphs as CSR arrays on the host or on the device, a
captured handle, a network with a kept training batch), `run` is one pass
through the public entry points with its whole results, `work` what the pass
cannot do without, and `exact` the 64-bit value of the results that are
computed numbers (path lists are whole numbers and have none).

Graphs are the repository's own: diamond chains, the two structured CFGs, the
batch distribution (10-150 vertices) and looped chains for wide bitsets.  The
seed numbers the vertices of a single graph anew, as a front end numbers basic
blocks when it reaches them (looped chains: it places the loops), and shuffles
the graphs of a batch.  Volumes therefore depend on the case alone.
"""
from __future__ import annotations

import functools
import random

import numpy as np
import torch

from paper_2210_16998_gb300 import cfggen, tpg

# Prime paths, their vertices, test paths and their vertices of the batch
# distribution's graphs, 256 graphs to a row (graph i uses BATCH_SEED0 + i).
BLOCK = 256
VOLUMES = (
    (472518, 13362379, 451544, 14815664), (554064, 16070535, 488782, 17588607),
    (4106939, 158051040, 2896644, 167662927), (428680, 11432389, 403781, 13140984),
    (366354, 10387014, 355005, 11481260), (232132, 5905131, 211706, 6623644),
    (289935, 7513379, 257048, 8085174), (552729, 15306923, 436901, 17872903),
    (445771, 12016940, 426377, 13262939), (1139023, 38470677, 814526, 37598875),
    (540680, 14773172, 493442, 16648474), (521056, 14677673, 502525, 16063679),
    (312336, 7987470, 289849, 9035614), (1852861, 66191249, 1180673, 58709615),
    (1240598, 39153489, 1160952, 46974592), (404517, 11476315, 394255, 12775986),
)
BATCH_VERTICES, BATCH_ARCS = 41, 54  # mean per graph of the batch distribution


def listed():
    return [
        # one plain method at a time: the smallest call, launches and latency
        {"name": "method24", "kind": "graph", "family": "structured24", "size": 24, "pad": 0, "on": "device", "call": "paths"},
        # a small method with the binding's defaults: host arrays in, host results out
        {"name": "chain10_host", "kind": "graph", "family": "chain", "size": 10, "pad": 0, "on": "host", "call": "paths"},
        # an ordinary branchy method: 65,536 paths
        {"name": "chain16", "kind": "graph", "family": "chain", "size": 16, "pad": 0, "on": "device", "call": "paths"},
        # the benchmark's graph, the largest single method: 4,194,304 paths of 45 vertices
        {"name": "chain22", "kind": "graph", "family": "chain", "size": 22, "pad": 0, "on": "device", "call": "paths"},
        # a loop-heavy method whose test paths need merging and deduplication
        {"name": "loops120", "kind": "graph", "family": "structured120", "size": 120, "pad": 0, "on": "device",
         "call": "paths"},
        # the same with results read by a host program
        {"name": "loops120_host", "kind": "graph", "family": "structured120", "size": 120, "pad": 0, "on": "host",
         "call": "paths"},
        # a long generated function: bitsets of 64 words, hundreds of levels, few paths
        {"name": "long1100", "kind": "graph", "family": "looped", "size": 1100, "pad": 0, "on": "device", "call": "paths"},
        # a module: a ragged number of methods in one handle
        {"name": "batch333", "kind": "batch", "first": 1024, "count": 333, "on": "device", "call": "paths"},
        # the smaller, longest-first test-path set of a module
        {"name": "greedy333", "kind": "batch", "first": 1024, "count": 333, "on": "device", "call": "greedy"},
        # a code base: the 4096-graph batch, loaded and enumerated in one pass
        {"name": "batch4096", "kind": "batch", "first": 0, "count": 4096, "on": "device", "call": "paths"},
        # a captured batch replayed, as a service that re-enumerates one module does
        {"name": "replay1024", "kind": "batch", "first": 1024, "count": 1024, "on": "device", "call": "replay"},
        # a training step of the learned sizer and its prediction for a batch
        {"name": "sizer256", "kind": "sizer", "first": 0, "count": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    what = rng.choice(["chain", "chain", "loops", "looped", "batch", "batch", "greedy", "replay", "sizer"])
    on = rng.choice(["device", "device", "host"])
    if what in ("chain", "loops"):
        family, size = ("chain", rng.randint(4, 21)) if what == "chain" else rng.choice(
            [("structured24", 24), ("structured120", 120)])
        return {"kind": "graph", "family": family, "size": size, "pad": rng.randint(1, 24), "on": on, "call": "paths"}
    if what == "looped":
        return {"kind": "graph", "family": "looped", "size": _log_int(rng, 300, 1500), "pad": 0, "on": on,
                "call": "paths"}
    if what == "sizer":
        return {"kind": "sizer", "first": rng.randint(0, 4096), "count": _log_int(rng, 32, 512)}
    count = _log_int(rng, 16, {"batch": 2048, "greedy": 512, "replay": 1024}[what])
    first = rng.randint(0, len(VOLUMES) * BLOCK - count)
    return {"kind": "batch", "first": first, "count": count, "on": on if what == "batch" else "device",
            "call": "paths" if what == "batch" else what}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _looped_chain(n, rng):
    """0 -> 1 -> ... -> n-1 with a loop of six vertices in every ten, at a drawn place."""
    ends = [i + rng.randrange(5) for i in range(10, n - 5, 10)]
    rp, col = cfggen.csr_from_arcs(n, [(i, i + 1) for i in range(n - 1)] + [(e, e - 5) for e in ends])
    return cfggen.CFG(n, rp, col, 0, n - 1, f"looped-chain-{n}")


@functools.lru_cache(maxsize=None)
def _graph(family, size):
    if family == "chain":
        return cfggen.diamond_chain(size)
    if family == "structured24":
        return cfggen.config1_cfg()
    return cfggen.config3_cfg()


@functools.lru_cache(maxsize=None)
def _batch_graph(i):
    return cfggen.random_cfg(cfggen.BATCH_SEED0 + i)


@functools.lru_cache(maxsize=None)
def _sizer_graph(i):
    return cfggen.random_cfg(cfggen.TRAIN_SEED0 + i, n_max=64)


def _renumber(cfg, rng):
    """The same graph with its vertices numbered as a worklist that starts at
    the entry and is taken from at drawn places reaches them."""
    rp, col = cfg.row_ptr.tolist(), cfg.col.tolist()
    succ = [col[rp[v]:rp[v + 1]] for v in range(cfg.n)]
    new, order, work_list = {cfg.entry: -1}, [], [cfg.entry]
    while work_list:
        at = rng.randrange(len(work_list))
        work_list[at], work_list[-1] = work_list[-1], work_list[at]
        v = work_list.pop()
        new[v] = len(order)
        order.append(v)
        for w in succ[v]:
            if w not in new:
                new[w] = -1
                work_list.append(w)
    rows = [sorted(new[w] for w in succ[v]) for v in order]
    row_ptr = np.zeros(cfg.n + 1, np.int32)
    np.cumsum([len(r) for r in rows], out=row_ptr[1:])
    flat = np.asarray([w for r in rows for w in r], np.int32)
    return cfggen.CFG(cfg.n, row_ptr, flat, new[cfg.entry], new[cfg.exit], cfg.name)


def _padded(cfg, pad):
    """cfg behind `pad` straight-line blocks."""
    if not pad:
        return cfg
    head = np.arange(pad, dtype=np.int32)
    row_ptr = np.concatenate([head, cfg.row_ptr + pad]).astype(np.int32)
    col = np.concatenate([head[1:], [cfg.entry + pad], cfg.col + pad]).astype(np.int32)
    return cfggen.CFG(cfg.n + pad, row_ptr, col, 0, cfg.exit + pad, cfg.name)


def _cfgs(case, seed):
    rng = random.Random(seed)
    if case["kind"] == "graph":
        if case["family"] == "looped":
            return [_looped_chain(case["size"], rng)]
        return [_renumber(_padded(_graph(case["family"], case["size"]), case["pad"]), rng)]
    make = _batch_graph if case["kind"] == "batch" else _sizer_graph
    cfgs = [make(i) for i in range(case["first"], case["first"] + case["count"])]
    rng.shuffle(cfgs)
    return cfgs


def _parameters(seed):
    """Network weights as the library draws them: He-uniform, small random biases."""
    g = np.random.default_rng(seed)
    u = lambda n, bound: g.uniform(-bound, bound, n)  # noqa: E731
    parts = [u(64 * 8, (6 / 8) ** 0.5), u(64, 0.1)]
    for _ in range(3):
        parts += [u(64 * 192, (6 / 192) ** 0.5), u(64, 0.1)]
    parts += [u(3 * 64, (3 / 64) ** 0.5), u(3, 0.1)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    tpg.load_library()
    cfgs = _cfgs(case, seed)
    state = {"case": case, "held": ()}
    if case["kind"] == "graph":
        c = cfgs[0]
        state["cfg"] = c
        if case["on"] == "device":
            state["row_ptr"] = torch.as_tensor(c.row_ptr, device="cuda")
            state["col"] = torch.as_tensor(c.col, device="cuda")
        return state
    state["arrays"] = cfggen.concat_batch(cfgs)
    if case["kind"] == "sizer":
        state["num_vertices"] = int(state["arrays"][0].sum())
        state["handle"] = tpg.tpg_load_cfg_batch(*state["arrays"])
        state["sizer"] = tpg.tpg_sizer_create(0)
        tpg.tpg_sizer_set_params(state["sizer"], _parameters(seed))
        tpg.tpg_sizer_add_batch(state["sizer"], state["handle"])
    elif case["call"] == "replay":
        state["handle"] = tpg.tpg_load_cfg_batch(*state["arrays"], location=tpg.TPG_RESULT_DEVICE)
        tpg.tpg_graph_capture(state["handle"])
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _load(state):
    case = state["case"]
    where = tpg.TPG_RESULT_DEVICE if case["on"] == "device" else tpg.TPG_RESULT_HOST
    if case["kind"] == "batch":
        return tpg.tpg_load_cfg_batch(*state["arrays"], location=where)
    c = state["cfg"]
    if case["on"] == "device":
        return tpg.tpg_load_cfg_device(c.n, c.m, state["row_ptr"], state["col"], c.entry, c.exit)
    return tpg.tpg_load_cfg(c.n, c.row_ptr, c.col, c.entry, c.exit)


def run(state):
    for p in state["held"]:  # the last pass's results have been used
        p.free()
    state["held"] = ()
    case = state["case"]
    if case["kind"] == "sizer":
        loss, grad = tpg.tpg_sizer_loss_grad(state["sizer"], 0)
        pred, totals = tpg.tpg_sizer_predict(state["sizer"], state["handle"], state["num_vertices"])
        return [loss, grad, pred, totals]
    if case["call"] == "replay":
        held = tpg.tpg_graph_launch(state["handle"])
    else:
        h = _load(state)
        pp = tpg.tpg_prime_paths(h)
        held = (pp, tpg.tpg_test_paths_greedy(h) if case["call"] == "greedy" else tpg.tpg_test_paths(h))
        h.close()
    state["held"] = held
    return [a for p in held for a in (p.graph_path_ptr, p.offsets, p.vertices)]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _volumes(first, count):
    """(PPs, PP vertices, TPs, TP vertices) of batch graphs first .. first+count-1."""
    tot = [0.0] * 4
    for b, row in enumerate(VOLUMES):
        share = max(0, min(first + count, (b + 1) * BLOCK) - max(first, b * BLOCK)) / BLOCK
        tot = [t + share * r for t, r in zip(tot, row)]
    return [int(t) for t in tot]


def work(case):
    if case["kind"] == "sizer":
        n, m, params = 25 * case["count"], 32 * case["count"], 37827
        macs = n * (8 * 64 + 3 * 192 * 64 + 64 * 3)
        # features, labels and CSR read twice (step and prediction), weights, gradient, predictions
        return {"bytes": 2 * 4 * (8 * n + n + m) + 12 * n + 3 * 4 * params + 12 * n, "flops": 8 * macs}
    if case["kind"] == "batch":
        n, m, graphs = BATCH_VERTICES * case["count"], BATCH_ARCS * case["count"], case["count"]
        pps, ppv, tps, tpv = _volumes(case["first"], case["count"])
    elif case["family"] == "looped":
        n, graphs = case["size"], 1
        loops = (n - 6) // 10
        m = n - 1 + loops
        pps, ppv, tps, tpv = 6 * loops + 1, 52 * loops, loops + 1, (loops + 1) * (n + 6)
    else:
        pad, graphs = case["pad"], 1
        if case["family"] == "chain":
            k = case["size"]
            n, m, pps, ppv = 3 * k + 1, 4 * k, 2 ** k, (2 * k + 1) * 2 ** k
            tps = tpv = 0  # every test path is its prime path: one list serves both
            from_entry = pps
        elif case["family"] == "structured24":
            n, m, pps, ppv, tps, tpv, from_entry = 24, 29, 76, 730, 45, 856, 20
        else:
            n, m, pps, ppv, tps, tpv, from_entry = 120, 164, 1086398, 42668919, 944136, 56283823, 6415
        n, m, ppv, tpv = n + pad, m + pad, ppv + pad * from_entry, tpv + pad * tps
    lists = 8 * (pps + tps) + 4 * (ppv + tpv) + 2 * 8 * (graphs + 1)
    return {"bytes": 4 * (n + 1 + m) + lists, "flops": 0}


# ---------------------------------------------------------------------------
# 64-bit values of computed numbers
# ---------------------------------------------------------------------------
def _root_counts(c):
    """Per first vertex of one graph of at most 64 vertices: simple paths,
    prime paths, prime-path vertices (level-synchronous, visited sets as words)."""
    one = np.uint64(1)
    bit = one << np.arange(c.n, dtype=np.uint64)
    src = np.repeat(np.arange(c.n), np.diff(c.row_ptr))
    preds = np.zeros(c.n, np.uint64)
    np.bitwise_or.at(preds, c.col, bit[src])
    deg = np.diff(c.row_ptr)
    out = np.zeros((c.n, 3), np.int64)
    first = last = np.arange(c.n)
    seen = bit.copy()
    length = 1
    while len(first):
        closed = (first == last) if length > 1 else np.zeros(len(first), bool)
        d = np.where(closed, 0, deg[last])
        parent = np.repeat(np.arange(len(first)), d)
        arc = np.arange(len(parent)) - np.repeat(np.cumsum(d) - d, d) + c.row_ptr[last][parent]
        w = c.col[arc]
        ok = (w == first[parent]) | ((seen[parent] & bit[w]) == 0)
        parent, w = parent[ok], w[ok]
        grows = np.bincount(parent, minlength=len(first)) > 0
        prime = closed | (~grows & ((preds[first] & ~seen) == 0) & ((preds[first] & bit[last]) == 0))
        out[:, 0] += np.bincount(first, minlength=c.n)
        out[:, 1] += np.bincount(first[prime], minlength=c.n)
        out[:, 2] += length * np.bincount(first[prime], minlength=c.n)
        first, last, seen = first[parent], w, seen[parent] | bit[w]
        length += 1
    return out


def _features(c):
    n = c.n
    adj = np.zeros((n, n), bool)
    adj[np.repeat(np.arange(n), np.diff(c.row_ptr)), c.col] = True
    dist = np.where(np.eye(n, dtype=bool), 0, -1)
    reach, d = np.eye(n, dtype=bool), 0
    while True:
        nxt = (reach.astype(np.float32) @ adj.astype(np.float32)) > 0
        new = nxt & (dist < 0)
        if not new.any():
            break
        d += 1
        dist[new] = d
        reach = new
    scc = ((dist >= 0) & (dist.T >= 0)).sum(1)
    depth = lambda x: np.where(x >= 0, x / n, 2.0)  # noqa: E731
    ids = np.arange(n)
    return np.stack([np.log1p(adj.sum(0)), np.log1p(adj.sum(1)), ids == c.entry, ids == c.exit, np.log1p(scc),
                     depth(dist[c.entry]), depth(dist[:, c.exit]), np.full(n, np.log(n) / 5)], 1).astype(np.float64)


def exact(case, seed):
    if case["kind"] != "sizer":
        return None
    cfgs = _cfgs(case, seed)
    x = torch.as_tensor(np.concatenate([_features(c) for c in cfgs]))
    t = torch.as_tensor(np.log1p(np.concatenate([_root_counts(c) for c in cfgs]).astype(np.float64)))
    base = np.cumsum([0] + [c.n for c in cfgs])
    u = torch.as_tensor(np.concatenate([b + np.repeat(np.arange(c.n), np.diff(c.row_ptr)) for b, c in zip(base, cfgs)]))
    w = torch.as_tensor(np.concatenate([b + c.col.astype(np.int64) for b, c in zip(base, cfgs)]))
    p = torch.as_tensor(_parameters(seed).astype(np.float64)).requires_grad_(True)
    at = 0

    def take(*shape):
        nonlocal at
        n = int(np.prod(shape))
        at += n
        return p[at - n:at].reshape(shape)

    w0, b0 = take(64, 8), take(64)
    h = torch.relu(x @ w0.T + b0)
    for _ in range(3):
        wl, bl = take(64, 192), take(64)
        from_pred = torch.zeros_like(h).index_add(0, w, h[u])
        from_succ = torch.zeros_like(h).index_add(0, u, h[w])
        h = torch.relu(torch.cat([h, from_pred, from_succ], 1) @ wl.T + bl)
    wo, bo = take(3, 64), take(3)
    y = h @ wo.T + bo
    loss = ((y - t) ** 2).mean()
    loss.backward()
    totals = torch.expm1(torch.relu(y.detach())).sum(0)
    return [float(loss.detach()), p.grad.numpy(), y.detach().numpy(), totals.numpy()]
