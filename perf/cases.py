"""What is measured of the library's speed: its public calls over the sizes
its workloads have (include/cupc.h, bench.py).

A case is a dict of plain values. `prepare` makes what a program has in hand
before the call: a graph whose sketches are resident on the device, the edges
and pairs of the next request, a batcher, a server or a cutset. `run` makes
one pass of that program. An update pass inserts its batch of absent edges or,
the next time, deletes them again, so that the stream stays valid however
often it runs.

Outputs: the sketches after the pass (the library keeps them at the start of
the workspace the caller lends to cupc_init, in the layout of
cupc_export_sketches, so they are returned as a view of it), and the answers,
labels or forest of the query calls. Every output is a whole number, so none
has a value in 64-bit floating point to be compared with (`exact` is None).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_14433_gb300 import autotune as AT
from paper_2509_14433_gb300 import cupc as C
from paper_2509_14433_gb300 import workloads as WL

RMAT = AT.RMAT_PROBS
CLIQUES_V = 131072


def listed():
    return [
        # one small request of a client that cannot wait for more updates (the
        # bottom of the batch-size range the bench sweeps): launches and latency
        {"name": "update_v1024_n64", "kind": "update", "V": 1024, "n": 64, "dist": "uniform"},
        # the smallest batches of the R-MAT stream, on its graph of 9.5 GB
        {"name": "update_rmat_n1000", "kind": "update", "V": 131072, "n": 1000, "dist": "rmat"},
        # an ordinary batch on a graph of no special size (odd V and n)
        {"name": "update_v5003_n30011", "kind": "update", "V": 5003, "n": 30011, "dist": "uniform"},
        # the dense workload's batches
        {"name": "update_v16384_n1m", "kind": "update", "V": 16384, "n": 1 << 20, "dist": "uniform"},
        # the headline's launches: joined R-MAT batches of 4M edges
        {"name": "update_rmat_n4m", "kind": "update", "V": 131072, "n": 1 << 22, "dist": "rmat"},
        # the plain stream: 10k toggles of a G(1024, 1/2), then 1k Connected pairs
        {"name": "query_v1024", "kind": "query", "V": 1024, "base": 261888, "n": 10000, "ask": "query", "pairs": 1000},
        # the dense graph's spanning forest after a small update
        {"name": "forest_v16384", "kind": "query", "V": 16384, "base": 1 << 23, "n": 1024, "ask": "forest", "pairs": 0},
        # many components: 256 cliques joined and split by 64k bridges, 1k pairs each time
        {"name": "query_cliques", "kind": "cliques", "size": 512, "n": 65536, "pairs": 1000},
        # many independent graphs in one launch sequence
        {"name": "batch_64x1000", "kind": "batch", "graphs": 64, "V": 1024, "V_hi": 8192, "n": 1000},
        # the paper's fixed-forest stream: a burst of non-tree updates and rho/9
        # pairs with labels kept incrementally
        {"name": "incremental_v8192", "kind": "incremental", "V": 8192, "base": 1 << 21, "n": 1501, "pairs": 167,
         "tree": False},
        # the serving loop: every graph gets an update and a query, from host memory
        {"name": "serve_16", "kind": "serve", "graphs": 16, "V": 1024, "V_hi": 32768, "n": 1000, "n_hi": 30000,
         "pairs": 1000},
        # the parallel cutset: a batch of cuts (or links) and the replacement-edge
        # queries of the split trees
        {"name": "cutset_v1024", "kind": "cutset", "V": 1024, "base": 32768, "n": 64, "asks": 4},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["update"] * 5 + ["query"] * 3 + ["cliques", "batch", "incremental", "serve", "cutset"])
    if kind == "update":
        if rng.random() < 0.4:
            V = 1 << rng.randint(10, 17)
            return {"kind": kind, "V": V, "n": min(_log(rng, 64, 1 << 22), V * V // 32), "dist": "rmat"}
        V = _log(rng, 1024, 131072)
        return {"kind": kind, "V": V, "n": min(_log(rng, 64, 1 << 21), V * V // 32), "dist": "uniform"}
    if kind == "query":
        V = _log(rng, 1024, 131072)
        ask = rng.choice(["query", "query", "labels", "forest"])
        return {"kind": kind, "V": V, "base": int(V * 2 ** rng.uniform(0.0, 6.0)), "n": _log(rng, 16, 30000),
                "ask": ask, "pairs": _log(rng, 100, 100000) if ask == "query" else 0}
    if kind == "cliques":
        return {"kind": kind, "size": rng.choice([64, 128, 256, 512]), "n": _log(rng, 64, 65536),
                "pairs": _log(rng, 100, 10000)}
    if kind == "batch":
        V = _log(rng, 512, 4096)
        return {"kind": kind, "graphs": rng.randint(4, 64), "V": V, "V_hi": _log(rng, V, 8192), "n": _log(rng, 100, 4000)}
    if kind == "incremental":
        V = _log(rng, 1024, 16384)
        return {"kind": kind, "V": V, "base": V * rng.randint(8, 64), "n": _log(rng, 100, 4000),
                "pairs": _log(rng, 20, 500), "tree": rng.random() < 0.5}
    if kind == "serve":
        V, n = _log(rng, 1024, 4096), _log(rng, 200, 2000)
        return {"kind": kind, "graphs": rng.randint(3, 16), "V": V, "V_hi": _log(rng, V, 32768), "n": n,
                "n_hi": _log(rng, n, 30000), "pairs": _log(rng, 100, 1000)}
    V = _log(rng, 256, 2048)
    return {"kind": kind, "V": V, "base": V * rng.randint(2, 32), "n": _log(rng, 8, V // 4), "asks": rng.randint(1, 8)}


# ---- what a program holds


class Graph:
    """A graph in a workspace lent by torch."""

    def __init__(self, V, seed, max_batch, ws=None):
        params = (0, 0, 0, max_batch)
        self.V = V
        self.ws = torch.empty(C.cupc_workspace_bytes(V, params), dtype=torch.uint8, device="cuda") if ws is None else ws
        st, self.h = C.cupc_init(V, seed, params, self.ws, None)
        C.check(st, "cupc_init")
        p = np.zeros(4, np.uint32)
        C.check(C.cupc_get_params(self.h, p))
        self.L, _, _, self.W = (int(x) for x in p)
        AT.apply_buckets(self.h, V)
        self.sketches = self.ws[:self.L * V * self.W * 16].view(torch.int64)

    def __del__(self):
        if getattr(self, "h", None):
            C.cupc_destroy(self.h)
            self.h = None


class Owned:
    """A handle and the call that gives it back."""

    def __init__(self, h, destroy, keep=()):
        self.h, self.destroy, self.keep = h, destroy, keep

    def __del__(self):
        self.destroy(self.h)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _pair_ids(V, count, gen, dist):
    """`count` distinct edge ids u*V+v (u < v) in a random order."""
    if dist == "uniform" and count * 8 > V * V:
        x = torch.randperm(V * V, generator=gen, device="cuda")
        return x[x // V < x % V][:count]
    have = torch.empty(0, dtype=torch.int64, device="cuda")
    while have.numel() < count:
        m = min(1 << 24, (count - have.numel()) * 3 // 2 + 1024)
        if dist == "rmat":
            u, v = WL.rmat_pairs(m, V.bit_length() - 1, RMAT, gen, "cuda")
        else:
            u = torch.randint(0, V, (m,), generator=gen, device="cuda")
            v = torch.randint(0, V, (m,), generator=gen, device="cuda")
        ok = u != v
        have = torch.unique(torch.cat([have, torch.minimum(u, v)[ok] * V + torch.maximum(u, v)[ok]]))
    return have[torch.randperm(have.numel(), generator=gen, device="cuda")[:count]]


def _edges(ids, V):
    return torch.stack([ids // V, ids % V], 1).to(torch.int32).reshape(-1).contiguous()


def _ops(n):
    return [torch.full((n,), s, dtype=torch.int8, device="cuda") for s in (1, -1)]


def _pairs(V, m, gen):
    return torch.randint(0, V, (2 * m,), generator=gen, device="cuda").to(torch.int32)


def _insert(g, ids):
    if ids.numel():
        C.check(C.cupc_update_batch(g.h, _edges(ids, g.V), _ops(ids.numel())[0], ids.numel(), None))
        torch.cuda.synchronize()


def _spread(lo, hi, k):
    """k sizes from lo to hi, evenly spread over their logarithm."""
    return [int(round(lo * (hi / lo) ** (i / max(1, k - 1)))) for i in range(k)]


def _turn(s):
    s["turn"] ^= 1
    return s["turn"] ^ 1


def prepare(case, seed):
    return {"update": _prepare_update, "query": _prepare_query, "cliques": _prepare_cliques, "batch": _prepare_batch,
            "incremental": _prepare_incremental, "serve": _prepare_serve, "cutset": _prepare_cutset}[case["kind"]](
                case, seed, _generator(seed))


def run(state):
    return state["run"](state)


def exact(case, seed):
    return None


# ---- update batches


def _prepare_update(c, seed, gen):
    V, n = c["V"], c["n"]
    base = min(1 << 20, 2 * V)  # edges already in the graph
    ids = _pair_ids(V, base + n, gen, c["dist"])
    g = Graph(V, seed, max(n, 1 << 20))
    _insert(g, ids[:base])
    return {"run": _run_update, "g": g, "e": _edges(ids[base:], V), "o": _ops(n), "n": n, "turn": 0}


def _run_update(s):
    g = s["g"]
    C.check(C.cupc_update_batch(g.h, s["e"], s["o"][_turn(s)], s["n"], None))
    return g.sketches


# ---- an update, then a query call that recovers the components


def _prepare_query(c, seed, gen):
    V, n = c["V"], c["n"]
    ids = _pair_ids(V, c["base"] + n, gen, "uniform")
    g = Graph(V, seed, 1 << 20)
    _insert(g, ids[:c["base"]])
    return {"run": _run_query, "g": g, "e": _edges(ids[c["base"]:], V), "o": _ops(n), "n": n, "turn": 0,
            "ask": c["ask"], "m": c["pairs"], "pairs": _pairs(V, max(1, c["pairs"]), gen),
            "answers": torch.zeros(max(1, c["pairs"]), dtype=torch.uint8, device="cuda"),
            "labels": torch.zeros(V, dtype=torch.int32, device="cuda"),
            "forest": torch.zeros(V, dtype=torch.int64, device="cuda")}


def _prepare_cliques(c, seed, gen):
    V, size, n = CLIQUES_V, c["size"], c["n"]
    perm = torch.randperm(V, generator=gen, device="cuda").view(V // size, size)
    i, j = torch.triu_indices(size, size, 1, device="cuda")
    u, v = perm[:, i].reshape(-1), perm[:, j].reshape(-1)
    g = Graph(V, seed, 1 << 20)
    _insert(g, torch.minimum(u, v) * V + torch.maximum(u, v))
    clique = torch.empty(V, dtype=torch.int64, device="cuda")
    clique[perm.reshape(-1)] = torch.arange(V, device="cuda") // size
    ids = _pair_ids(V, 2 * n + 1024, gen, "uniform")
    ids = ids[clique[ids // V] != clique[ids % V]][:n]
    return {"run": _run_query, "g": g, "e": _edges(ids, V), "o": _ops(n), "n": ids.numel(), "turn": 0,
            "ask": "query", "m": c["pairs"], "pairs": _pairs(V, c["pairs"], gen),
            "answers": torch.zeros(c["pairs"], dtype=torch.uint8, device="cuda")}


def _run_query(s):
    g = s["g"]
    C.check(C.cupc_update_batch(g.h, s["e"], s["o"][_turn(s)], s["n"], None))
    if s["ask"] == "query":
        C.check(C.cupc_query(g.h, s["pairs"], s["m"], s["answers"], None))
        return s["answers"], g.sketches
    if s["ask"] == "labels":
        C.check(C.cupc_labels(g.h, s["labels"], None))
        return s["labels"], g.sketches
    st, k = C.cupc_spanning_forest(g.h, s["forest"], g.V, None)
    C.check(st, "cupc_spanning_forest", ok=(C.CUPC_OK, C.CUPC_EINCOMPLETE))
    return s["forest"][:k], g.sketches


# ---- one batch for each of many graphs


def _prepare_batch(c, seed, gen):
    k, n = c["graphs"], c["n"]
    sizes = _spread(c["V"], c["V_hi"], k)
    params = (0, 0, 0, 1 << 16)
    per = [C.cupc_workspace_bytes(V, params) for V in sizes]
    at = np.concatenate([[0], np.cumsum([(b + 255) // 256 * 256 for b in per])]).tolist()
    arena = torch.zeros(at[-1], dtype=torch.uint8, device="cuda")  # every graph's workspace in one allocation
    gs = [Graph(V, seed + i, 1 << 16, arena[at[i]:at[i] + per[i]]) for i, V in enumerate(sizes)]
    e = []
    for g in gs:
        ids = _pair_ids(g.V, 2 * g.V + n, gen, "uniform")
        _insert(g, ids[:2 * g.V])
        e.append(_edges(ids[2 * g.V:], g.V))
    st, b = C.cupc_batcher_create(k, True)
    C.check(st, "cupc_batcher_create")
    return {"run": _run_batch, "b": Owned(b, C.cupc_batcher_destroy), "gs": gs, "hs": [g.h for g in gs], "e": e,
            "o": [[o] * k for o in _ops(n)], "n": [n] * k, "turn": 0}


def _run_batch(s):
    C.check(C.cupc_batcher_update(s["b"].h, s["hs"], s["e"], s["o"][_turn(s)], s["n"], None))
    return [g.sketches for g in s["gs"]][:: max(1, len(s["gs"]) // 16)]  # every fourth graph of 64


# ---- incremental labels


def _prepare_incremental(c, seed, gen):
    V, n = c["V"], c["n"]
    ids = _pair_ids(V, c["base"] + n, gen, "uniform")
    g = Graph(V, seed, 1 << 20)
    C.check(C.cupc_set_incremental(g.h, 1, None))
    _insert(g, ids[:c["base"]])
    answers = torch.zeros(c["pairs"], dtype=torch.uint8, device="cuda")
    pairs = _pairs(V, c["pairs"], gen)
    C.check(C.cupc_query(g.h, pairs, c["pairs"], answers, None))  # the stream's labels so far
    ops = _ops(n)
    # "tree": bursts over edges of the graph itself, so that deletes hit its
    # spanning forest; else edges outside it, inserted and deleted again
    burst = ids[:n] if c["tree"] else ids[c["base"]:]
    return {"run": _run_query, "g": g, "e": _edges(burst, V), "o": ops[::-1] if c["tree"] else ops, "n": burst.numel(),
            "turn": 0, "ask": "query", "m": c["pairs"], "pairs": pairs, "answers": answers}


# ---- the serving loop


def _prepare_serve(c, seed, gen):
    k, m = c["graphs"], c["pairs"]
    sizes, counts = _spread(c["V"], c["V_hi"], k), _spread(c["n"], c["n_hi"], k)
    cap = 1 << 17
    mem = sum(C.cupc_workspace_bytes(V, (0, 0, 0, cap)) + 512 for V in sizes)
    st, srv = C.cupc_server_create(mem, k, cap, 4, 64 << 20)
    C.check(st, "cupc_server_create")
    owner = Owned(srv, C.cupc_server_destroy)
    reqs, waits = [], []
    for i, V in enumerate(sizes):
        n = counts[(5 * i) % k]  # big and small batches on big and small graphs
        st, gid = C.cupc_server_open(srv, V, seed + i)
        C.check(st, "cupc_server_open")
        ids = _pair_ids(V, 2 * V + n, gen, "uniform")
        first = _edges(ids[:2 * V], V).cpu().numpy()
        st, t = C.cupc_server_update(srv, gid, first, np.ones(2 * V, np.int8), 2 * V)
        C.check(st, "cupc_server_update")
        waits.append(t)
        reqs.append((gid, _edges(ids[2 * V:], V).cpu().numpy(), [np.full(n, x, np.int8) for x in (1, -1)], n,
                     _pairs(V, m, gen).cpu().numpy()))
    for t in waits:
        C.check(C.cupc_server_wait(srv, t)[0], "cupc_server_wait")
    return {"run": _run_serve, "srv": owner, "reqs": reqs, "m": m, "answers": np.zeros((k, m), np.uint8), "turn": 0}


def _run_serve(s):
    srv, turn, waits = s["srv"].h, _turn(s), []
    for (gid, e, o, n, pairs), answers in zip(s["reqs"], s["answers"]):
        st, t = C.cupc_server_update(srv, gid, e, o[turn], n)
        C.check(st, "cupc_server_update")
        waits.append(t)
        st, t = C.cupc_server_query(srv, gid, pairs, s["m"], answers)
        C.check(st, "cupc_server_query")
        waits.append(t)
    for t in waits:
        C.check(C.cupc_server_wait(srv, t)[0], "cupc_server_wait")
    return s["answers"]


# ---- the parallel cutset


def _prepare_cutset(c, seed, gen):
    V, n = c["V"], c["n"]
    g = Graph(V, seed, 1 << 16)
    _insert(g, _pair_ids(V, c["base"], gen, "uniform"))
    st, cs = C.cupc_cutset_create(g.h, None)
    C.check(st, "cupc_cutset_create")
    owner = Owned(cs, C.cupc_cutset_destroy, (g,))
    rng = np.random.default_rng(seed)
    parent = rng.integers(0, np.arange(1, V))  # a random recursive tree: (v, parent of v), v = 1 .. V-1
    tree = np.stack([np.arange(1, V), parent], 1)
    link = np.concatenate([np.full((V - 1, 1), C.CUPC_CUTSET_LINK), tree], 1).astype(np.uint32).reshape(-1)
    st, done = C.cupc_cutset_apply(cs, link, None)
    C.check(st, "cupc_cutset_apply")
    some = tree[rng.permutation(V - 1)[:n]]
    ops = [np.concatenate([np.full((n, 1), kind), some], 1).astype(np.uint32).reshape(-1)
           for kind in (C.CUPC_CUTSET_CUT, C.CUPC_CUTSET_LINK)]
    return {"run": _run_cutset, "cs": owner, "ops": ops, "asks": [int(x) for x in some[:c["asks"], 0]], "turn": 0,
            "sketch": torch.zeros(g.L * g.W * 2, dtype=torch.int64, device="cuda")}


def _run_cutset(s):
    cs = s["cs"].h
    st, done = C.cupc_cutset_apply(cs, s["ops"][_turn(s)], None)
    C.check(st, "cupc_cutset_apply")
    found = np.zeros((len(s["asks"]), 2), np.int64)
    for i, w in enumerate(s["asks"]):
        st, res, edge = C.cupc_cutset_query(cs, w, 0, None)
        C.check(st, "cupc_cutset_query")
        found[i] = res, edge
    C.check(C.cupc_cutset_tree_sketch(cs, s["asks"][0], s["sketch"], None))
    return found, s["sketch"]


# ---- what a pass cannot do without


def _dims(V):
    lg = max(1, (V - 1).bit_length())
    return lg + 2, 7, 2 * lg  # layers, columns, rows per column


def _touched(V, n, dist):
    """Expected distinct buckets that a batch of n edges changes: a vertex
    with a Poisson number of records of mean m changes the bucket of depth
    probability p with probability 1 - exp(-m p)."""
    L, cols, D = _dims(V)
    probs = [2.0 ** -(d + 1) for d in range(D - 1)] + [2.0 ** -(D - 1)]

    def per_vertex(m):
        return (1 - math.exp(-m)) + cols * sum(1 - math.exp(-m * p) for p in probs)

    if dist == "uniform":
        return L * V * per_vertex(2.0 * n / V)
    lv, zero = V.bit_length() - 1, RMAT[0] + RMAT[1]
    return L * sum(math.comb(lv, k) * per_vertex(2.0 * n * zero ** (lv - k) * (1 - zero) ** k) for k in range(lv + 1))


def _update_bytes(V, n, dist="uniform"):
    return 9.0 * n + 32.0 * _touched(V, n, dist)  # the batch; each changed bucket read and written


def _recovery_bytes(V):
    L, cols, D = _dims(V)
    return 2.0 * V * (1 + cols * D) * 16 + 8.0 * V  # two layers of every vertex, labels, forest


def work(case):
    k = case["kind"]
    if k == "update":
        return {"bytes": _update_bytes(case["V"], case["n"], case["dist"]), "flops": 0}
    if k == "query":
        return {"bytes": _update_bytes(case["V"], case["n"]) + _recovery_bytes(case["V"]) + 9.0 * case["pairs"], "flops": 0}
    if k == "cliques":
        return {"bytes": _update_bytes(CLIQUES_V, case["n"]) + _recovery_bytes(CLIQUES_V) + 9.0 * case["pairs"], "flops": 0}
    if k == "batch":
        return {"bytes": sum(_update_bytes(V, case["n"]) for V in _spread(case["V"], case["V_hi"], case["graphs"])),
                "flops": 0}
    if k == "incremental":
        more = _recovery_bytes(case["V"]) if case["tree"] else 0.0
        return {"bytes": _update_bytes(case["V"], case["n"]) + 9.0 * case["pairs"] + more, "flops": 0}
    if k == "serve":
        sizes = _spread(case["V"], case["V_hi"], case["graphs"])
        counts = _spread(case["n"], case["n_hi"], case["graphs"])
        return {"bytes": sum(_update_bytes(V, counts[(5 * i) % len(sizes)]) + _recovery_bytes(V) + 9.0 * case["pairs"]
                             for i, V in enumerate(sizes)), "flops": 0}
    # a cut or link changes the aggregates over about 4 log2(3V) tour nodes
    L, cols, D = _dims(case["V"])
    nodes = min(3.0 * case["V"], case["n"] * 4 * math.log2(3 * case["V"]))
    return {"bytes": nodes * 4 * L * (1 + cols * D) * 16, "flops": 0}
