"""Timed cases: connectivity calls as a user's program makes them.

Every case is one call path of the library on a seeded graph made on the GPU:
``prepare`` builds the graph and whatever plan or handle such a program keeps,
``run`` is one pass through the public entry points.  Graphs follow the
repository's own workloads (Erdos-Renyi, RMAT with the Graph500 parameters,
grid + long paths, a batch of small graphs, an insert / query stream).

All outputs are whole numbers that are the same for every correct run
(canonical labels, forest counts, query answers).  A spanning forest's edge ids
are one of many valid choices and change from run to run, so the forest case
returns its edge count and labels.
"""
import math

import numpy as np
import torch

import paper_2008_11839_gb300 as gc

DEV = "cuda"
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19      # d = 0.05 (Graph500)


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # The smallest call: components of a graph of a thousand vertices,
        # where launches and the host path are all there is.
        {"name": "coo_tiny", "path": "coo", "graph": "er", "n": 1000, "m": 4000, "link": "default"},
        # The plain method on a small uniform random edge list (Union-Rem-CAS,
        # no on-the-fly compression): the benchmark's first configuration.
        {"name": "coo_er_64k", "path": "coo", "graph": "er", "n": 65536, "m": 1048576, "link": "remcas"},
        # The default finish over a whole large power-law edge list, as a user
        # has it who never builds a CSR.  Largest input of the static calls.
        {"name": "coo_rmat22", "path": "coo", "graph": "rmat", "n": 1 << 22, "m": 1 << 26, "link": "default"},
        # Road-like input: a 2D grid with holes plus long paths (high diameter,
        # low degree), edges in random order.
        {"name": "coo_grid_paths", "path": "coo", "graph": "grid", "side": 4096, "npaths": 64, "plen": 1 << 18,
         "link": "default"},
        # The headline: the default two-phase method on a CSR with 32-bit
        # offsets, replayed from a captured plan on changing contents.
        {"name": "csr32_rmat22_plan", "path": "csr", "graph": "rmat", "n": 1 << 22, "m": 1 << 26, "bits": 32,
         "sample": "kout", "link": "default", "plan": True},
        # The same method called directly, 64-bit offsets, HB sampling with
        # Union-Async, and a vertex count that is no power of two.
        {"name": "csr64_hb_rmat20", "path": "csr", "graph": "rmat", "n": 1000003, "m": 16000003, "bits": 64,
         "sample": "hb", "link": "async", "plan": False},
        # The two-phase method on the road-like input: sampling leaves work
        # for the finish here.
        {"name": "csr32_grid_paths", "path": "csr", "graph": "grid", "side": 2048, "npaths": 64, "plen": 1 << 16,
         "bits": 32, "sample": "kout", "link": "default", "plan": False},
        # Spanning forest with labels from a CSR (Algorithm 2), direct call.
        {"name": "forest_rmat20", "path": "forest", "graph": "rmat", "n": 1 << 20, "m": 1 << 24, "bits": 32,
         "sample": "kout", "link": "default"},
        # Thousands of small graphs of uneven size in one captured launch:
        # n log-uniform in [256, 65536], mean degree 4 to 32, half ER, half RMAT.
        {"name": "batched_4096", "path": "batched", "graphs": 4096, "nmin": 256, "nmax": 65536},
        # Incremental handle, small requests: one insert batch and one query
        # batch of a thousand pairs (the latency end of the stream).
        {"name": "inc_small", "path": "inc", "n": 1 << 20, "prefix": 1 << 22, "b": 1000, "q": 1000,
         "link": "default"},
        # Incremental handle, large requests in the middle of a long RMAT
        # stream (the throughput end): ten million inserts, as many queries.
        {"name": "inc_large", "path": "inc", "n": 1 << 24, "prefix": 1 << 26, "b": 10_000_000, "q": 10_000_000,
         "link": "early"},
        # A round-based finish (Liu-Tarjan PRF) on an edge list, for users of
        # the non-union-find half of the design space.
        {"name": "coo_lt_rmat20", "path": "coo", "graph": "rmat", "n": 1 << 20, "m": 1 << 24, "link": "lt"},
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["coo", "coo", "coo_grid", "csr", "csr", "csr_grid", "forest", "batched", "inc", "inc", "rounds"])
    if kind == "coo":
        n = logint(1000, 1 << 22)
        return {"path": "coo", "graph": rng.choice(["er", "rmat"]), "n": n, "m": int(n * rng.uniform(2, 16)),
                "link": rng.choice(["default", "default", "remcas", "async", "early"])}
    if kind == "coo_grid":
        return {"path": "coo", "graph": "grid", "side": logint(64, 4096), "npaths": rng.randint(1, 64),
                "plen": logint(256, 1 << 18), "link": "default"}
    if kind == "csr":
        n = logint(1000, 1 << 22)
        return {"path": "csr", "graph": rng.choice(["er", "rmat"]), "n": n, "m": int(n * rng.uniform(2, 16)),
                "bits": rng.choice([32, 64]), "sample": rng.choice(["kout", "kout", "hb", "none"]),
                "link": rng.choice(["default", "default", "async"]), "plan": rng.random() < 0.5}
    if kind == "csr_grid":
        return {"path": "csr", "graph": "grid", "side": logint(64, 2048), "npaths": rng.randint(1, 64),
                "plen": logint(256, 1 << 16), "bits": rng.choice([32, 64]), "sample": "kout", "link": "default",
                "plan": rng.random() < 0.5}
    if kind == "forest":
        n = logint(1000, 1 << 20)
        return {"path": "forest", "graph": rng.choice(["er", "rmat"]), "n": n, "m": int(n * rng.uniform(2, 16)),
                "bits": rng.choice([32, 64]), "sample": "kout", "link": "default"}
    if kind == "batched":
        nmin = logint(64, 1024)
        return {"path": "batched", "graphs": logint(128, 4096), "nmin": nmin, "nmax": logint(4 * nmin, 65536)}
    if kind == "inc":
        n = logint(1 << 18, 1 << 24)
        return {"path": "inc", "n": n, "prefix": int(n * rng.uniform(0.5, 4)), "b": logint(1000, 10_000_000),
                "q": logint(1000, 10_000_000), "link": rng.choice(["default", "early"])}
    n = logint(1000, 1 << 20)
    return {"path": "coo", "graph": rng.choice(["er", "rmat"]), "n": n, "m": int(n * rng.uniform(2, 16)),
            "link": rng.choice(["lt", "sv"])}


# -------------------------------------------------------------------- inputs
def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _rmat_ids(levels, m, g):
    """Two int32 id columns of m RMAT edges, `levels` quadrant draws each."""
    u = torch.zeros(m, dtype=torch.int32, device=DEV)
    v = torch.zeros(m, dtype=torch.int32, device=DEV)
    r = torch.empty(m, dtype=torch.float32, device=DEV)
    for _ in range(levels):
        r.uniform_(generator=g)
        down = r >= RMAT_A + RMAT_B
        right = (r >= RMAT_A) ^ down | (r >= RMAT_A + RMAT_B + RMAT_C)
        u.mul_(2).add_(down)
        v.mul_(2).add_(right)
    return u, v


def _rmat(n, m, g):
    """(m, 2) int32 RMAT edges on n vertices with randomly permuted ids; ids
    beyond n (n no power of two) are scaled into range."""
    levels = max(1, (n - 1).bit_length())
    perm = torch.randperm(n, device=DEV, generator=g).to(torch.int32)
    out = torch.empty(m, 2, dtype=torch.int32, device=DEV)
    for c, ids in enumerate(_rmat_ids(levels, m, g)):
        if n != 1 << levels:
            ids = (ids.to(torch.int64) * n >> levels).to(torch.int32)
        out[:, c] = perm[ids]
    return out


def _grid_paths(side, npaths, plen, g):
    """A side x side grid with 5 % of its edges removed plus npaths paths over
    randomly permuted vertices; edges in random order."""
    ids = torch.arange(side * side, dtype=torch.int32, device=DEV).view(side, side)
    right = torch.stack([ids[:, :-1].reshape(-1), ids[:, 1:].reshape(-1)], 1)
    down = torch.stack([ids[:-1].reshape(-1), ids[1:].reshape(-1)], 1)
    e = torch.cat([right, down])
    e = e[torch.rand(e.shape[0], device=DEV, generator=g) >= 0.05]
    p = (torch.randperm(npaths * plen, device=DEV, generator=g) + side * side).to(torch.int32).view(npaths, plen)
    e = torch.cat([e, torch.stack([p[:, :-1].reshape(-1), p[:, 1:].reshape(-1)], 1)])
    return side * side + npaths * plen, e[torch.randperm(e.shape[0], device=DEV, generator=g)].contiguous()


def _edges(case, seed):
    g = _gen(seed)
    if case["graph"] == "grid":
        return _grid_paths(case["side"], case["npaths"], case["plen"], g)
    n, m = case["n"], case["m"]
    if case["graph"] == "er":             # one id in 32 is unused, as in id spaces with gaps
        used = torch.randperm(n, device=DEV, generator=g)[:n - n // 32].to(torch.int32)
        return n, used[torch.randint(0, used.numel(), (m, 2), dtype=torch.int32, device=DEV, generator=g)]
    return n, _rmat(n, m, g)


def _csr(n, e, bits):
    """Symmetric CSR with sorted rows: offsets (int32 / int64) and int32 cols."""
    u, v = e[:, 0].to(torch.int64), e[:, 1].to(torch.int64)
    key = torch.cat([(u << 32) | v, (v << 32) | u]).sort().values
    off = torch.searchsorted(key, torch.arange(n + 1, device=DEV, dtype=torch.int64) << 32)
    return off.to(torch.int32 if bits == 32 else torch.int64), (key & 0xFFFFFFFF).to(torch.int32)


def _batch(case, seed):
    """Offsets (int64, host) and local-id edges of the batch's graphs; the
    graphs' sizes go with the case, their edges with the seed."""
    G, rs = case["graphs"], np.random.RandomState(case["graphs"])
    ns = np.floor(case["nmin"] * (case["nmax"] / case["nmin"]) ** rs.rand(G)).astype(np.int64)
    ms = np.maximum(1, np.rint(ns * rs.uniform(4.0, 32.0, G) / 2)).astype(np.int64)
    vo, eo = np.zeros(G + 1, np.int64), np.zeros(G + 1, np.int64)
    np.cumsum(ns, out=vo[1:])
    np.cumsum(ms, out=eo[1:])
    levels = max(1, int(case["nmax"] - 1).bit_length())
    edges = torch.empty(int(eo[-1]), 2, dtype=torch.int32, device=DEV)
    g, step = _gen(seed, 1), 256
    for lo in range(0, G, step):          # some hundred graphs at a time bound the temporaries
        hi = min(G, lo + step)
        a, b = int(eo[lo]), int(eo[hi])
        rep = torch.from_numpy(ms[lo:hi]).to(DEV)
        nn = torch.repeat_interleave(torch.from_numpy(ns[lo:hi]).to(DEV), rep)
        odd = torch.repeat_interleave(torch.arange(lo, hi, device=DEV) % 2 == 1, rep)
        for c, ids in enumerate(_rmat_ids(levels, b - a, g)):
            uni = torch.randint(0, 1 << levels, (b - a,), dtype=torch.int32, device=DEV, generator=g)
            edges[a:b, c] = (torch.where(odd, ids, uni).to(torch.int64) * nn >> levels).to(torch.int32)
    return vo, eo, edges


def _variant(case):
    link = case.get("link", "default")
    sample = case.get("sample", "none")
    if link == "default":
        v = gc.gconn_variant_default()
        v.sample = gc.SAMPLES[sample]
        return v
    if link == "remcas":
        return gc.make_variant(sample=sample, link="remcas", find="fullshortcut", splice="splice")
    if link == "lt":
        return gc.make_variant(sample=sample, link="lt", lt="PRF")
    return gc.make_variant(sample=sample, link=link)


class _Handle:
    """A plan or batch handle that goes with its state."""

    def __init__(self, h, destroy):
        self.h, self._destroy = h, destroy

    def __del__(self):
        self._destroy(self.h)


def prepare(case, seed):
    p = case["path"]
    s = {"case": dict(case)}
    if p == "batched":
        vo, eo, s["edges"] = _batch(case, seed)
        s["labels"] = torch.empty(int(vo[-1]), dtype=torch.int32, device=DEV)
        s["plan"] = _Handle(gc.gconn_batch_create(case["graphs"], vo, eo, s["edges"], s["labels"]),
                            gc.gconn_batch_destroy)
        return s
    if p == "inc":
        n, g = case["n"], _gen(seed, 2)
        stream = _rmat(n, case["prefix"] + case["b"], g)
        s["inc"] = gc.Incremental(n, gc.make_variant(link="early") if case["link"] == "early" else None)
        s["inc"].insert(stream[:case["prefix"]].contiguous())
        s["batch"] = stream[case["prefix"]:].clone()
        s["pairs"] = torch.randint(0, n, (case["q"], 2), dtype=torch.int32, device=DEV, generator=g)
        s["answers"] = torch.empty(case["q"], dtype=torch.uint8, device=DEV)
        return s
    n, e = _edges(case, seed)
    s["n"], s["variant"] = n, _variant(case)
    if p == "coo":
        s["edges"] = e
        return s
    s["off"], s["cols"] = _csr(n, e, case["bits"])
    s["labels"] = torch.empty(n, dtype=torch.int32, device=DEV)
    if p == "forest":
        s["forest"] = torch.empty(n, dtype=torch.int64, device=DEV)
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    elif case["plan"]:
        make = gc.gconn_plan_create_cc_csr32 if case["bits"] == 32 else gc.gconn_plan_create_cc_csr
        s["plan"] = _Handle(make(n, s["off"], s["cols"], s["labels"], s["variant"]), gc.gconn_plan_destroy)
    return s


# ---------------------------------------------------------------------- runs
def run(s):
    case = s["case"]
    p = case["path"]
    if p == "coo":
        return gc.cc(s["n"], s["edges"], s["variant"])
    if p == "csr":
        if case["plan"]:
            gc.gconn_plan_run(s["plan"].h)
        elif case["bits"] == 32:
            gc.gconn_cc_csr32(s["n"], s["off"], s["cols"], s["labels"], s["variant"])
        else:
            gc.gconn_cc_csr(s["n"], s["off"], s["cols"], s["labels"], s["variant"])
        return s["labels"]
    if p == "forest":
        f = gc.gconn_spanning_forest_csr32 if case["bits"] == 32 else gc.gconn_spanning_forest_csr
        f(s["n"], s["off"], s["cols"], s["forest"], s["count"], s["labels"], s["variant"])
        return {"count": s["count"], "labels": s["labels"]}
    if p == "batched":
        gc.gconn_batch_run(s["plan"].h)
        return s["labels"]
    s["inc"].insert(s["batch"])
    return s["inc"].query(s["pairs"], s["answers"])


def work(case):
    """Bytes a pass has to move: inputs once, outputs once.  A sampled CSR pass
    needs the offsets, two columns per vertex and the labels, not every arc; an
    insert is its pair, a query its pair and its answer.  There is no floating
    point arithmetic."""
    p = case["path"]
    if p == "inc":
        return {"bytes": 8 * case["b"] + 9 * case["q"], "flops": 0}
    if p == "batched":
        lo, hi = case["nmin"], case["nmax"]
        mean_n = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        return {"bytes": int(case["graphs"] * mean_n * (8 * 9 + 4)), "flops": 0}
    if case.get("graph") == "grid":
        n = case["side"] ** 2 + case["npaths"] * case["plen"]
        m = int(0.95 * 2 * case["side"] * (case["side"] - 1)) + case["npaths"] * (case["plen"] - 1)
    else:
        n, m = case["n"], case["m"]
    if p == "coo":
        return {"bytes": 8 * m + 4 * n, "flops": 0}
    arcs = 2 * m if case["sample"] == "none" else min(2 * m, 2 * n)
    return {"bytes": case["bits"] // 8 * (n + 1) + 4 * arcs + 4 * n + (8 * n if p == "forest" else 0), "flops": 0}
