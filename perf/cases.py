"""The calls this library is measured on, as a program that uses it makes them.

A case is one call pattern at one size: ``prepare`` makes what the program has
in hand (graphs on the device or the host, buffers, a planned batch), ``run``
makes the call through the public binding and hands back its results, ``draw``
gives more cases of the same ranges.  Results are whole numbers (counts,
histograms, hashes modulo 2^64, clique listings), so two correct builds agree
bit for bit.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1801_00202_gb300 as mce

_CTX = None


def _ctx():
    """The program's one context on GPU 0."""
    global _CTX
    if _CTX is None:
        _CTX = mce.Context(0)
    return _CTX


# ---------------------------------------------------------------------------
# Cases

def listed():
    return [
        # the smallest request: a neighbourhood-sized graph already on the
        # device, enumerated with caller-owned buffers; launches and latency
        # are the whole cost
        {"name": "gnp45", "kind": "device", "graph": "gnp", "n": 45, "p": 0.5, "pivot": "greedy"},
        # the small benchmark graph G(100, 0.5), same call
        {"name": "gnp100", "kind": "device", "graph": "gnp", "n": 100, "p": 0.5, "pivot": "greedy"},
        # structured worst case: the complement of 15 triangles (3^15 maximal
        # cliques on 45 vertices), a resident graph enumerated to host results
        {"name": "moonmoser45", "kind": "plain", "graph": "moonmoser", "n": 45, "del": 0.0, "pivot": "greedy"},
        # the same with 5 % of its edges removed: a lopsided search tree
        {"name": "moonmoser45_del", "kind": "plain", "graph": "moonmoser", "n": 45, "del": 0.05, "pivot": "greedy"},
        # a Table 1 shape under the pivot rule that scores every candidate
        {"name": "gnp300_tomita", "kind": "plain", "graph": "gnp", "n": 300, "p": 0.5, "pivot": "tomita"},
        # the flagship graph, host edge list in, result out, graph freed
        {"name": "gnp1000_load", "kind": "load", "graph": "gnp", "n": 1000, "p": 0.3, "pivot": "greedy"},
        # the heaviest dense Table 1 shape but one: about 10^8 maximal cliques
        {"name": "gnp500", "kind": "plain", "graph": "gnp", "n": 500, "p": 0.5, "pivot": "greedy"},
        # many vertices, low density: rows too large for shared memory
        {"name": "gnp3000", "kind": "device", "graph": "gnp", "n": 3000, "p": 0.1, "pivot": "greedy"},
        # every maximal clique listed to host memory in lexicographic order (an
        # unsorted listing has no fixed order to compare)
        {"name": "list700", "kind": "list", "graph": "gnp", "n": 700, "p": 0.3, "pivot": "greedy", "mix": 7},
        # a planned batch of uneven graphs, n in [32, 512], p in [0.2, 0.8]
        {"name": "batch512", "kind": "batch", "count": 512, "n_lo": 32, "n_hi": 512, "mix": 4},
        # a burst of served requests, n log-uniform in [64, 2048], p in [0.1, 0.9]
        {"name": "served256", "kind": "served", "count": 256, "n_lo": 64, "n_hi": 2048, "mix": 5},
        # a sparse graph beyond the bitset path: the degeneracy-ordered outer
        # loop of Alg. 3 (a Table 1 shape)
        {"name": "sparse10000", "kind": "plain", "graph": "gnp", "n": 10000, "p": 0.005, "pivot": "greedy"},
    ]


def draw(rng):
    kind = rng.choice(["device", "device", "plain", "plain", "load", "list", "batch", "served", "sparse", "moonmoser"])
    if kind in ("batch", "served"):
        count = int(round(math.exp(rng.uniform(math.log(24), math.log(512 if kind == "batch" else 256)))))
        lo, hi = (32, 512) if kind == "batch" else (64, 2048)
        return {"kind": kind, "count": count, "n_lo": lo, "n_hi": hi, "mix": rng.randrange(1 << 20)}
    if kind == "sparse":
        n = int(round(math.exp(rng.uniform(math.log(4200), math.log(10000)))))
        return {"kind": "plain", "graph": "gnp", "n": n, "p": round(rng.uniform(0.001, 0.008), 5),
                "pivot": rng.choice(["greedy", "tomita"])}
    pivot = rng.choice(["greedy", "greedy", "tx", "nx", "tomita"])
    if kind == "moonmoser":
        return {"kind": rng.choice(["plain", "device"]), "graph": "moonmoser", "n": 3 * rng.randint(8, 14),
                "del": round(rng.uniform(0.0, 0.1), 4), "pivot": pivot}
    top = 1e6 if kind == "list" else 1e7
    while True:
        n = int(round(math.exp(rng.uniform(math.log(33), math.log(3000)))))
        p = round(rng.uniform(0.05, 0.9), 4)
        if expected_cliques(n, p) <= top:
            break
    case = {"kind": kind, "graph": "gnp", "n": n, "p": p, "pivot": pivot}
    if kind == "list":
        case["mix"] = rng.randrange(1 << 20)
    return case


# ---------------------------------------------------------------------------
# Graphs

_LOGF = np.concatenate([[0.0], np.cumsum(np.log(np.arange(1, 65537, dtype=np.float64)))])


def expected_cliques(n, p):
    """Expected maximal cliques of G(n, p): sum over sizes k of
    C(n, k) p^C(k, 2) (1 - p^k)^(n - k)."""
    k = np.arange(1, min(n, 400) + 1)
    with np.errstate(divide="ignore", under="ignore"):
        t = (_LOGF[n] - _LOGF[k] - _LOGF[n - k] + 0.5 * k * (k - 1.0) * math.log(p)
             + (n - k) * np.log1p(-np.power(float(p), k)))
        return float(np.exp(np.minimum(t, 700.0)).sum())


def _gnp(n, p, gen):
    """Symmetric adjacency of G(n, p) as a bool matrix on the GPU."""
    a = torch.triu(torch.rand(n, n, device="cuda", generator=gen) < p, 1)
    return a | a.T


def _moonmoser(n, frac, gen):
    """Complement of n/3 disjoint triangles with a share of its edges removed
    and its vertices relabelled at random."""
    part = torch.arange(n, device="cuda") // 3
    part = part[torch.randperm(n, device="cuda", generator=gen)]
    a = torch.triu(part[:, None] != part[None, :], 1)
    uv = a.nonzero()
    drop = int(round(frac * uv.shape[0]))
    if drop:
        uv = uv[torch.randperm(uv.shape[0], device="cuda", generator=gen)[:drop]]
        a[uv[:, 0], uv[:, 1]] = False
    return a | a.T


def _bits(a):
    """Bitset rows (bit j of row i = word j // 32, bit j % 32) as int32."""
    n = a.shape[0]
    w = (n + 31) // 32
    pad = torch.zeros(n, w * 32, dtype=torch.bool, device=a.device)
    pad[:, :n] = a
    weight = torch.ones(32, dtype=torch.int64, device=a.device) << torch.arange(32, device=a.device)
    return (pad.view(n, w, 32) * weight).sum(-1).to(torch.int32).contiguous()


def _adjacency(case, gen):
    if case["graph"] == "moonmoser":
        return _moonmoser(case["n"], case["del"], gen)
    if case["kind"] == "list":
        # one graph of the case's own stream, its vertices relabelled by the
        # seed: every seed's listing has the same length
        a = _gnp(case["n"], case["p"], _gen(case["mix"]))
        perm = torch.randperm(case["n"], device="cuda", generator=gen)
        return a[perm][:, perm]
    return _gnp(case["n"], case["p"], gen)


def _edges(a):
    return torch.triu(a, 1).nonzero().to(torch.int32).cpu().numpy().view(np.uint32)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _mixed_sizes(case):
    """(n, p) of the graphs of a batch or a request burst: drawn from the
    case's own stream, redrawn while they expect over 10^6 maximal cliques."""
    rng = random.Random(case["mix"])
    out = []
    while len(out) < case["count"]:
        if case["kind"] == "batch":
            n, p = rng.randint(case["n_lo"], case["n_hi"]), rng.uniform(0.2, 0.8)
        else:
            n = int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
            p = rng.uniform(0.1, 0.9)
        if expected_cliques(n, p) <= 1e6:
            out.append((n, p))
    return out


# ---------------------------------------------------------------------------
# Calls

def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind in ("batch", "served"):
        sizes = _mixed_sizes(case)
        rows = [_bits(_gnp(n, p, gen)).cpu().numpy().view(np.uint32) for n, p in sizes]
        graphs = [_ctx().load_bitset(n, r) for (n, _), r in zip(sizes, rows)]
        state = {"kind": kind, "graphs": graphs}
        if kind == "batch":
            state["batch"] = mce.Batch(_ctx(), graphs)
        return state
    n = case["n"]
    adj = _adjacency(case, gen)
    opts = mce.options(pivot=case["pivot"], flags=mce.MCE_LIST_SORTED if kind == "list" else 0)
    state = {"kind": kind, "n": n, "opts": opts}
    if kind == "device":
        state["rows"] = _bits(adj)
        state["bytes"] = mce.mce_scratch_bytes(n, opts)
        state["scratch"] = torch.empty(state["bytes"], dtype=torch.uint8, device="cuda")
        out = torch.zeros(mce.MCE_OUT_WORDS(n), dtype=torch.int64, device="cuda")
        # the result words of the caller's buffer (the rest are scheduling diagnostics)
        state["out"] = out
        state["result"] = {"words": out[:mce.MCE_OUT_MAX_SIZE + 1], "hist": out[mce.MCE_OUT_HIST:]}
    elif kind == "load" or n > mce.MCE_NMAX:
        state["uv"] = _edges(adj)
        if kind != "load":
            state["graph"] = _ctx().load_edges(n, state.pop("uv"))
    else:
        state["graph"] = _ctx().load_bitset(n, _bits(adj).cpu().numpy().view(np.uint32))
    return state


def _signed(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _result(r):
    out = {k: r[k] for k in ("count", "nodes", "internal", "dead_ends", "max_size")}
    out["hash"] = _signed(r["hash"])
    out["hist"] = r["hist"].view(np.int64)
    for k in ("list_off", "list_ids"):
        if k in r:
            out[k] = r[k].view(np.int64 if k == "list_off" else np.int32)
    return out


def _results(rs):
    words = [[r["count"], r["nodes"], r["internal"], r["dead_ends"], r["max_size"], _signed(r["hash"])] for r in rs]
    return {"words": np.array(words, dtype=np.int64), "hist": np.concatenate([r["hist"] for r in rs]).view(np.int64)}


def run(state):
    kind = state["kind"]
    if kind == "device":
        rows, n = state["rows"], state["n"]
        rc = mce.mce_enumerate_device(n, rows.shape[1], rows, state["opts"], state["scratch"], state["bytes"],
                                      state["out"], torch.cuda.current_stream())
        if rc != 0:
            raise mce.MceError(rc, "mce_enumerate_device")
        return state["result"]
    if kind in ("plain", "list"):
        return _result(state["graph"].enumerate(state["opts"]))
    if kind == "load":
        g = _ctx().load_edges(state["n"], state["uv"])
        r = g.enumerate(state["opts"])
        g.free()
        return _result(r)
    if kind == "batch":
        return _results(state["batch"].run())
    ctx = _ctx()
    tickets = [ctx.submit(g) for g in state["graphs"]]
    return _results([ctx.wait(t) for t in tickets])


# ---------------------------------------------------------------------------
# What a pass cannot do without

def _one(n, cliques, deg):
    """Bytes in and out of one graph, and word operations of one search node
    (AND for P and X, two emptiness tests, ANDNOT, first bit: six per word of
    the candidate set) per maximal clique."""
    w = max(1, (int(min(n, deg + 1)) + 31) // 32)
    return n * ((n + 31) // 32) * 4 + (n + 8) * 8, 6.0 * w * cliques


def work(case):
    kind = case["kind"]
    if kind in ("batch", "served"):
        each = [_one(n, expected_cliques(n, p), n) for n, p in _mixed_sizes(case)]
        return {"bytes": float(sum(b for b, _ in each)), "flops": float(sum(f for _, f in each))}
    n = case["n"]
    if case["graph"] == "moonmoser":
        # a choice of one vertex per triangle stays a clique when none of its
        # n (n - 3) / 18 edges is removed
        cliques = 3.0 ** (n / 3.0) * (1.0 - case["del"]) ** (n * (n - 3) / 18.0)
        b, f = _one(n, max(cliques, float(n)), n)
        return {"bytes": float(b), "flops": float(f)}
    cliques, deg = expected_cliques(n, case["p"]), case["p"] * n
    b, f = _one(n, cliques, n if n <= 4096 else deg)
    if n > 4096:
        b = (n + 1) * 4 + n * deg * 4 + (n + 8) * 8
    if kind == "load":
        b += n * (n - 1) * case["p"] / 2 * 8
    if kind == "list":
        size = max(1.0, math.log(max(n, 2)) / -math.log(case["p"]))  # members of a typical maximal clique
        b += cliques * (4 * size + 8)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# The same results from the definition, for graphs small enough for plain Python

_M64 = (1 << 64) - 1


def _mix64(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def exact(case, seed):
    """Histogram, count, hash and sorted listing by Bron-Kerbosch over Python
    integers; the search-tree counters belong to the library's own tree and
    have no value here."""
    if case["kind"] in ("batch", "served"):
        return None
    n = case["n"]
    cliques = 3.0 ** (n / 3.0) if case["graph"] == "moonmoser" else expected_cliques(n, case["p"])
    if cliques > 1e5 or n > 1000:
        return None
    a = _adjacency(case, _gen(seed)).cpu().numpy()
    nb = [sum(1 << int(j) for j in np.nonzero(a[i])[0]) for i in range(n)]
    found = []

    def bits(s):
        while s:
            low = s & -s
            yield low.bit_length() - 1
            s ^= low

    def search(r, p, x):
        if not p:
            if not x:
                found.append(sorted(r))
            return
        u = max(bits(p | x), key=lambda v: (p & nb[v]).bit_count())
        for v in bits(p & ~nb[u]):
            search(r + [v], p & nb[v], x & nb[v])
            p &= ~(1 << v)
            x |= 1 << v

    search([], (1 << n) - 1, 0)
    hist = np.zeros(n + 1, dtype=np.int64)
    total = 0
    for c in found:
        hist[len(c)] += 1
        s = sum(_mix64(v + 1) for v in c) & _M64
        total = (total + _mix64(s ^ _mix64(len(c)))) & _M64
    if case["kind"] == "device":
        return {"words": None, "hist": hist}
    out = {"count": len(found), "nodes": None, "internal": None, "dead_ends": None,
           "max_size": max(len(c) for c in found), "hash": _signed(total), "hist": hist}
    if case["kind"] == "list":
        found.sort()
        out["list_off"] = np.cumsum([0] + [len(c) for c in found]).astype(np.int64)
        out["list_ids"] = np.array([v for c in found for v in c], dtype=np.int32)
    return out
