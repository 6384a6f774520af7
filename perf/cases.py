"""The work that a user of this library has it do, as cases that can be timed.

Each case opens a seeded synthetic graph (Erdos-Renyi, or a Chung-Lu power-law
graph, the stand-in for the social and web graphs the library is for) and makes
calls on it through ``paper_2308_14493_gb300.gc``: the static count, single
batches in both forms (region recount and edge-local delta), what-if queries,
batched runs, local counts, and the serving loop.  Graph sizes are those of the
workloads in ``synth/gen.py``.

A pass that applies batches also applies their inverses in reverse order, so
that it leaves the graph as it found it: a window that slides forward and back.
All outputs are whole numbers (counts); uint64 words come back as int64 views.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_14493_gb300 import gc as gcb

OPS = ("count", "apply", "whatif", "run", "whatifs", "vertex_orbits", "edge_orbits", "edge_counts", "serve")


def _case(name, op, n, m, gamma, dmax, size=0, ins=0.0, local=0, k=0):
    return {"name": name, "op": op, "n": n, "m": m, "gamma": gamma, "dmax": dmax, "size": size, "ins": ins,
            "local": local, "k": k}


def listed():
    return [
        # a small graph counted from scratch: one short call, bound by launches
        _case("count_er_2k", "count", 2000, 20000, 0.0, 0.0),
        # the largest resident graph of the serving workload, recounted (the recount baseline)
        _case("count_cl_4800k", "count", 4800000, 69000000, 2.4, 11747.0),
        # a vote network of 7,000 vertices followed by batches of 1,000 updates, library defaults
        _case("apply_cl_7k_1000", "apply", 7000, 100000, 2.1, 1000.0, 1000, 0.5),
        # the same network, insert-only, asked "what if" with 10,000 pairs already on the device
        _case("whatif_cl_7k_10000", "whatif", 7000, 100000, 2.1, 1000.0, 10000, 1.0),
        # a social network kept current by small frequent batches (the paper's batch size)
        _case("apply_cl_1600k_100", "apply", 1600000, 30000000, 2.3, 10000.0, 100, 0.7, 65536),
        # ... and by larger, less frequent ones
        _case("apply_cl_1600k_10000", "apply", 1600000, 30000000, 2.3, 10000.0, 10000, 0.6, 65536),
        # bulk updates of the social network: a run of 100,000-update batches in one call
        _case("run_cl_1600k_100000", "run", 1600000, 30000000, 2.3, 10000.0, 100000, 0.6, 65536, 4),
        # independent what-if batches of very uneven sizes on a talk network with huge hubs
        _case("whatifs_cl_2400k", "whatifs", 2400000, 5000000, 1.8, 100000.0, 50000, 0.5, 2048, 16),
        # orbit features of every vertex of the social network
        _case("vertex_orbits_cl_1600k", "vertex_orbits", 1600000, 30000000, 2.3, 10000.0),
        # orbit features of every edge of a mid-sized network
        _case("edge_orbits_cl_302k", "edge_orbits", 302000, 3350000, 2.114, 2588.0),
        # per-edge graphlet counts of the small network
        _case("edge_counts_cl_7k", "edge_counts", 7000, 100000, 2.1, 1000.0),
        # several graphs served at once, requests of 100 to 100,000 updates
        _case("serve_4_graphs", "serve", 525000, 6140000, 2.171, 3504.0, 100000, 0.7, 16384, 12),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(OPS)
    m = int(_log(rng, 20000, {"count": 4e7, "serve": 6e6, "edge_orbits": 4e6, "edge_counts": 4e6}.get(op, 2.5e7)))
    n = max(1000, int(m / _log(rng, 2.0, 20.0)))
    gamma = round(rng.uniform(1.8, 2.4), 3)
    # maximum expected degree around sqrt(2m); sparse graphs may have far larger hubs
    dmax = math.sqrt(2.0 * m) * _log(rng, 0.5, 6.0 if m < 5e6 else 1.5)
    dmax = round(min(max(dmax, 8.0 * m / n), n / 8.0), 1)
    size = int(_log(rng, 10, min(100000, m / 10)))
    ins = rng.choice((0.5, 0.6, 0.7, 1.0))
    # thresholds as the autotuner finds them: low where hubs are huge (each pair then costs far more probes)
    local = rng.choice((0, 2048, 16384, 65536) if dmax <= 1.5 * math.sqrt(2.0 * m) else (0, 512, 2048))
    k = {"run": rng.randint(2, 5), "whatifs": rng.randint(3, 16), "serve": rng.randint(3, 12)}.get(op, 0)
    if op not in ("apply", "whatif", "run", "whatifs", "serve"):
        size, ins, local = 0, 0.0, 0
    c = _case("", op, n, m, gamma, dmax, size, ins, local, k)
    del c["name"]
    return c


# ---- inputs --------------------------------------------------------------------


def _weights(n, m, gamma, dmax):
    """Expected degrees proportional to i^(-1/(gamma-1)), capped at dmax, sum 2m."""
    base = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    lo, hi = 0.0, 2.0 * m
    while float(torch.clamp(hi * base, max=dmax).sum()) < 2.0 * m * 0.999 and hi < 1e18:
        hi *= 2.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        if float(torch.clamp(mid * base, max=dmax).sum()) < 2.0 * m:
            lo = mid
        else:
            hi = mid
    return torch.clamp(hi * base, max=dmax)


def _keys(u, v):
    ok = u != v
    u, v = u[ok], v[ok]
    return (torch.minimum(u, v) << 32) | torch.maximum(u, v)


def _graph(gen, n, m, gamma, dmax):
    """Sorted canonical keys of m distinct pairs, vertex ids randomly permuted."""
    cdf = None
    if gamma:
        cdf = torch.cumsum(_weights(n, m, gamma, dmax), 0)
        cdf /= cdf[-1].clone()
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        need = int((m - keys.numel()) * 1.15) + 1024
        if cdf is None:
            e = torch.randint(0, n, (2, need), generator=gen, device="cuda")
        else:
            e = torch.searchsorted(cdf, torch.rand((2, need), generator=gen, device="cuda", dtype=torch.float64),
                                   right=True).clamp_(max=n - 1)
        keys = torch.unique(torch.cat([keys, _keys(e[0], e[1])]))
    if keys.numel() > m:
        keys = keys[torch.randperm(keys.numel(), generator=gen, device="cuda")[:m]]
    ids = torch.randperm(n, generator=gen, device="cuda")
    return torch.sort(_keys(ids[keys >> 32], ids[keys & 0xFFFFFFFF]))[0]


def _csr(n, keys):
    u, v = keys >> 32, keys & 0xFFFFFFFF
    both = torch.sort(torch.cat([keys, (v << 32) | u]))[0]
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(both >> 32, minlength=n), 0)
    return rp.to(torch.int32).cpu().numpy(), (both & 0xFFFFFFFF).to(torch.int32).cpu().numpy()


def _batch(gen, n, keys, n_ins, n_del):
    """n_del distinct edges, n_ins distinct non-edges with endpoints in proportion to degree + 1."""
    m = keys.numel()
    pick = torch.empty(0, dtype=torch.int64, device="cuda")
    while pick.numel() < n_del:
        more = torch.randint(0, m, (n_del + 16,), generator=gen, device="cuda")
        pick = torch.unique(torch.cat([pick, more]))
    dels = keys[pick[torch.randperm(pick.numel(), generator=gen, device="cuda")[:n_del]]]
    ins = torch.empty(0, dtype=torch.int64, device="cuda")
    while ins.numel() < n_ins:
        r = torch.randint(0, 2 * m + n, (2, 2 * n_ins + 64), generator=gen, device="cuda")
        k = keys[torch.clamp(r >> 1, max=m - 1)]
        e = torch.where(r < 2 * m, torch.where((r & 1) == 1, k >> 32, k & 0xFFFFFFFF), r - 2 * m)
        cand = _keys(e[0], e[1])
        at = torch.searchsorted(keys, cand).clamp_(max=m - 1)
        ins = torch.unique(torch.cat([ins, cand[keys[at] != cand]]))
    ins = ins[torch.randperm(ins.numel(), generator=gen, device="cuda")[:n_ins]]

    def pairs(k):
        flip = torch.rand(k.numel(), generator=gen, device="cuda") < 0.5
        a, b = k >> 32, k & 0xFFFFFFFF
        return torch.stack([torch.where(flip, b, a), torch.where(flip, a, b)], 1).to(torch.int32).contiguous()

    return pairs(ins), pairs(dels)


def _split(size, ins):
    n_ins = int(round(size * ins))
    return n_ins, size - n_ins


def _there_and_back(batches):
    """The batches, then their inverses in reverse order: the graph ends as it began."""
    return list(batches) + [(d, i) for i, d in reversed(batches)]


class _Serving:
    """A server over its graphs; closed before them."""

    def __init__(self, graphs, slots):
        self.graphs = graphs
        self.server = gcb.Server(graphs, slots=slots)

    def __del__(self):
        self.server.close()
        for g in self.graphs:
            g.close()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    op, n, m, k = case["op"], case["n"], case["m"], case["k"]

    def opened(n, m, gamma, dmax):
        keys = _graph(gen, n, m, gamma, dmax)
        rp, col = _csr(n, keys)
        return gcb.Graph(n, rp, col, local_max_pairs=case["local"]), keys

    def host(b):
        return tuple(x.cpu().numpy() for x in b)

    state = {"op": op}
    if op == "serve":
        graphs, reqs = [], []
        for i in range(4):  # sizes from a sixth of the largest up to it
            f = 6.14 ** (-(3 - i) / 3.0)
            gn, gm = max(1000, int(n * f)), max(10000, int(m * f))
            g, keys = opened(gn, gm, case["gamma"], min(max(case["dmax"] * f ** 0.5, 8.0 * gm / gn), gn / 8.0))
            graphs.append(g)
            # k requests over the graphs in turn, sizes spread over the logarithm of their range
            mine = range(i, k, 4)
            lo, hi = math.log(min(100, case["size"])), math.log(min(case["size"], gm // 10))
            sizes = [int(math.exp(lo + (hi - lo) * ((j * 0.618034) % 1.0))) for j in mine]
            batches = [host(_batch(gen, gn, keys, *_split(s, case["ins"]))) for s in sizes]
            reqs += [(j, i, b) for j, b in enumerate(_there_and_back(batches))]
        reqs.sort(key=lambda r: r[:2])
        state["serving"] = _Serving(graphs, 4)
        state["requests"] = [(i, b[0], b[1]) for _, i, b in reqs]
        return state
    g, keys = opened(n, m, case["gamma"], case["dmax"])
    state["graph"] = g
    if op == "apply":
        state["batches"] = _there_and_back([host(_batch(gen, n, keys, *_split(case["size"], case["ins"])))])
    elif op == "whatif":
        state["pairs"] = _batch(gen, n, keys, *_split(case["size"], case["ins"]))
    elif op == "run":
        half = [host(_batch(gen, n, keys, *_split(case["size"], case["ins"]))) for _ in range(max(1, k // 2))]
        state["batches"] = _there_and_back(half)
    elif op == "whatifs":
        lo, hi = math.log(10), math.log(max(11, case["size"]))
        sizes = [int(math.exp(lo + (hi - lo) * ((j * 0.618034 + 0.5) % 1.0))) for j in range(k)]
        state["batches"] = [host(_batch(gen, n, keys, *_split(s, case["ins"]))) for s in sizes]
    return state


# ---- one pass ------------------------------------------------------------------


def _words(x):
    return np.ascontiguousarray(x).view(np.int64) if isinstance(x, np.ndarray) else np.array(x, np.uint64).view(np.int64)


def run(state):
    op = state["op"]
    if op == "serve":
        s = state["serving"].server
        tickets = [s.submit(i, ins, dels) for i, ins, dels in state["requests"]]
        return [_words([s.wait(t)["counts"] for t in tickets])]
    g = state["graph"]
    if op == "count":
        return [_words(g.count_static())]
    if op == "apply":
        return [_words([g.apply(ins, dels) for ins, dels in state["batches"]]), _words(g.counts3())]
    if op == "whatif":
        ins, dels = state["pairs"]
        return [_words(gcb.gc_count_batch_device(g.h, ins.data_ptr(), len(ins), dels.data_ptr(), len(dels)))]
    if op == "run":
        return [_words(g.apply_many(state["batches"])), _words(g.counts3())]
    if op == "whatifs":
        return [_words(g.apply_many(state["batches"], independent=True))]
    if op == "vertex_orbits":
        return [_words(g.vertex_orbits())]
    edges, counts = g.edge_orbits() if op == "edge_orbits" else g.edge_counts()
    return [edges, _words(counts)]


def work(case):
    """Bytes: the adjacency entries that the counts depend on, the pairs, the outputs, each once.

    A recount reads the whole CSR.  A batch in the edge-local form reads the
    rows of its endpoints (about 2m / n entries each; hubs are more) once."""
    op, n, m, size, k = case["op"], case["n"], case["m"], case["size"], case["k"]
    csr = 4 * (n + 1) + 8 * m

    def batch(s, n=n, m=m, csr=csr):
        rows = min(csr, 2 * s * 4 * (2 * m // n + 1))
        return 8 * s + 48 + (rows if 0 < s <= case["local"] else csr)

    if op == "apply":
        b = 2 * batch(size)
    elif op == "whatif":
        b = batch(size)
    elif op == "run":
        b = 2 * max(1, k // 2) * batch(size)
    elif op == "whatifs":
        lo, hi = math.log(10), math.log(max(11, size))
        b = sum(batch(int(math.exp(lo + (hi - lo) * ((j * 0.618034 + 0.5) % 1.0)))) for j in range(k))
    elif op == "serve":
        b = 0
        for i in range(4):
            f = 6.14 ** (-(3 - i) / 3.0)
            gn, gm = max(1000, int(n * f)), max(10000, int(m * f))
            lo, hi = math.log(min(100, size)), math.log(min(size, gm // 10))
            for j in range(i, k, 4):
                b += 2 * batch(int(math.exp(lo + (hi - lo) * ((j * 0.618034) % 1.0))), gn, gm, 4 * (gn + 1) + 8 * gm)
    elif op == "vertex_orbits":
        b = csr + 88 * n
    elif op == "edge_orbits":
        b = csr + 88 * m
    elif op == "edge_counts":
        b = csr + 56 * m
    else:
        b = csr + 48
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Every output is a whole number: there is nothing to round."""
    return None
