"""The library's work as its users call it, as cases to be timed.

A user of the library has graphs and wants the exact top-k closeness of each
(create, preprocess, top-k, release), or keeps graphs resident and asks for
top-k again and again (serving), runs many small graphs as one batch, wants
the farness of every vertex, or only the SCCs and reach bounds.  The graphs
are the kinds the repository's generators and benchmark use: Chung-Lu and
Barabasi-Albert power-law graphs, R-MAT digraphs, damaged grids.  They are
drawn here on the GPU, from the seed alone, with the same recipes.

Every output is a whole number: ids, farness, reach, SCC labels, bounds.
"""
import functools
import math

import numpy as np
import torch

from paper_1507_01490_gb300 import bcm


def listed():
    return [
        # one request on a small resident graph: what launches and latency cost
        {"name": "ba2000_top10", "what": "topk", "graph": "ba", "n": 2000, "deg": 3, "k": 10},
        # the benchmark's step: handle from device CSR, preprocessing, top-10, release
        {"name": "graph_chunglu1m_top10", "what": "graph", "graph": "chunglu", "n": 1 << 20, "deg": 10, "k": 10},
        # the same step on the benchmark's digraph: SCCs, bounds and the widest waves
        {"name": "graph_rmat20_top10", "what": "graph", "graph": "rmat", "scale": 20, "deg": 16, "k": 10},
        # end to end from host arrays, an ordinary odd size, a longer list
        {"name": "host_chunglu200k_top100", "what": "host", "graph": "chunglu", "n": 200003, "deg": 10, "k": 100},
        # a request on a large resident graph of the serving mix: most sources outlive the wide waves
        {"name": "ba1m_top10", "what": "topk", "graph": "ba", "n": 1 << 20, "deg": 4, "k": 10},
        # lattices: deep, thin searches, one source at a time; a small one and the largest of all cases
        {"name": "grid128_top1", "what": "topk", "graph": "grid", "rows": 128, "cols": 128, "k": 1},
        {"name": "grid512_top10", "what": "topk", "graph": "grid", "rows": 512, "cols": 512, "k": 10},
        # the textbook answer for every vertex, undirected and directed
        {"name": "farness_chunglu16k", "what": "farness", "graph": "chunglu", "n": 1 << 14, "deg": 10},
        {"name": "farness_rmat16", "what": "farness", "graph": "rmat", "scale": 16, "deg": 8},
        # the same without any allocation
        {"name": "noalloc_chunglu10k", "what": "noalloc", "graph": "chunglu", "n": 10007, "deg": 10},
        # only the SCCs and the reach bounds of a digraph
        {"name": "scc_rmat18", "what": "scc", "graph": "rmat", "scale": 18, "deg": 16},
        # many small graphs recorded as one batch
        {"name": "batch64_top10", "what": "batch", "graph": "ba", "count": 64, "n": 8000, "deg": 4, "k": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["topk", "topk", "graph", "graph", "host", "farness", "noalloc", "scc", "batch"])
    k = rng.choice([1, 10, 100])
    if what == "topk":
        if rng.random() < 0.5:
            return {"what": what, "graph": "ba", "n": _log(rng, 1000, 1 << 20), "deg": rng.randint(2, 8), "k": k}
        return {"what": what, "graph": "grid", "rows": _log(rng, 40, 500), "cols": _log(rng, 40, 500), "k": k}
    if what in ("graph", "host", "scc"):
        rmat = {"what": what, "graph": "rmat", "scale": rng.randint(12, 19), "deg": rng.randint(4, 15)}
        if what == "scc":
            return rmat
        if rng.random() < 0.5:
            return dict(rmat, k=k)
        return {"what": what, "graph": "chunglu", "n": _log(rng, 5000, 1 << 20), "deg": rng.randint(6, 16), "k": k}
    if what == "farness":
        if rng.random() < 0.5:
            return {"what": what, "graph": "rmat", "scale": rng.randint(10, 15), "deg": rng.randint(4, 16)}
        return {"what": what, "graph": "chunglu", "n": _log(rng, 1000, 30000), "deg": rng.randint(6, 16)}
    if what == "noalloc":
        return {"what": what, "graph": "chunglu", "n": _log(rng, 1000, 12000), "deg": rng.randint(6, 16)}
    return {"what": what, "graph": "ba", "count": rng.randint(8, 64), "n": _log(rng, 1500, 8000),
            "deg": rng.randint(2, 8), "k": k}


# ------------------------------------------------------------------ graphs
def _csr(n, src, dst, directed):
    """CSR of an arc list: both directions unless directed, no self-loop, no repeat, rows sorted."""
    if not directed:
        src, dst = torch.cat([src, dst]), torch.cat([dst, src])
    key = src * n + dst
    key = torch.unique(key[src != dst])
    row, col = key // n, key % n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rp, col.to(torch.int32)


def _chunglu(n, deg, gen):
    """Endpoints drawn by power-law weights (degree exponent 2.3, mean deg, capped at sqrt(deg n))."""
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen).clamp_min(1e-12)
    w = ((u ** (-1 / 1.3)) * 1024).to(torch.int64)
    scale = deg * n / (int(w.sum()) / 1024)
    q = ((w.to(torch.float64) / 1024 * scale).clamp_max(math.sqrt(deg * n)) * (1 << 20)).to(torch.int64) + 1
    cum = torch.cumsum(q, 0)
    draws = n * deg // 2
    t = (torch.rand(2 * draws, dtype=torch.float64, device="cuda", generator=gen) * int(cum[-1])).to(torch.int64)
    e = torch.searchsorted(cum, t, right=True).clamp_max(n - 1)
    return _csr(n, e[:draws], e[draws:], False)


def _rmat(scale, deg, gen):
    """R-MAT arcs (0.57, 0.19, 0.19, 0.05), relabelled."""
    n, arcs = 1 << scale, deg << scale
    src = torch.zeros(arcs, dtype=torch.int64, device="cuda")
    dst = torch.zeros(arcs, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        q = torch.rand(arcs, dtype=torch.float32, device="cuda", generator=gen)
        src = src * 2 + (q >= 0.76)
        dst = dst * 2 + (((q >= 0.57) & (q < 0.76)) | (q >= 0.95))
    perm = torch.randperm(n, device="cuda", generator=gen)
    return _csr(n, perm[src], perm[dst], True)


def _ba(n, m, gen):
    """Preferential attachment: vertex t > m links to the endpoints at m random positions of the edge list
    before it (position 2e is edge e's new vertex, 2e + 1 its older one, followed until it is known)."""
    first = torch.combinations(torch.arange(m + 1, device="cuda"))
    k0 = first.shape[0]
    new = torch.arange(m + 1, n, device="cuda").repeat_interleave(m)
    src = torch.cat([first[:, 1], new])
    limit = 2 * (k0 + m * (new - (m + 1)))
    pos = (torch.rand(new.shape[0], dtype=torch.float64, device="cuda", generator=gen) * limit).to(torch.int64)
    pos = torch.cat([torch.full((k0,), -1, device="cuda"), pos])   # -1: a starting edge, known
    at = pos.clone()
    while True:   # an odd position whose edge is not a starting one: take that edge's position
        go = (at >= 0) & (at % 2 == 1) & (pos[(at // 2).clamp_min(0)] >= 0)
        if not bool(go.any()):
            break
        at = torch.where(go, pos[(at // 2).clamp_min(0)], at)
    old = torch.cat([first[:, 0], torch.zeros_like(new)])
    e = (at // 2).clamp_min(0)
    dst = torch.where(at < 0, old, torch.where(at % 2 == 0, src[e], old[e]))
    return _csr(n, src, dst, False)


def _grid(rows, cols, gen):
    """rows x cols grid with 5% of its edges deleted; the largest component, in id order."""
    v = torch.arange(rows * cols, device="cuda").view(rows, cols)
    a = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1)])
    b = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1)])
    keep = torch.randperm(a.shape[0], device="cuda", generator=gen)[int(round(0.05 * a.shape[0])):].sort()[0]
    a, b = a[keep], b[keep]
    label = torch.arange(rows * cols, device="cuda")
    while True:   # smallest label per component: hook roots under smaller ones, then flatten
        la, lb = label[a], label[b]
        if bool((la == lb).all()):
            break
        low = torch.minimum(la, lb)
        label = label.scatter_reduce(0, la, low, "amin").scatter_reduce(0, lb, low, "amin")
        while not torch.equal(label, label[label]):
            label = label[label]
    big = torch.bincount(label).argmax()
    inside = label == big
    rank = torch.cumsum(inside, 0) - 1
    a, b = a[inside[a]], b[inside[b]]
    n = int(inside.sum())
    return n, _csr(n, rank[a], rank[b], False)


def _graph(case, seed):
    """(n, row_ptr, col, directed) of a case, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["graph"]
    if kind == "chunglu":
        return (case["n"], *_chunglu(case["n"], case["deg"], gen), False)
    if kind == "ba":
        return (case["n"], *_ba(case["n"], case["deg"], gen), False)
    if kind == "rmat":
        return (1 << case["scale"], *_rmat(case["scale"], case["deg"], gen), True)
    n, (rp, col) = _grid(case["rows"], case["cols"], gen)
    return (n, rp, col, False)


def _size(case):
    """Vertices and arcs of a case's graph, as its recipe gives them."""
    if case["graph"] == "grid":
        n = case["rows"] * case["cols"]
        return n, int(0.95 * 4 * n)
    if case["graph"] == "rmat":
        return 1 << case["scale"], case["deg"] << case["scale"]
    if case["graph"] == "ba":
        return case["n"], 2 * case["deg"] * case["n"]
    return case["n"], case["deg"] * case["n"]


# ------------------------------------------------------------------- cases
def _batch_sizes(case):
    """Sizes of a batch's graphs: spread from a fifth of n up to n."""
    return [max(64, case["n"] * (20 + (i * 37) % 81) // 100) for i in range(case["count"])]


def prepare(case, seed):
    what = case["what"]
    if what == "batch":
        # resident graphs, their output arrays and the recorded batch, as a program that replays it keeps them
        count, k = case["count"], case["k"]
        handles = []
        for i, n in enumerate(_batch_sizes(case)):
            n, rp, col, directed = _graph(dict(case, n=n), seed * 1000 + i)
            handles.append(bcm.BcmGraph(rp, col, n, directed, on_device=True))
        ids = torch.zeros(count, k, dtype=torch.int32, device="cuda")
        far = torch.zeros(count, k, dtype=torch.int64, device="cuda")
        reach = torch.zeros(count, k, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        batch = bcm.BcmBatch([h.h for h in handles], [k] * count, list(zip(ids, far, reach)), stream)
        return {"what": what, "batch": batch, "handles": handles, "out": [ids, far, reach], "stream": stream}
    n, rp, col, directed = _graph(case, seed)
    state = {"what": what, "n": n, "directed": directed, "k": case.get("k", 0)}
    if what in ("topk", "farness"):
        # a resident graph, preprocessed once
        state["handle"] = bcm.BcmGraph(rp, col, n, directed, on_device=True)
        bcm.bcm_preprocess(state["handle"].h)
    elif what == "host":
        state["rp"] = rp.cpu().numpy().view(np.uint64)
        state["col"] = col.cpu().numpy().view(np.uint32)
    else:
        state["rp"], state["col"] = rp, col
    if what in ("noalloc", "farness"):
        state["far"] = torch.zeros(n, dtype=torch.int64, device="cuda")
        state["reach"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    if what == "scc":
        state["out"] = [torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)]
    return state


def run(state):
    what = state["what"]
    if what == "topk":
        ids, far, reach, _ = state["handle"].topk(state["k"])
        return {"ids": ids, "farness": far, "reach": reach}
    if what in ("graph", "host"):
        with bcm.BcmGraph(state["rp"], state["col"], state["n"], state["directed"],
                          on_device=what == "graph") as g:
            ids, far, reach, _ = g.topk(state["k"])
        return {"ids": ids, "farness": far, "reach": reach}
    if what == "farness":
        bcm.bcm_farness_all(state["handle"].h, bcm.make_options(flags=bcm.BCM_OUT_DEVICE), state["far"],
                            state["reach"])
        return {"farness": state["far"], "reach": state["reach"]}
    if what == "noalloc":
        bcm.bcm_farness_all_noalloc(state["rp"], state["col"], state["n"], state["col"].shape[0], None,
                                    state["far"], state["reach"])
        return {"farness": state["far"], "reach": state["reach"]}
    if what == "scc":
        with bcm.BcmGraph(state["rp"], state["col"], state["n"], True, on_device=True) as g:
            count = bcm.bcm_scc_bounds(g.h, *state["out"], out_on_device=True)
        return {"comp": state["out"][0], "alpha": state["out"][1], "omega": state["out"][2], "count": count}
    state["batch"].run()
    return {"ids": state["out"][0], "farness": state["out"][1], "reach": state["out"][2]}


def work(case):
    """The graph read once, the outputs written once; a textbook answer also needs one OR of a 64-source word per
    arc and 64 sources (a top-k run's searches are cut, so no number of them can be named beforehand)."""
    if case["what"] == "batch":
        sizes = [_size(dict(case, n=n)) for n in _batch_sizes(case)]
        return {"bytes": sum(4 * (n + 1) + 4 * m + 16 * case["k"] for n, m in sizes), "flops": 0}
    n, m = _size(case)
    offsets = 4 if case["what"] in ("topk", "farness") else 8   # a resident graph's are 32-bit
    graph = offsets * (n + 1) + 4 * m
    if case["what"] in ("farness", "noalloc"):
        return {"bytes": graph + 12 * n, "flops": n * m / 64}
    if case["what"] == "scc":
        return {"bytes": graph + 12 * n, "flops": 0}
    return {"bytes": graph + 16 * case["k"], "flops": 0}


# ------------------------------------------------------- the textbook answer
def _levels(n, rp, col):
    """(farness, reach) of every vertex by BFS from all of them at once, as products of 0/1 matrices (counts below
    2^24 are exact in 32 bits); whole numbers."""
    dev = rp.device
    row = torch.repeat_interleave(torch.arange(n, device=dev), rp.diff())
    adj = torch.zeros(n, n, device=dev)
    adj[row, col.long()] = 1
    seen = torch.eye(n, dtype=torch.bool, device=dev)
    front = seen.float()
    far = torch.zeros(n, dtype=torch.int64, device=dev)
    d = 0
    while True:
        d += 1
        new = (front @ adj > 0) & ~seen
        count = new.sum(1)
        if not bool(count.any()):
            return far, seen.sum(1)
        far += d * count
        seen |= new
        front = new.float()


def exact(case, seed):
    if case["what"] in ("scc", "batch") or case["graph"] == "grid" or _size(case)[0] > 17000:
        return None
    n, rp, col, _ = _graph(case, seed)
    tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        far, reach = _levels(n, rp, col)
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32
    if case["what"] in ("farness", "noalloc"):
        return {"farness": far, "reach": reach.to(torch.int32)}
    f, r = far.tolist(), reach.tolist()

    def before(a, b):   # larger (r-1)^2 / f first, equal ones by id
        x = ((r[a] - 1) ** 2 * max(f[b], 1)) - ((r[b] - 1) ** 2 * max(f[a], 1))
        return -1 if x > 0 or (x == 0 and a < b) else 1

    ids = sorted(range(n), key=functools.cmp_to_key(before))[:case["k"]]
    return {"ids": np.array(ids, np.uint32), "farness": np.array([f[i] for i in ids], np.uint64),
            "reach": np.array([r[i] for i in ids], np.uint32)}
