"""Performance cases: what users of this library have it do, over the range of sizes it is used at.

Each case goes through the public Python entry points on a synthetic graph made on the GPU from a seed: R-MAT (skewed
degrees with hubs), planted partition (narrow degrees) or LFR-style (power-law degrees inside planted communities,
integer weights). Sizes come from the benchmark's workloads and the tests: the 10,000-vertex planted partition, the
1,000,000-vertex LFR-style graph, R-MAT scales 16 to 24, batches of 50 to 5,000 vertices a graph, the served stream.

A case's ``call`` says which entry points run:
  noalloc    cd_modularity_noalloc on caller-owned device arrays
  modularity Graph.modularity of a given partition
  solve      upload of one graph from device arrays, Louvain to convergence, release
  lpa        Label Propagation to convergence on a kept handle
  louvain    Louvain to convergence on a kept handle
  step       upload, Label Propagation and Louvain to convergence, release
  warm       Louvain local moving from an earlier partition on a kept handle
  aggregate  coarse graph of a given partition, its modularity and the next level's first local-moving round
  batch_lpa, batch_louvain   many small graphs packed block-diagonally, one call
  serve      requests on host graphs through the serving engine, submitted at once and waited for
"""
import math

import numpy as np
import torch

import paper_2507_06471_gb300 as cd

DEVICE = "cuda"


def listed():
    return [
        # A partition scored by a process that owns its device memory: the shortest call there is.
        {"name": "noalloc-lfr100k", "call": "noalloc", "graph": "lfr", "n": 100_003, "wmax": 8},
        # A partition scored on a large skewed graph that is already on the device: one pass over the arcs.
        {"name": "modularity-rmat23", "call": "modularity", "graph": "rmat", "n": 1 << 23, "ef": 16, "wmax": 1},
        # One small weighted graph per call, as a program that meets graphs one at a time: latency and host work.
        {"name": "solve-sbm600", "call": "solve", "graph": "sbm", "n": 613, "k": 12, "wmax": 4},
        # The benchmark's 10,000-vertex planted partition: rounds of a few microseconds of work each.
        {"name": "lpa-sbm10k", "call": "lpa", "graph": "sbm", "n": 10_000, "k": 100, "wmax": 1},
        # The benchmark's weighted LFR-style graph: many rounds, several levels, narrow degrees.
        {"name": "louvain-lfr1m", "call": "louvain", "graph": "lfr", "n": 1_000_000, "wmax": 8},
        # Label Propagation on a web-like graph whose labels fit in L2, hubs included.
        {"name": "lpa-rmat22", "call": "lpa", "graph": "rmat", "n": 1 << 22, "ef": 16, "wmax": 1},
        # The benchmark's step (upload, LPA, Louvain) on its R-MAT graph, at the largest scale timed here.
        {"name": "step-rmat24", "call": "step", "graph": "rmat", "n": 1 << 24, "ef": 16, "wmax": 1},
        # A graph that changed a little: local moving from the earlier partition, loops and weights so large that
        # vol(V) >= 2^31 (the 128-bit keys).
        {"name": "warm-lfr300k-wide", "call": "warm", "graph": "lfr", "n": 299_993, "wmax": 5000, "loops": True},
        # One coarsening step on its own: the way callers drive the levels by hand.
        {"name": "aggregate-rmat22", "call": "aggregate", "graph": "rmat", "n": 1 << 22, "ef": 16, "wmax": 4},
        # A hundred small unweighted graphs in one call.
        {"name": "batch-lpa-100", "call": "batch_lpa", "graph": "batch", "count": 100, "nmax": 600, "wmax": 1},
        # The benchmark's batch: weighted planted partitions of 50 to 5,000 vertices.
        {"name": "batch-louvain-1024", "call": "batch_louvain", "graph": "batch", "count": 1024, "nmax": 5000, "wmax": 4},
        # The served stream: mixed sizes and algorithms from host memory.
        {"name": "serve-48", "call": "serve", "graph": "stream", "count": 48, "nmax": 100_000, "wmax": 1},
    ]


def draw(rng):
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))

    call = rng.choice(["noalloc", "modularity", "solve", "lpa", "lpa", "louvain", "louvain", "step", "warm", "aggregate",
                       "batch_lpa", "batch_louvain", "serve"])
    wmax = rng.choice([1, 1, 4, 8, 5000])
    if call == "serve":
        return {"call": call, "graph": "stream", "count": rng.randint(8, 64), "nmax": size(1000, 200_000), "wmax": 1}
    if call in ("batch_lpa", "batch_louvain"):
        return {"call": call, "graph": "batch", "count": size(8, 1500), "nmax": size(200, 5000), "wmax": min(wmax, 8)}
    top = {"noalloc": 2_000_000, "modularity": 8_000_000, "solve": 50_000, "lpa": 4_000_000, "louvain": 3_000_000,
           "step": 2_500_000, "warm": 1_000_000, "aggregate": 4_000_000}[call]
    low = {"solve": 50, "noalloc": 1000}.get(call, 3000)
    graph = rng.choice(["rmat", "sbm", "lfr"])
    c = {"call": call, "graph": graph, "n": size(low, top), "wmax": wmax}
    if graph == "rmat":
        c["ef"] = rng.choice([8, 16])
    elif graph == "sbm":
        c["k"] = max(1, min(c["n"] // rng.randint(40, 200), 20_000))
    if call == "warm" or (wmax > 1 and rng.random() < 0.3):
        c["loops"] = rng.random() < 0.5
    return c


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _rand(gen, m, dtype=torch.float32):
    return torch.rand(m, generator=gen, device=DEVICE, dtype=dtype)


def _csr(u, v, n, wmax, gen, loops=False):
    """Symmetric CSR (rows sorted, no repeated arcs) of the undirected pairs; weights uniform in 1..wmax per edge."""
    keep = u != v
    u, v = u[keep], v[keep]
    keys = torch.unique((torch.minimum(u, v) << 32) | torch.maximum(u, v), sorted=True)
    lo, hi = keys >> 32, keys & 0xFFFFFFFF
    del u, v, keep, keys
    arcs = torch.cat([(lo << 32) | hi, (hi << 32) | lo])
    w = None
    if wmax > 1:
        e = torch.randint(1, wmax + 1, (lo.numel(),), generator=gen, device=DEVICE, dtype=torch.int32)
        w = torch.cat([e, e])
    if loops:
        ids = torch.arange(n, device=DEVICE, dtype=torch.int64)
        arcs = torch.cat([arcs, (ids << 32) | ids])
        lw = torch.randint(1, wmax + 1, (n,), generator=gen, device=DEVICE, dtype=torch.int32)
        w = torch.cat([lw.new_ones(arcs.numel() - n) if w is None else w, lw])
    del lo, hi
    if w is None:
        arcs = torch.sort(arcs).values
    else:
        arcs, order = torch.sort(arcs)
        w = w[order]
    off = torch.searchsorted(arcs, torch.arange(n + 1, device=DEVICE, dtype=torch.int64) << 32)
    return off, (arcs & 0xFFFFFFFF).to(torch.int32), w


def _rmat_pairs(n, ef, gen):
    """Edge factor * 2^scale R-MAT edges (0.57, 0.19, 0.19, 0.05) at scale = ceil(log2 n); endpoints >= n rejected."""
    scale = max(1, (n - 1).bit_length())
    m = ef << scale
    u = torch.zeros(m, dtype=torch.int32, device=DEVICE)
    v = torch.zeros(m, dtype=torch.int32, device=DEVICE)
    for _ in range(scale):
        x = _rand(gen, m)
        low = x >= 0.76
        u = (u << 1) | low
        v = (v << 1) | (((x >= 0.57) & ~low) | (x >= 0.95))
    keep = (u < n) & (v < n)
    return u[keep].to(torch.int64), v[keep].to(torch.int64)


def _planted_pairs(ns, ks, p_in, p_out, gen):
    """Planted partitions of ns[b] vertices in ks[b] blocks side by side, ids shuffled inside each graph: pairs sampled
    with the expected counts of p_in inside and p_out across blocks. Returns (u, v, block id of every vertex)."""
    ns, ks = np.asarray(ns, np.int64), np.asarray(ks, np.int64)
    base = np.concatenate([[0], np.cumsum(ns)])
    blk = np.repeat(np.arange(len(ns)), ks)                          # graph of every block
    j = np.arange(len(blk)) - np.repeat(np.cumsum(ks) - ks, ks)      # its number inside the graph
    bs = np.maximum(ns // ks, 1)[blk]
    bbase = base[blk] + j * bs
    size = np.where(j == ks[blk] - 1, ns[blk] - j * bs, bs)
    m_in = np.rint(p_in * size * (size - 1) / 2).astype(np.int64)
    m_out = np.rint(p_out * ns * (ns - 1) / 2).astype(np.int64)
    first = torch.from_numpy(np.concatenate([np.repeat(bbase, m_in), np.repeat(base[:-1], m_out)])).to(DEVICE)
    span = torch.from_numpy(np.concatenate([np.repeat(size, m_in), np.repeat(ns, m_out)])).to(DEVICE)
    u = first + (_rand(gen, first.numel(), torch.float64) * span).to(torch.int64)
    v = first + (_rand(gen, first.numel(), torch.float64) * span).to(torch.int64)
    n = int(base[-1])
    graph = torch.from_numpy(np.repeat(np.arange(len(ns)), ns)).to(DEVICE)
    perm = torch.argsort(graph + _rand(gen, n, torch.float64) * 0.999)  # a shuffle inside every graph
    block = torch.empty(n, dtype=torch.int64, device=DEVICE)
    block[perm] = torch.from_numpy(np.repeat(np.arange(len(blk)), size)).to(DEVICE)
    return perm[u], perm[v], block, base


def _powerlaw(gen, count, tau, lo, hi):
    k = torch.arange(lo, hi + 1, device=DEVICE, dtype=torch.float64)
    cdf = torch.cumsum(k ** -tau, 0)
    return lo + torch.searchsorted(cdf / cdf[-1], _rand(gen, count, torch.float64)).clamp(max=hi - lo)


def _lfr_pairs(n, gen):
    """LFR-style: degrees ~ k^-2.5 on [5, 1000], community sizes ~ s^-1.5 on [20, 5000], mixing 0.3, wired by
    configuration models inside and across communities. Returns (u, v, community of every vertex)."""
    deg = _powerlaw(gen, n, 2.5, 5, min(1000, max(6, n // 4)))
    size = _powerlaw(gen, n // 20 + 1, 1.5, 20, min(5000, max(21, n // 4)))
    ends = torch.cumsum(size, 0)
    comm = torch.searchsorted(ends, torch.arange(n, device=DEVICE), right=True)
    comm = comm[torch.argsort(_rand(gen, n, torch.float64))]
    kin = torch.minimum(torch.round(0.7 * deg).to(torch.int64), size[comm] - 1)

    def wire(stubs, group):
        order = torch.argsort(group + _rand(gen, stubs.numel(), torch.float64) * 0.999)
        s, g = stubs[order], group[order]
        m = s.numel() // 2 * 2
        a, b, same = s[0:m:2], s[1:m:2], g[0:m:2] == g[1:m:2]
        return a[same], b[same]

    ids = torch.arange(n, device=DEVICE)
    inner = torch.repeat_interleave(ids, kin)
    outer = torch.repeat_interleave(ids, deg - kin)
    a, b = wire(inner, comm[inner])
    c, d = wire(outer, torch.zeros_like(outer))
    return torch.cat([a, c]), torch.cat([b, d]), comm


def _graph(case, gen):
    """(off, cols, w, planted or None) on the device."""
    n, planted = case["n"], None
    if case["graph"] == "rmat":
        u, v = _rmat_pairs(n, case["ef"], gen)
    elif case["graph"] == "sbm":
        s = max(n // case["k"], 2)  # about ten arcs a vertex inside its block and ten across
        u, v, planted, _ = _planted_pairs([n], [case["k"]], min(1.0, 10 / s), min(1.0, 10 / n), gen)
    else:
        u, v, planted = _lfr_pairs(n, gen)
    off, cols, w = _csr(u, v, n, case["wmax"], gen, bool(case.get("loops")))
    return off, cols, w, planted


def _partition(off, cols, planted, n, gen):
    """A partition as a caller has it: the planted one with one vertex in twenty astray, or, without one, half of the
    vertices joining a random neighbour (what a first round of moves gives). Labels are vertex ids."""
    ids = torch.arange(n, device=DEVICE)
    if planted is not None:
        rep = torch.full((int(planted.max()) + 1,), n, device=DEVICE, dtype=torch.int64)
        rep.scatter_reduce_(0, planted, ids, "amin")  # a community goes by its smallest member
        lab = rep[planted]
        astray = _rand(gen, n) < 0.05
        other = torch.randint(0, n, (n,), generator=gen, device=DEVICE)
        return torch.where(astray, lab[other], lab).to(torch.int32)
    deg = off[1:] - off[:-1]
    pick = off[:-1] + (_rand(gen, n, torch.float64) * deg).to(torch.int64)
    nb = cols[pick.clamp(max=max(cols.numel() - 1, 0))].to(torch.int64)
    move = (deg > 0) & (_rand(gen, n) < 0.5)
    return torch.where(move, nb, ids).to(torch.int32)


def _batch_sizes(case):
    """Vertices and blocks per graph of a batch or stream; fixed per case, so that seeds compare."""
    r = np.random.RandomState(case["count"] * 7919 + case["nmax"])
    lo = 100 if case["graph"] == "stream" else 50
    ns = np.exp(r.uniform(math.log(lo), math.log(case["nmax"] + 1), case["count"])).astype(np.int64)
    ks = np.minimum(r.randint(2, 51, case["count"]), ns // 2)
    return ns, ks, r


def prepare(case, seed):
    gen = _gen(seed)
    call = case["call"]
    params = cd.cd_params_default()
    if call == "serve":
        ns, ks, r = _batch_sizes(case)
        requests = []
        for n, k in zip(ns.tolist(), ks.tolist()):
            kind = cd.CD_REQ_LOUVAIN if r.rand() < 0.7 else cd.CD_REQ_LPA
            if r.rand() < 0.5:
                u, v = _rmat_pairs(n, 8, gen)
            else:
                u, v, _, _ = _planted_pairs([n], [k], min(1.0, 15 / max(n // k, 15)), min(1.0, 1 / n), gen)
            off, cols, _ = _csr(u, v, n, 1, gen)
            requests.append((kind, off.cpu().numpy(), cols.cpu().numpy()))
        return {"call": call, "server": cd.Server(params, slots=4, small_n=8192, batch_arcs=1 << 22), "requests": requests}
    if call in ("batch_lpa", "batch_louvain"):
        ns, ks, _ = _batch_sizes(case)
        u, v, _, base = _planted_pairs(ns, ks, 0.2, 0.002, gen)
        off, cols, w = _csr(u, v, int(base[-1]), case["wmax"], gen)
        g = cd.Graph(off, cols, w)
        g.set_batches(base)
        return {"call": call, "params": params, "g": g}
    off, cols, w, planted = _graph(case, gen)
    state = {"call": call, "params": params}
    if call in ("noalloc", "solve", "step"):
        state["csr"] = (off, cols, w)
    else:
        state["g"] = cd.Graph(off, cols, w)
    if call in ("noalloc", "modularity", "aggregate", "warm"):
        state["labels"] = _partition(off, cols, planted, case["n"], gen)
    if call == "aggregate":
        state["newid"] = torch.empty_like(state["labels"])
        state["one"] = cd.cd_params_default(max_iter=1)
    return state


def run(state):
    call = state["call"]
    if call == "noalloc":
        off, cols, w = state["csr"]
        return {"q": cd.cd_modularity_noalloc(off, cols, w, state["labels"])}
    if call == "modularity":
        return {"q": state["g"].modularity(state["labels"])}
    if call == "solve":
        g = cd.Graph(*state["csr"])
        labels, levels, q = g.louvain(state["params"])
        g.close()
        return {"labels": labels, "levels": levels, "q": q}
    if call == "lpa":
        labels, rounds = state["g"].lpa(state["params"])
        return {"labels": labels, "rounds": rounds}
    if call == "louvain":
        labels, levels, q = state["g"].louvain(state["params"])
        return {"labels": labels, "levels": levels, "q": q}
    if call == "step":
        g = cd.Graph(*state["csr"])
        lpa, rounds = g.lpa(state["params"])
        labels, levels, q = g.louvain(state["params"])
        g.close()
        return {"lpa": lpa, "rounds": rounds, "labels": labels, "levels": levels, "q": q}
    if call == "warm":
        labels, moves, rounds = state["g"].local_move(state["params"], labels=state["labels"])
        return {"labels": labels, "moves": moves, "rounds": rounds}
    if call == "aggregate":
        coarse, k = state["g"].aggregate(state["labels"], state["newid"])
        alone = torch.arange(k, dtype=torch.int32, device=DEVICE)
        q = coarse.modularity(alone)
        labels, moves, _ = coarse.local_move(state["one"])
        composed = labels[state["newid"][state["labels"]]]  # the next level's communities of the input's vertices
        out = {"newid": state["newid"], "k": k, "arcs": coarse.nnz, "vol": coarse.vol, "q": q, "labels": composed,
               "moves": moves}
        coarse.close()
        return out
    if call == "batch_lpa":
        labels, rounds = state["g"].batch_lpa(state["params"])
        return {"labels": labels, "rounds": rounds}
    if call == "batch_louvain":
        labels, levels, q = state["g"].batch_louvain(state["params"])
        return {"labels": labels, "levels": levels, "q": q}
    server = state["server"]
    ids = [server.submit(kind, off, cols) for kind, off, cols in state["requests"]]
    done = [server.result(i) for i in ids]
    return {"labels": np.concatenate([lab for lab, _ in done]), "iters": np.array([res.iters for _, res in done]),
            "q": np.array([res.q for _, res in done])}


def _arcs(case):
    """Expected arcs of a case's graph or graphs, before repeated pairs fall out."""
    if case["graph"] == "batch":
        ns, ks, _ = _batch_sizes(case)
        return float(np.sum(0.2 * ns * (ns / ks - 1) + 0.002 * ns * ns))
    if case["graph"] == "stream":
        return 16.0 * float(np.sum(_batch_sizes(case)[0]))
    per = {"rmat": 2 * case.get("ef", 0) * 0.94, "sbm": 20.0, "lfr": 12.5}[case["graph"]]
    return case["n"] * (per + (1 if case.get("loops") else 0))


def work(case):
    """Bytes of one pass: the CSR (offsets, columns, weights) and any given partition read once, the labels written
    once. Integer work is not counted."""
    n = case.get("n") or float(np.sum(_batch_sizes(case)[0]))
    graph = 8 * n + _arcs(case) * (4 + (4 if case["wmax"] > 1 or case.get("loops") else 0))
    given = 4 * n if case["call"] in ("noalloc", "modularity", "warm", "aggregate") else 0
    out = 0 if case["call"] in ("noalloc", "modularity") else 8 * n if case["call"] in ("step", "aggregate") else 4 * n
    return {"bytes": graph + given + out, "flops": 0}


def exact(case, seed):
    """Modularity where the partition is an input: integer sums in 64 bits, the quotient in 64-bit floating point."""
    if case["call"] not in ("noalloc", "modularity", "aggregate"):
        return None
    gen = _gen(seed)
    off, cols, w, planted = _graph(case, gen)
    lab = _partition(off, cols, planted, case["n"], gen).to(torch.int64)
    rows = torch.repeat_interleave(torch.arange(case["n"], device=DEVICE), off[1:] - off[:-1])
    w = torch.ones_like(rows) if w is None else w.to(torch.int64)
    w = torch.where(rows == cols, 2 * w, w)
    inside = int(w[lab[rows] == lab[cols.to(torch.int64)]].sum())
    vol = torch.zeros(case["n"], dtype=torch.int64, device=DEVICE).index_add_(0, lab[rows], w)
    total = int(vol.sum())
    q = 0.0 if total == 0 else inside / total - float(((vol.to(torch.float64) / total) ** 2).sum())
    return {"q": q} if case["call"] != "aggregate" else \
        {"newid": None, "k": None, "arcs": None, "vol": None, "q": q, "labels": None, "moves": None}
