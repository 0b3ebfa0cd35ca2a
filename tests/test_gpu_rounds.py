"""The resident round loop against the host round loop and the oracle at the sizes where it can go wrong: degrees at the
edges of the tiles, the warp and the half-CTA classes, vertex counts around a flag word and around what a CTA takes at
a time, every weight kind and key width, each parameter that changes a round. Integers: everything must be equal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

EDGES = [1, 4, 5, 8, 9, 16, 17, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 1023, 1024]


def degrees_graph(n, degs, seed, wmax, loops=0):
    """Vertices of the given degrees (and one arc more or fewer where they meet) in a sparse random graph on n."""
    rng = np.random.default_rng(seed)
    edges = set()
    for i, d in enumerate(degs):
        if d >= n:
            continue
        others = rng.choice(np.setdiff1d(np.arange(n), [i]), d, replace=False)
        edges |= {(min(i, int(x)), max(i, int(x))) for x in others}
    edges |= {(int(a), int(b)) for a, b in np.sort(rng.integers(0, n, (n, 2)), axis=1) if a != b}
    edges = sorted(edges)
    ws = rng.integers(1, wmax + 1, len(edges)).tolist() if wmax > 1 else None
    lo = {int(v): int(rng.integers(1, wmax + 1)) for v in rng.choice(n, loops, replace=False)} if loops else None
    return synth.from_edge_list(n, edges, ws, lo)


def check(g, params):
    import paper_2507_06471_gb300 as cd
    G = cd.Graph(g.off.cuda(), g.cols.cuda(), None if g.w is None else g.w.cuda())
    out = []
    for loop in (1, 0):
        lab, rounds = G.lpa(device_loop=loop, **params)
        tr = [(t["active"], t["arcs"], t["moved"], t["deferred"], t["cands"], t["moved_arcs"]) for t in G.trace()]
        lab2, moves, rounds2 = G.local_move(device_loop=loop, **params)
        tr2 = [(t["active"], t["arcs"], t["moved"], t["deferred"], t["cands"], t["moved_arcs"]) for t in G.trace()]
        lab3, moves3, rounds3 = G.local_move(labels=lab, device_loop=loop, **params)
        lv = G.louvain(device_loop=loop, **params)
        out.append((lab.cpu().numpy(), rounds, tr, lab2.cpu().numpy(), moves, rounds2, tr2, lab3.cpu().numpy(), moves3,
                    rounds3, lv[0].cpu().numpy(), lv[1], lv[2]))
    G.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b) if isinstance(a, np.ndarray) else a == b
    return out[0]


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 613, 1131, 2048, 2049, 5000])
@pytest.mark.parametrize("wmax,loops", [(1, 0), (9, 0), (7, 11), (300_000, 1), (2_000_000_000, 0)])
def test_equals_host_loop_and_oracle(n, wmax, loops):
    g = degrees_graph(n, [d for d in EDGES if d < n // 2], n + wmax % 97, wmax, min(loops, n))
    got = check(g, {})
    off, cols, w = g.numpy()
    lab, tr = oracle.lpa(off, cols, w)
    assert np.array_equal(got[0], lab) and got[1] == tr.rounds
    lab, lv, q, _ = oracle.louvain(off, cols, w)
    assert np.array_equal(got[10], lab) and got[11] == lv and abs(got[12] - q) <= 1e-12 * max(1.0, abs(q))


@pytest.mark.parametrize("wmax,loops", [(1, 0), (9, 30), (2_000_000_000, 0)])
@pytest.mark.parametrize("degs", [[1025], [2047, 2048, 2049, 1024], [9000, 1300, 4097], [1030] * 40 + EDGES])
def test_hubs(degs, wmax, loops):
    g = degrees_graph(12_000, degs, sum(degs), wmax, loops)
    got = check(g, {})
    off, cols, w = g.numpy()
    lab, tr = oracle.lpa(off, cols, w)
    assert np.array_equal(got[0], lab) and got[1] == tr.rounds
    lab, lv, q, _ = oracle.louvain(off, cols, w)
    assert np.array_equal(got[10], lab) and got[11] == lv and abs(got[12] - q) <= 1e-12 * max(1.0, abs(q))


@pytest.mark.parametrize("n,k,p_in,p_out,wmax", [(4000, 4, "0.3", "0.02", 1), (4000, 1, "0.15", "0", 5), (3500, 40, "0.9", "0.08", 3)])
def test_many_wide_rows(n, k, p_in, p_out, wmax):
    # rows of 257 to 1,024 arcs in every CTA: few labels each, and so many that the warps' tables overflow
    g = synth.sbm(n, k, p_in, p_out, seed=n + k, wmax=wmax)
    got = check(g, {"max_iter": 12})
    off, cols, w = g.numpy()
    assert int((np.diff(off) > 256).sum()) == n
    lab, moves, tr = oracle.local_move(off, cols, w, max_iter=12)
    assert np.array_equal(got[3], lab) and got[4] == moves


def test_hub_parameters():
    g = degrees_graph(6000, [5000, 1100, 1024], 8, 3)
    for params in ({"use_frontier": 0}, {"threshold": 40}, {"tie_keep_current": 0}, {"max_iter": 2}):
        check(g, params)


@pytest.mark.parametrize("params", [{"use_frontier": 0}, {"threshold": 40}, {"tie_keep_current": 0}, {"max_iter": 1},
                                    {"max_iter": 300, "sched_seed": 77}, {"singleton_rule": 0}])
def test_parameters(params):
    check(degrees_graph(3000, EDGES, 5, 3), params)


def test_batched_equals_host_loop():
    import paper_2507_06471_gb300 as cd
    graphs = [degrees_graph(n, [d for d in EDGES + [1500] if d < n // 2], n, 4) for n in (1, 2, 40, 700, 33, 4000, 64, 3)]
    packed, vstart = synth.pack_batch(graphs)
    G = cd.Graph(packed.off.cuda(), packed.cols.cuda(), packed.w.cuda())
    G.set_batches(vstart)
    for params in ({}, {"threshold": 5}, {"max_iter": 3}, {"use_frontier": 0}):
        a, b = (G.batch_lpa(device_loop=loop, **params) for loop in (1, 0))
        assert np.array_equal(a[0].cpu().numpy(), b[0].cpu().numpy()) and np.array_equal(a[1], b[1])
        a, b = (G.batch_louvain(device_loop=loop, **params) for loop in (1, 0))
        assert np.array_equal(a[0].cpu().numpy(), b[0].cpu().numpy()) and np.array_equal(a[1], b[1])
        assert np.array_equal(a[2], b[2])
    G.close()


@pytest.mark.parametrize("isolated", [100_000, (1 << 23), (1 << 23) + 1])
def test_mostly_isolated(isolated):
    # both sides of the line from which graphs of isolated vertices take the per-round kernels
    import torch
    g = degrees_graph(2000, [300, 40, 17], 4, 3)
    alone = int((np.diff(g.numpy()[0]) == 0).sum())
    tail = torch.full((isolated - alone,), int(g.off[-1]), dtype=g.off.dtype)
    got = check(type("G", (), {"off": torch.cat([g.off, tail]), "cols": g.cols, "w": g.w}), {})
    n = len(got[0])
    lab, tr = oracle.lpa(*g.numpy())
    assert np.array_equal(got[0], np.concatenate([lab, np.arange(2000, n)])) and got[1] == tr.rounds
