"""The three forms of the round loop (one resident kernel, one captured graph, the host loop) on graphs small enough for
the resident one: which form a run takes, and equal results of the captured one with every kind of hub table and key.
Integers: everything must be equal."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

KEYS = ("level", "round", "active", "arcs", "moved", "deferred", "cands", "moved_arcs")


def hub_graph(wmax, loops):
    """Two hubs (1,500 and 3,000 arcs) over a planted partition, weights up to wmax, loops on some vertices."""
    rng = np.random.default_rng(wmax % 1000 + loops)
    base = synth.sbm(6000, 60, "0.08", "0.0005", seed=9)
    bu = np.repeat(np.arange(base.n), np.diff(base.off.numpy()))
    edges = {(int(a), int(b)) for a, b in zip(bu, base.cols.numpy()) if a < b}
    for hub, d in ((0, 1500), (1, 3000)):
        edges |= {(hub, int(x)) for x in rng.choice(np.arange(2, base.n), d, replace=False)}
    edges = sorted(edges)
    ws = rng.integers(max(1, wmax // 2), wmax + 1, len(edges)).tolist() if wmax > 1 else None
    lo = {int(v): int(rng.integers(1, wmax + 1)) for v in rng.choice(base.n, loops, replace=False)} if loops else None
    return synth.from_edge_list(base.n, edges, ws, lo)


def upload(g):
    import paper_2507_06471_gb300 as cd
    return cd.Graph(g.off.cuda(), g.cols.cuda(), None if g.w is None else g.w.cuda())


def run(G, loop, call, **params):
    """(results, kernels launched) of one call."""
    import paper_2507_06471_gb300 as cd
    before = cd.cd_launch_count()
    out = getattr(G, call)(device_loop=loop, **params)
    launches = cd.cd_launch_count() - before
    out = [x.cpu().numpy() if torch.is_tensor(x) else x for x in out]
    return out, [{k: t[k] for k in KEYS} for t in G.trace()], launches


# packed tables; loops; 128-bit keys with packed tables (vol(V) >= 2^31 but every deg_w < 2^32); two-word tables
@pytest.mark.parametrize("wmax,loops", [(1, 0), (7, 40), (100_000, 0), (2_000_000_000, 3)])
@pytest.mark.parametrize("call", ["lpa", "local_move", "louvain"])
def test_captured_graph(wmax, loops, call):
    g = hub_graph(wmax, loops)
    off, cols, w = g.numpy()
    dw, vol = oracle.degw(off, cols, w)
    assert (vol >= 2**31) == (wmax >= 100_000) and (dw.max() >= 2**32) == (wmax > 10**9)
    G = upload(g)
    for loop in (0, 1, 2):  # lays the structures of the form out
        getattr(G, call)(device_loop=loop)
    res = {loop: run(G, loop, call) for loop in (0, 1, 2)}
    few = {loop: run(G, loop, call, max_iter=4) for loop in (0, 1, 2)}
    G.close()
    for r in (res, few):
        for loop in (1, 2):
            for a, b in zip(r[loop][0], r[0][0]):
                assert np.array_equal(a, b)
            assert r[loop][1] == r[0][1]
    if call != "louvain":
        # launches: the resident loop's two kernels, a captured graph's however many rounds it runs, the host loop's more
        # with every round
        assert res[1][2] == few[1][2] <= 3 < few[2][2] == res[2][2] < res[0][2]
        assert few[0][2] < res[0][2]
    if call == "lpa":
        lab, tr = oracle.lpa(off, cols, w)
        assert np.array_equal(res[2][0][0], lab) and res[2][0][1] == tr.rounds
    elif call == "local_move":
        lab, moves, tr = oracle.local_move(off, cols, w)
        assert np.array_equal(res[2][0][0], lab) and res[2][0][1:] == [moves, tr.rounds]
    else:
        lab, lv, q, _ = oracle.louvain(off, cols, w)
        assert np.array_equal(res[2][0][0], lab) and res[2][0][1] == lv


@pytest.mark.parametrize("loop", [3, -1, 0x10001, 0x10004, 0x10040])
def test_other_values_of_device_loop_are_the_default(loop):
    # no value of the public field stands for the serving engine's workers, which take no captured graphs
    import paper_2507_06471_gb300 as cd
    graphs = [synth.sbm(n, 5, "0.2", "0.002", seed=n, wmax=3) for n in (300, 900, 80)]
    packed, vstart = synth.pack_batch(graphs)
    G = cd.Graph(packed.off.cuda(), packed.cols.cuda(), packed.w.cuda())
    G.set_batches(vstart)
    G.batch_lpa(threshold=3)
    want, trace, launches = run(G, 1, "batch_lpa", threshold=3)
    got = run(G, loop, "batch_lpa", threshold=3)
    host = run(G, 0, "batch_lpa", threshold=3)
    G.close()
    assert np.array_equal(got[0][0], want[0]) and list(got[0][1]) == list(want[1]) and got[1] == trace
    assert got[2] == launches != host[2]


def set_loop(G, polls, ctas):
    import ctypes
    import paper_2507_06471_gb300 as cd
    f = cd.lib().cd_test_resident_loop
    f.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64]
    assert f(G.h, polls, ctas) == cd.CD_OK


@pytest.mark.parametrize("hubs", [False, True])
@pytest.mark.parametrize("call", ["lpa", "local_move"])
def test_wait_that_runs_out(hubs, call):
    # a barrier that gives up at its first look ends the run with CD_ETIMEOUT; the handle's next run is right, hub tables
    # cut short included
    import paper_2507_06471_gb300 as cd
    g = hub_graph(5, 0) if hubs else synth.sbm(20_000, 100, "0.08", "0.0005", seed=4, wmax=5)
    assert len(g.cols) > 100 * 512  # a hundred CTAs or more, which do not all arrive at once
    G = upload(g)
    want = run(G, 0, call)
    for _ in range(2):
        set_loop(G, 1, 0)
        with pytest.raises(cd.CDError) as e:
            run(G, 1, call)
        assert e.value.status == cd.CD_ETIMEOUT
        set_loop(G, 0, 0)
        got = run(G, 1, call)
        assert got[1] == want[1] and all(np.array_equal(a, b) for a, b in zip(got[0], want[0]))
    G.close()


@pytest.mark.parametrize("hubs", [False, True])
def test_launch_that_is_refused(hubs):
    # more CTAs than fit at once: the runtime refuses the launch and the per-round kernels take the run
    import paper_2507_06471_gb300 as cd
    g = hub_graph(5, 3) if hubs else synth.sbm(5000, 20, "0.05", "0.0005", seed=4, wmax=5)
    G = upload(g)
    start = torch.arange(g.n, dtype=torch.int32, device="cuda") // 3
    calls = [("lpa", {}), ("local_move", {}), ("local_move", {"labels": start}), ("louvain", {})]
    want = [run(G, 0, call, **kw) for call, kw in calls]
    set_loop(G, 0, 32_000)
    got = [run(G, 1, call, **kw) for call, kw in calls]
    G.close()
    for a, b in zip(got, want):
        assert a[1] == b[1] and all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
    assert all(a[2] > 20 for a in got)  # a kernel or more a round
    # a batched run, whose graphs stop by themselves
    graphs = [synth.sbm(n, 5, "0.2", "0.002", seed=n, wmax=3) for n in (300, 900, 80)]
    packed, vstart = synth.pack_batch(graphs)
    B = cd.Graph(packed.off.cuda(), packed.cols.cuda(), packed.w.cuda())
    B.set_batches(vstart)
    for call in ("batch_lpa", "batch_louvain"):
        want = run(B, 0, call)
        set_loop(B, 0, 32_000)
        got = run(B, 1, call)
        set_loop(B, 0, 0)
        assert got[1] == want[1] and all(np.array_equal(x, y) for x, y in zip(got[0], want[0]))
    B.close()


@pytest.mark.parametrize("hubs", [False, True])
def test_autotune_prepares_what_its_runs_use(hubs):
    # the kernels launched are those of the same runs by hand: nothing is laid out that no run uses
    import paper_2507_06471_gb300 as cd
    g = hub_graph(5, 3) if hubs else synth.sbm(5000, 20, "0.05", "0.0005", seed=4, wmax=5)
    A, B = upload(g), upload(g)
    before = cd.cd_launch_count()
    best = cd.cd_autotune(A.h, cd.cd_params_default(), 2)
    tuned = cd.cd_launch_count() - before
    before = cd.cd_launch_count()
    for t_warp in (64, 128, 256):
        for t_hub in (512, 1024, 2048, 4096):
            cd.cd_graph_set_bins(B.h, t_warp, t_hub)
            B.lpa(max_iter=2)
            B.local_move(max_iter=2)
    cd.cd_graph_set_bins(B.h, *best)
    by_hand = cd.cd_launch_count() - before
    lab, rounds = A.lpa()
    olab, otr = oracle.lpa(*g.numpy())
    A.close()
    B.close()
    assert tuned == by_hand
    assert rounds == otr.rounds and np.array_equal(lab.cpu().numpy(), olab)


def graph_of(arcs, mean, hub):
    """A random graph of exactly `arcs` arcs, of mean degree `mean` or so, with a hub of 1,500 arcs or without."""
    n = arcs // mean
    gen = torch.Generator(device="cuda")
    gen.manual_seed(arcs % 1000 + mean)
    u, v = torch.randint(1, n, (2, int(arcs * 0.53)), generator=gen, device="cuda")
    keys = synth.canonical_keys(u[u != v], v[u != v])
    star = torch.arange(1, 1501 if hub else 1, device="cuda")  # 0 is in no pair: keys (0, leaf)
    m = arcs // 2 - len(star)
    assert len(keys) >= m
    keys = torch.sort(torch.cat([keys[torch.randperm(len(keys), generator=gen, device="cuda")[:m]], star])).values
    return synth.csr_from_edge_keys(keys, n, None)


# (arcs the resident loop takes at most, mean degree, hub, call, use_frontier)
LINES = [(1 << 23, 40, True, "lpa", 1), (1 << 22, 40, True, "local_move", 1), (1 << 22, 40, True, "lpa", 0),
         (1 << 21, 40, True, "local_move", 0), (1 << 24, 40, False, "local_move", 1), (1 << 24, 40, False, "lpa", 0),
         (1 << 23, 40, False, "local_move", 0), (1 << 23, 12, False, "local_move", 0), (1 << 25, 40, False, "lpa", 1)]


@pytest.mark.parametrize("most,mean,hub,call,frontier", LINES)
def test_resident_loop_up_to_so_many_arcs(most, mean, hub, call, frontier):
    for arcs in (most, most + 2):
        g = graph_of(arcs, mean, hub)
        G = upload(g)
        assert G.nnz == arcs
        getattr(G, call)(use_frontier=frontier, max_iter=3)  # lays the structures out
        a, b = (run(G, loop, call, use_frontier=frontier, max_iter=3) for loop in (1, 0))
        G.close()
        assert a[1] == b[1] and all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
        assert (a[2] == 2) == (arcs <= most) and (a[2] == b[2]) == (arcs > most)


@pytest.mark.parametrize("mean,call", [(3, "lpa"), (3, "local_move"), (20, "lpa")])
def test_resident_loop_of_low_degrees_has_no_such_line(mean, call):
    G = upload(graph_of((1 << 25) + 1000, mean, False))
    a, b = (run(G, loop, call, max_iter=3) for loop in (1, 0))
    G.close()
    assert a[2] == 2 and a[1] == b[1] and all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))


@pytest.mark.parametrize("frontier", [0, 1])
def test_resident_loop_of_batches_up_to_so_many_arcs(frontier):
    for arcs in (1 << 24, (1 << 24) + 2):
        g = graph_of(arcs, 40, False)
        G = upload(g)
        G.set_batches(np.array([0, g.n]))
        kw = dict(use_frontier=frontier, max_iter=3, max_levels=1)
        G.batch_louvain(**kw)
        a, b, c = (run(G, loop, "batch_louvain", **kw) for loop in (1, 0, 2))
        G.close()
        assert a[1] == b[1] and all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
        assert (a[2] == c[2]) == (frontier == 0 and arcs > 1 << 24)
