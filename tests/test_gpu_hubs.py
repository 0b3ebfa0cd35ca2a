"""Hub histograms of the per-round kernels where a table or the update log runs out: the run must still equal the oracle
round for round. Integers: everything must be equal. Each test first shows with the oracle that its graph gets there."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


def upload(g, t_hub=None):
    import paper_2507_06471_gb300 as cd
    G = cd.Graph(g.off.cuda(), g.cols.cuda(), None if g.w is None else g.w.cuda())
    if t_hub:
        cd.cd_graph_set_bins(G.h, 256, t_hub)
    return G


def same_trace(G, otr):
    for f in ("moved", "deferred", "active", "arcs", "cands", "moved_arcs"):
        assert [t[f] for t in G.trace()] == list(getattr(otr, f)), f


def table_slots(deg):
    return deg + deg // 2 + 64


# the host loop; the captured graph (rows of 1,025 to 4,096 arcs that are no hubs keep a graph from the resident loop)
FORMS = [(0, None), (0, 4096), (2, 4096)]


@pytest.mark.parametrize("wmax", [1, 5])
def test_log_full_in_the_round_that_builds_by_items(wmax):
    # a hub too large for a cluster's shared memory, and a majority of isolated vertices so that round 0 is not a heavy
    # one: round 1 builds the hub by items and logs more updates to it than the log holds
    n, leaves, deg = 300_000, 100_000, 80_000
    rng = np.random.default_rng(1)
    hub = 1 + rng.choice(leaves, deg, replace=False)
    e = rng.integers(1, leaves + 1, (leaves, 2))
    wide = rng.integers(1, leaves + 1, 2000)
    u = np.concatenate([np.zeros(deg, np.int64), e[:, 0], np.full(2000, 1)])
    v = np.concatenate([hub, e[:, 1], wide])
    keys = synth.canonical_keys(torch.from_numpy(u[u != v]), torch.from_numpy(v[u != v]))
    g = synth.csr_from_edge_keys(keys, n, synth.edge_weights(keys, 3, wmax) if wmax > 1 else None)
    off, cols, w = g.numpy()
    d = np.diff(off)
    assert d[0] == deg and 1024 < d[1] < 4096 and (d > 1024).sum() == 2
    assert table_slots(deg) > 8 * 12288  # the largest cluster build
    after = [oracle.lpa(off, cols, w, max_iter=k)[0] for k in (1, 2)]
    assert 4 * (after[0] != np.arange(n)).sum() <= n  # round 1 updates the histograms
    records = (after[1] != after[0])[cols[off[0]:off[1]]].sum()
    assert records > (table_slots(deg) + table_slots(int(d[1]))) * 2 // 3 // 4  # more than the log holds
    olab, otr = oracle.lpa(off, cols, w)
    for loop, t_hub in FORMS:
        G = upload(g, t_hub)
        for _ in range(5):
            lab, rounds = G.lpa(device_loop=loop)
            assert rounds == otr.rounds and np.array_equal(lab.cpu().numpy(), olab)
            same_trace(G, otr)
        G.close()


def scattering_graph(degs, weighted):
    """Hubs of the given degrees. Each hub and its leaves start in one community; a leaf is tied more closely to a pair
    of its own (unit weights) or to one vertex (weighted), which start in a community each, so that leaves scatter."""
    us, vs, ws, lab = [], [], [], []
    at = len(degs)
    lab = list(range(len(degs)))
    per = 2 if weighted else 3  # vertices per leaf
    for h, d in enumerate(degs):
        leaf = at + per * np.arange(d)
        us += [np.full(d, h), leaf] + ([] if weighted else [leaf, leaf + 1])
        vs += [leaf, leaf + 1] + ([] if weighted else [leaf + 2, leaf + 2])
        ws += [np.full(d, 1), np.full(d, 9)]
        block = np.empty((d, per), np.int64)
        block[:, 0] = h
        block[:, 1:] = (leaf + 1)[:, None]
        lab += block.ravel().tolist()
        at += per * d
    u, v = (torch.from_numpy(np.concatenate(x)) for x in (us, vs))
    keys = synth.canonical_keys(u, v)
    w = None
    if weighted:
        # weights in the order of the sorted keys
        raw = torch.minimum(u, v) << 32 | torch.maximum(u, v)
        order = torch.argsort(raw)
        assert torch.equal(raw[order], keys)
        w = torch.from_numpy(np.concatenate(ws)).to(torch.int32)[order]
    return synth.csr_from_edge_keys(keys, at, w), np.array(lab, np.int32)


def scatters(g, lab, degs):
    """Does every hub see one label in round 0 and, after it, more than its rebuild lays out slots for?"""
    off, cols, w = g.numpy()
    one = oracle.local_move(off, cols, w, max_iter=1, labels_in=lab)[0]
    for h, d in enumerate(degs):
        nb = cols[off[h]:off[h + 1]]
        slots = 2 * 1 + 256
        if len(nb) != d or len(set(lab[nb].tolist())) != 1 or slots >= table_slots(d) or len(np.unique(one[nb])) <= slots:
            return False
    return True


# a hub for each build class of the undersized rebuild: 256 threads, 512, clusters of 2, 4 and 8
@pytest.mark.parametrize("degs", [[1100], [8149, 1500], [20_000], [40_000], [80_000], [140_000], [1100, 20_000, 40_000, 80_000]])
@pytest.mark.parametrize("weighted", [False, True])
def test_rebuild_that_runs_out_of_slots(degs, weighted):
    g, start = scattering_graph(degs, weighted)
    assert scatters(g, start, degs)
    off, cols, w = g.numpy()
    olab, omoves, otr = oracle.local_move(off, cols, w, labels_in=start)
    dev = torch.from_numpy(start).cuda()
    for loop, t_hub in ((0, None), (1, None), (2, None)):
        G = upload(g, t_hub)
        for _ in range(2):
            lab, moves, rounds = G.local_move(labels=dev, device_loop=loop)
            assert (moves, rounds) == (omoves, otr.rounds) and np.array_equal(lab.cpu().numpy(), olab)
            same_trace(G, otr)
        G.close()


def test_retried_rebuilds_count_as_builds():
    degs = [1100, 20_000, 60_000]
    g, start = scattering_graph(degs, True)
    assert scatters(g, start, degs)
    G = upload(g)
    G.local_move(labels=torch.from_numpy(start).cuda(), device_loop=0, max_iter=2, timing=1)
    p = {x["name"]: x for x in G.profile()}
    G.close()
    assert p["hub_prepare"]["alg_bytes"] == 8.0 * len(degs) * p["hub_prepare"]["launches"]  # nothing cleared or compacted
    # round 0 reads each row once, round 1 twice (the try and the rebuild by items): 12 bytes an arc; a retried table is
    # cleared whole
    assert p["hub_build"]["alg_bytes"] > 12.0 * 3 * sum(degs) + 8.0 * sum(table_slots(d) for d in degs)
