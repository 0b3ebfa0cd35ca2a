"""Sums over arcs split evenly over the warps (modularity and its batched and allocation-free forms) on rows that end,
start or repeat where a tile of 128 arcs does: empty rows in runs, one long row, rows of 1 to 4 arcs, offsets of the
caller's arrays that are not 16-byte aligned. Integer sums and one division, so results equal the oracle's to 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


def _star_mix(n, hub, arcs_hub, seed, wmax, loops):
    """A hub joined to `arcs_hub` vertices, pairs elsewhere, runs of isolated vertices between them."""
    rng = np.random.default_rng(seed)
    edges = {(min(hub, int(v)), max(hub, int(v))) for v in rng.choice(n, arcs_hub, replace=False) if v != hub}
    for u in range(0, n - 5, 97):
        edges.add((u, u + 1 + int(rng.integers(0, 4))))
    edges = sorted(edges)
    ws = rng.integers(1, wmax + 1, len(edges)).tolist()
    lo = {int(v): int(rng.integers(1, 4)) for v in rng.choice(n, loops, replace=False)} if loops else None
    return synth.from_edge_list(n, edges, ws if wmax > 1 else None, lo)


GRAPHS = [(2, 0, 1, 1, 0), (300, 299, 127, 1, 0), (300, 0, 128, 1, 5), (5000, 2500, 129, 7, 0), (20000, 19999, 9000, 5, 30)]


@pytest.mark.parametrize("n,hub,arcs,wmax,loops", GRAPHS)
def test_modularity_forms(n, hub, arcs, wmax, loops):
    import paper_2507_06471_gb300 as cd
    g = _star_mix(n, hub, arcs, 3 + n, wmax, loops)
    off, cols, w = g.numpy()
    rng = np.random.default_rng(1)
    G = cd.Graph(g.off.cuda(), g.cols.cuda(), None if g.w is None else g.w.cuda())
    # the allocation-free call on arrays that start 4 bytes past a 16-byte boundary
    dcols = torch.cat([torch.zeros(1, dtype=torch.int32), g.cols]).cuda()[1:]
    dw = None if g.w is None else torch.cat([torch.zeros(1, dtype=torch.int32), g.w]).cuda()[1:]
    for lab in (np.arange(n), rng.integers(0, 3, n), np.full(n, n - 1)):
        lab = lab.astype(np.int32)
        q = oracle.modularity(off, cols, w, lab)[0]
        tol = 1e-12 * max(1.0, abs(q))
        dl = torch.from_numpy(lab).cuda()
        assert abs(G.modularity(dl) - q) <= tol
        assert abs(cd.cd_modularity_noalloc(g.off.cuda(), dcols, dw, dl) - q) <= tol
    bad = torch.full((n,), n, dtype=torch.int32, device="cuda")
    for call in (lambda: G.modularity(bad), lambda: cd.cd_modularity_noalloc(g.off.cuda(), dcols, dw, bad)):
        with pytest.raises(cd.CDError) as e:
            call()
        assert e.value.status == cd.CD_EINVAL
    G.close()


def test_batched_modularity_of_many_graphs_per_tile():
    import paper_2507_06471_gb300 as cd
    graphs = [synth.from_edge_list(n, [(i, i + 1) for i in range(n - 1)]) for n in (2, 3, 5, 400, 1, 2, 7, 130)] * 3
    packed, vstart = synth.pack_batch(graphs)
    G = cd.Graph(packed.off.cuda(), packed.cols.cuda())
    G.set_batches(vstart)
    lab, levels, q = G.batch_louvain()
    lab = lab.cpu().numpy()
    for b, g in enumerate(graphs):
        off, cols, w = g.numpy()
        olab, olv, oq, _ = oracle.louvain(off, cols, w)
        assert np.array_equal(lab[vstart[b]:vstart[b + 1]], olab) and levels[b] == olv
        assert abs(q[b] - oq) <= 1e-12
    G.close()


@pytest.mark.parametrize("run", [511, 512, 543, 544, 545, 546, 577, 700, 5000])
@pytest.mark.parametrize("wmax", [1, 6])
def test_long_runs_of_empty_rows(run, wmax):
    # more rows start inside one tile than a warp marks: it searches the offsets instead, at the first and the last arcs
    # of a tile, in tiles that follow one another, and before tiles that mark again
    import paper_2507_06471_gb300 as cd
    rng = np.random.default_rng(run + wmax)
    edges, at = [], 0
    for deg in (1, 2, 126, 127, 128, 129, 3, 1, 300, 1, 1, 1):  # a vertex joined to the `deg` ones after it, then the run
        edges += [(at, at + 1 + i) for i in range(deg)]
        at += deg + 1 + run
    n = at + 1
    edges.append((0, n - 1))
    ws = rng.integers(1, wmax + 1, len(edges)).tolist() if wmax > 1 else None
    g = synth.from_edge_list(n, edges, ws, {int(v): 2 for v in rng.choice(n, 7, replace=False)})
    off, cols, w = g.numpy()
    dw = None if g.w is None else g.w.cuda()
    for _ in range(3):
        G = cd.Graph(g.off.cuda(), g.cols.cuda(), dw)
        for lab in (np.arange(n), rng.integers(0, 3, n), np.arange(n) // 7):
            lab = lab.astype(np.int32)
            q = oracle.modularity(off, cols, w, lab)[0]
            dl = torch.from_numpy(lab).cuda()
            assert abs(G.modularity(dl) - q) <= 1e-12 * max(1.0, abs(q))
            assert abs(cd.cd_modularity_noalloc(g.off.cuda(), g.cols.cuda(), dw, dl) - q) <= 1e-12 * max(1.0, abs(q))
            k, newid, coff, ccols, cw = oracle.aggregate(off, cols, w, lab)
            C, kg = G.aggregate(dl)
            goff, gcols, gw = C.download()
            assert kg == k and np.array_equal(goff, coff)
            for a, b in zip(goff[:-1], goff[1:]):
                i, j = np.argsort(gcols[a:b]), np.argsort(ccols[a:b])
                assert np.array_equal(gcols[a:b][i], ccols[a:b][j]) and np.array_equal(gw[a:b][i], cw[a:b][j])
            C.close()
        G.close()


@pytest.mark.parametrize("arc", [0, 3, 127, 128, 300])
def test_noalloc_reports_a_bad_column_before_a_bad_weight(arc):
    import paper_2507_06471_gb300 as cd
    g = _star_mix(300, 0, 250, 3, 5, 0)
    off, lab = g.off.cuda(), torch.zeros(300, dtype=torch.int32, device="cuda")
    for col, weight, status in ((-1, 0, cd.CD_EBOUNDS), (300, -7, cd.CD_EBOUNDS), (300, 2, cd.CD_EBOUNDS), (None, 0, cd.CD_EINVAL)):
        cols, w = g.cols.clone(), g.w.clone()
        if col is not None:
            cols[arc] = col
        w[arc] = weight
        with pytest.raises(cd.CDError) as e:
            cd.cd_modularity_noalloc(off, cols.cuda(), w.cuda(), lab)
        assert e.value.status == status


@pytest.mark.parametrize("n", [40, 3000, 20000])
def test_community_sums_past_32_bits(n):
    # every CTA's sum of one community takes carries out of its low word
    import paper_2507_06471_gb300 as cd
    rng = np.random.default_rng(n)
    edges = sorted({(int(a), int(b)) for a, b in np.sort(rng.integers(0, n, (4 * n, 2)), axis=1) if a != b})
    g = synth.from_edge_list(n, edges, rng.integers(2**30, 2**31 - 1, len(edges)).tolist())
    off, cols, w = g.numpy()
    G = cd.Graph(g.off.cuda(), g.cols.cuda(), g.w.cuda())
    for lab in (np.zeros(n), np.arange(n) % 3, np.arange(n)):
        lab = lab.astype(np.int32)
        q = oracle.modularity(off, cols, w, lab)[0]
        dl = torch.from_numpy(lab).cuda()
        for got in (G.modularity(dl), cd.cd_modularity_noalloc(g.off.cuda(), g.cols.cuda(), g.w.cuda(), dl)):
            assert abs(got - q) <= 1e-12 * max(1.0, abs(q))
        olab, omoves, otr = oracle.local_move(off, cols, w, labels_in=lab, max_iter=3)
        moved, moves, rounds = G.local_move(labels=dl, max_iter=3)
        assert np.array_equal(moved.cpu().numpy(), olab) and (moves, rounds) == (omoves, otr.rounds)
    G.close()
