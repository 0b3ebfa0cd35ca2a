"""Aggregation at the edges of its segment classes (8, 32, 256, 1,024 and 4,096 arcs, chunks of 4,096 above), with 32- and
64-bit weights, loops and isolated vertices, against a plain numpy summation. Integers: equal."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def graph(n, m, seed, wmax, loops):
    rng = np.random.default_rng(seed)
    e = np.sort(rng.integers(0, n, (m, 2)), axis=1)
    e = np.unique(e[e[:, 0] != e[:, 1]], axis=0)
    ws = rng.integers(1, wmax + 1, len(e)).tolist() if wmax > 1 else None
    lo = {int(v): int(rng.integers(1, wmax + 1)) for v in rng.choice(n, loops, replace=False)} if loops else None
    return synth.from_edge_list(n, e.tolist(), ws, lo)


@pytest.mark.parametrize("wmax,loops", [(1, 0), (6, 40), (1_000_000, 7)])
@pytest.mark.parametrize("sizes", [[1, 7, 8, 9, 31, 32, 33, 255, 256, 257], [1023, 1024, 1025, 2, 511], [4095, 4096, 4097, 8193, 3, 1], [30000, 9, 300]])
def test_segment_edges(sizes, wmax, loops):
    import paper_2507_06471_gb300 as cd
    n = 12_000
    g = graph(n, 40_000, len(sizes) + wmax % 7, wmax, loops)
    off, cols, w = g.numpy()
    deg = np.diff(off)
    rng = np.random.default_rng(2)
    # communities that reach the wanted arc counts one after another, named by one of their members
    labels = np.arange(n, dtype=np.int32)
    v = 0
    for want in sizes * (1 if max(sizes) > 5000 else 3):
        start, total = v, 0
        while v < n and total < want:
            total += deg[v]
            v += 1
        labels[start:v] = start
    perm = rng.permutation(n).astype(np.int32)  # scattered ids
    labels = perm[labels]
    G = cd.Graph(g.off.cuda(), g.cols.cuda(), None if g.w is None else g.w.cuda())
    coarse, k = G.aggregate(torch.from_numpy(labels).cuda())
    used = np.unique(labels)
    assert k == len(used)
    new = np.searchsorted(used, labels)
    rows = np.repeat(np.arange(n), deg)
    ww = np.ones(len(cols), np.int64) if w is None else w.astype(np.int64)
    ww = np.where(rows == cols, 2 * ww, ww)
    key = new[rows].astype(np.int64) * k + new[cols]
    uk, inv = np.unique(key, return_inverse=True)
    sums = np.zeros(len(uk), np.int64)
    np.add.at(sums, inv, ww)
    diag = uk // k == uk % k
    sums[diag] //= 2  # a loop arc carries the internal weight once
    coff, ccols, cw = coarse.download()
    ckey = np.repeat(np.arange(k), np.diff(coff)) * k + ccols
    order = np.argsort(ckey)
    assert np.array_equal(ckey[order], uk) and np.array_equal(cw[order], sums)
    assert coarse.vol == G.vol
    coarse.close()
    G.close()


@pytest.mark.parametrize("wmax", [1, 2_000_000_000])
@pytest.mark.parametrize("leaves", [20_000, 200_000])
def test_long_rows_spread_over_the_tables_that_read_them(leaves, wmax):
    # the columns of a long coarse row come in the order of the table they were merged in; read in chunks of 4,096 and
    # 1,024, they must spread over shared-memory tables of twice that many slots as any labels do (4,096 random ones have
    # 3,223 homes among 8,192 slots, 1,024 have 806 among 2,048), not crowd into a few
    import paper_2507_06471_gb300 as cd
    rng = np.random.default_rng(leaves)
    n = leaves + 1
    off = np.concatenate([[0], leaves + np.arange(leaves + 1)]).astype(np.int64)
    cols = np.concatenate([1 + np.arange(leaves), np.zeros(leaves)]).astype(np.int32)
    w = None
    if wmax > 1:
        ws = rng.integers(wmax // 2, wmax, leaves).astype(np.int32)
        w = torch.from_numpy(np.concatenate([ws, ws])).cuda()
    G = cd.Graph(torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), w)
    assert (G.vol < 2**31) == (wmax == 1)  # both widths of the segments
    coarse, k = G.aggregate(torch.arange(n, dtype=torch.int32, device="cuda"))
    coff, ccols, _ = coarse.download()
    coarse.close()
    G.close()
    assert k == n and coff[1] == leaves and np.array_equal(np.sort(ccols[:leaves]), np.arange(1, n))
    hashes = (ccols[:leaves].astype(np.uint64) * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF)
    for chunk, lg, least in ((4096, 13, 2500), (1024, 11, 600)):
        homes = hashes >> np.uint64(32 - lg)
        for at in range(0, leaves - chunk, chunk):
            assert len(np.unique(homes[at:at + chunk])) >= least, at
