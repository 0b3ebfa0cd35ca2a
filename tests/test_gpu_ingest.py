"""Ingest where its tiles of 128 arcs and its pieces meet: a row that repeats a column across such an edge has to be
noticed (the first round reads rows without repeats directly), and deg_w has to be whole for rows over several tiles.
Labels of one round depend on both. Integers: equal to the oracle's."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def repeated(p, leaves, pairs, weighted):
    """Vertex 0 joined to 1..leaves, its p-th arc repeating the column before; pairs of vertices after them."""
    x = p  # columns 1, 2, ..: arc p - 1 is vertex p
    row0 = np.concatenate([np.arange(1, p + 1), np.arange(x, leaves + 1)])
    n = 1 + leaves + 2 * pairs
    deg = np.ones(n, np.int64)
    deg[0] = len(row0)
    a = 1 + leaves + np.arange(2 * pairs)
    cols = np.concatenate([row0, np.zeros(leaves, np.int64), a ^ 1 if (1 + leaves) % 2 == 0 else ((a - 1) ^ 1) + 1])
    w = np.ones(len(cols), np.int64)
    if weighted:
        w[:] = 3
    w[len(row0) + x - 1] *= 2  # the other side carries both arcs
    off = np.concatenate([[0], np.cumsum(deg)])
    return off, cols.astype(np.int32), w.astype(np.int32)


@pytest.mark.parametrize("pairs", [40, 2_500_000])  # one tile a piece, several tiles a piece
@pytest.mark.parametrize("p", [1, 2, 3, 4, 127, 128, 129, 255, 256, 257, 511, 512, 600])
def test_repeated_column(p, pairs):
    import paper_2507_06471_gb300 as cd
    off, cols, w = repeated(p, 700, pairs, p % 2 == 0)
    G = cd.Graph(torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), torch.from_numpy(w).cuda())
    assert G.vol == int(w.sum())
    for seed in (1, 2, 3, 4):
        lab, _ = G.lpa(max_iter=1, sched_seed=seed)
        ref, _ = oracle.lpa(off, cols, w, max_iter=1, sched_seed=seed)
        assert np.array_equal(lab.cpu().numpy(), ref)
    G.close()


@pytest.mark.parametrize("wmax", [1, 2_000_000_000])
@pytest.mark.parametrize("n", [1, 33, 5000])
def test_vol_and_loops(n, wmax):
    import paper_2507_06471_gb300 as cd
    rng = np.random.default_rng(n)
    deg = rng.integers(0, 4, n) * rng.integers(0, 90, n)
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    cols = rng.integers(0, n, off[-1]).astype(np.int32)  # loops and repeats among them
    w = None if wmax == 1 else rng.integers(1, wmax, off[-1]).astype(np.int32)
    G = cd.Graph(torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), None if w is None else torch.from_numpy(w).cuda())
    ww = np.ones(len(cols), np.int64) if w is None else w.astype(np.int64)
    loop = np.repeat(np.arange(n), deg) == cols
    assert G.vol == int(ww.sum() + ww[loop].sum())
    one = torch.zeros(n, dtype=torch.int32, device="cuda")
    assert G.modularity(one) == 0.0  # one community: I = vol(V), and deg_w sums to it
    G.close()
