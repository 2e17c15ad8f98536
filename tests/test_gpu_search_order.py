"""The paper's order of an insertion search (expand_early -1: a vertex visits its
candidates only once its support exceeds its level) over launches of many
iterations, whose records it shares with the default order, and lists on both
sides of the length up to which short ones are walked together (256 slots).
Exact comparison with the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_search import _near_regular, _pairs, _sd, cm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hub_slots", [1024, 300, -1])
def test_many_iterations_in_the_papers_order(cm, hub_slots):  # noqa: F811
    import torch
    rng = np.random.default_rng(11)
    n = 3000
    # dense blocks of a few levels: long lists, whose vertices are searched in
    # one iteration after another and fail close together
    p = np.repeat([0.8, 0.55, 0.55, 0.3], n // 4)
    i, j = np.triu_indices(n, 1)
    keep = rng.random(len(i)) < p[i] * p[j]
    e = np.stack([i[keep], j[keep]], 1).astype(np.int32)
    g = cm.CoreGraph(n, torch.from_numpy(e).cuda(), block_mode_edges=-1, hub_slots=hub_slots, expand_early=-1)
    ref = oracle.OracleGraph(n, e, mode=oracle.SUPERIOR)
    hot = rng.choice(n, 40, replace=False)
    for b in range(2):
        x = np.stack([rng.choice(hot, 900), rng.integers(0, n, 900)], 1).astype(np.int32)
        x = x[x[:, 0] != x[:, 1]]
        applied = ref.insert_edges(x)
        cores = ref.cores()
        cur = np.sort(np.asarray(ref.edges(), dtype=np.int64), 1)
        sd = _sd(n, cur[:, 0] * n + cur[:, 1], cores)
        new = x[np.sort(np.unique(np.sort(x, 1), axis=0, return_index=True)[1])]
        fresh = None
        for again in range(4):                       # the same batch: out and in again
            if fresh is not None:
                g.delete_edges(torch.from_numpy(fresh).cuda())
            before = set(map(tuple, np.sort(g.edges(), 1).tolist())) if fresh is None else before
            assert g.insert_edges(torch.from_numpy(x).cuda()) == applied
            if fresh is None:
                fresh = np.asarray([t for t in new if tuple(sorted(t)) not in before], np.int32)
            st = g.stats()
            assert st["iterations"] == ref.last_iterations() == st["grid_iterations"] > 10
            assert (g.cores() == cores).all(), (b, again)
            assert (g.superior_degrees() == sd).all(), (b, again)
    g.close()


@pytest.mark.parametrize("expand_early", [0, -1])
@pytest.mark.parametrize("d", [258, 260, 264])
def test_lists_around_the_short_limit(cm, d, expand_early):  # noqa: F811
    import torch
    rng = np.random.default_rng(d)
    n = 2 * d + 241
    cur = _near_regular(rng, n, d)
    g = cm.CoreGraph(n, torch.from_numpy(_pairs(n, cur)).cuda(), block_mode_edges=-1, expand_early=expand_early)
    deg = np.bincount(np.concatenate([cur // n, cur % n]), minlength=n)
    assert deg.min() <= 256 <= deg.max()
    for b in range(4):
        if b % 2 == 0:
            x = rng.integers(0, n, (200, 2)).astype(np.int32)
            y = x[x[:, 0] != x[:, 1]].astype(np.int64)
            new = np.unique(np.concatenate([cur, y.min(1) * n + y.max(1)]))
            assert g.insert_edges(torch.from_numpy(x).cuda()) == len(new) - len(cur)
        else:
            drop = rng.permutation(len(cur))[:200]
            assert g.delete_edges(torch.from_numpy(_pairs(n, cur[drop])).cuda()) == len(drop)
            new = np.delete(cur, drop)
        cur = new
        ref = oracle.bz(n, _pairs(n, cur))
        assert (g.cores() == ref).all(), b
        assert (g.superior_degrees() == _sd(n, cur, ref)).all(), b
    g.close()


@pytest.mark.parametrize("leave", [4, 16, 64, 400])
def test_searches_handed_from_one_block_to_the_grid(cm, leave):  # noqa: F811
    """Searches that begin in single-block waves and go on grid-wide: both
    leave the vertices' words as the other expects them."""
    rng = np.random.default_rng(leave)
    n = 4000
    x = rng.integers(0, n, (5 * n, 2))
    y = x[x[:, 0] != x[:, 1]]
    keys = np.unique(np.minimum(y[:, 0], y[:, 1]) * n + np.maximum(y[:, 0], y[:, 1]))
    e = _pairs(n, keys)
    g = cm.CoreGraph(n, e, block_mode_enter=1 << 30, block_mode_leave=leave)
    ref = oracle.OracleGraph(n, e, mode=oracle.SUPERIOR)
    hot = rng.choice(n, 60, replace=False)
    for b in range(6):
        new = np.stack([rng.choice(hot, 300), rng.integers(0, n, 300)], 1).astype(np.int32)
        new = new[new[:, 0] != new[:, 1]]
        old = np.concatenate([new[::2], e[rng.choice(len(e), 400, replace=False)]]).astype(np.int32)
        for f, r, batch in ((g.insert_edges, ref.insert_edges, new), (g.delete_edges, ref.delete_edges, old)):
            assert f(batch) == r(batch)
            assert g.stats()["iterations"] == ref.last_iterations() > 1
            assert (g.cores() == ref.cores()).all(), b
    r = g.check()
    assert [r[k] for k in ("sd_mismatches", "key_mismatches", "kcore_violations")] == [0] * 3
    g.close()
