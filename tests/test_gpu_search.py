"""The grid-mode search at the sizes where its paths meet: lists that end at a
quad, a short walk (128 slots), a scan window (512), the candidate buffer and
the default hub threshold (1024); with hub items off (lists whose candidates
overflow the buffer are scanned twice), early expansion off, and greedy
claims.  Dense random graphs have one or two core levels, so nearly every
neighbour is a candidate and a batch searches the whole graph.  Core numbers
and superior degrees are integers with one right answer: exact comparison."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cm():
    import torch
    from paper_1612_09368_gb300 import build
    build.build()
    import paper_1612_09368_gb300 as cm
    torch.cuda.set_device(0)
    return cm


def _near_regular(rng, n, d):
    """About d neighbours each: d // 2 random cyclic shifts of the vertices,
    each with a few edges missing (degrees end on both sides of d)."""
    shifts = rng.permutation(np.arange(1, (n - 1) // 2))[: max(1, d // 2)]
    v = np.arange(n)
    keys = np.concatenate([np.minimum(v, (v + s) % n) * n + np.maximum(v, (v + s) % n) for s in shifts])
    return np.unique(keys[rng.random(len(keys)) > 0.01])


def _pairs(n, keys):
    return np.stack([keys // n, keys % n], 1).astype(np.int32)


def _sd(n, keys, cores):
    edges = _pairs(n, keys)
    cu, cv = cores[edges[:, 0]], cores[edges[:, 1]]
    return np.bincount(edges[:, 0][cv >= cu], minlength=n) + np.bincount(edges[:, 1][cu >= cv], minlength=n)


@pytest.mark.parametrize("opts", [{}, {"hub_slots": -1}, {"hub_slots": 256, "expand_early": -1}, {"task_claim": 8}],
                         ids=["default", "no-hubs", "hubs-256-paper-order", "claim-8"])
@pytest.mark.parametrize("d", [4, 30, 126, 132, 508, 516, 1020, 1032, 1600])
def test_list_lengths(cm, d, opts):
    import torch
    rng = np.random.default_rng(d)
    n = max(400, 2 * d + 41)
    e = _near_regular(rng, n, d)
    g = cm.CoreGraph(n, torch.from_numpy(_pairs(n, e)).cuda(), block_mode_edges=-1, **opts)
    cur = e
    for b in range(4):
        if b % 2 == 0:
            x = rng.integers(0, n, (60 * (b + 1), 2)).astype(np.int32)
            y = x[x[:, 0] != x[:, 1]].astype(np.int64)
            new = np.unique(np.concatenate([cur, y.min(1) * n + y.max(1)]))
            assert g.insert_edges(torch.from_numpy(x).cuda()) == len(new) - len(cur)
        else:
            drop = rng.permutation(len(cur))[: 200]
            assert g.delete_edges(torch.from_numpy(_pairs(n, cur[drop])).cuda()) == len(drop)
            new = np.delete(cur, drop)
        cur = new
        ref = oracle.bz(n, _pairs(n, cur))
        assert (g.cores() == ref).all(), (d, b)
        assert (g.superior_degrees() == _sd(n, cur, ref)).all(), (d, b)
    assert g.stats()["grid_iterations"] == g.stats()["iterations"] > 0
    g.close()


@pytest.mark.parametrize("hub_slots", [1024, 300, -1])
def test_many_iterations(cm, hub_slots):
    """A batch whose edges meet at a few vertices takes dozens of iterations in
    one launch: vertices are searched again from the records that earlier
    iterations left, which new edges and risen neighbours have joined.
    Iterations, cores and superior degrees against the oracle."""
    import torch
    rng = np.random.default_rng(5)
    n = 2600
    # dense blocks of several levels, so that vertices rise into occupied ones
    p = np.repeat([0.9, 0.6, 0.35, 0.2], n // 4)
    i, j = np.triu_indices(n, 1)
    keep = rng.random(len(i)) < p[i] * p[j]
    e = np.stack([i[keep], j[keep]], 1).astype(np.int32)
    g = cm.CoreGraph(n, torch.from_numpy(e).cuda(), block_mode_edges=-1, hub_slots=hub_slots)
    ref = oracle.OracleGraph(n, e, mode=oracle.SUPERIOR)
    hot = rng.choice(n, 40, replace=False)
    for b in range(3):
        x = np.stack([rng.choice(hot, 900), rng.integers(0, n, 900)], 1).astype(np.int32)
        x = x[x[:, 0] != x[:, 1]]
        for f, r in ((g.insert_edges, ref.insert_edges), (g.delete_edges, ref.delete_edges)):
            if b == 2 and f == g.delete_edges:
                break
            assert f(torch.from_numpy(x).cuda()) == r(x)
            st = g.stats()
            assert st["iterations"] == ref.last_iterations() == st["grid_iterations"]
            cores = ref.cores()
            assert (g.cores() == cores).all(), b
            cur = np.asarray(ref.edges(), dtype=np.int64)
            cur = np.sort(cur, 1)
            assert (g.superior_degrees() == _sd(n, cur[:, 0] * n + cur[:, 1], cores)).all(), b
    assert st["iterations"] > 10
    g.close()
