"""Small batches take their ingest in one launch: validation, dedupe, the filter
against the index, lists that are compacted in place or moved, and the pool
running short, at and around the size where the separate kernels take over
(1,024 edges).  Exact comparison with the oracle."""
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


def _same(g, ref):
    assert (g.cores() == ref.cores()).all()
    r = g.check()
    assert [r[k] for k in ("sd_mismatches", "key_mismatches", "degree_mismatches", "bad_neighbour_ids",
                           "kcore_violations")] == [0] * 5
    got = np.sort(g.edges(), 1)
    want = np.sort(np.asarray(ref.edges()), 1)
    assert set(map(tuple, got.tolist())) == set(map(tuple, want.tolist()))


@pytest.mark.parametrize("k", [1, 2, 31, 33, 1023, 1024, 1025, 3000])
@pytest.mark.parametrize("slack", [0, 25])
def test_sizes(cm, k, slack):
    """Repeats, reversed pairs, self-loops, edges that are there already; the
    same pairs again and again (lists fill with holes); every list can overflow
    at once (slack 0) and the pool runs short."""
    rng = np.random.default_rng(1000 * slack + k)
    n = 700
    base = rng.integers(0, n, (1500, 2)).astype(np.int32)
    g = cm.CoreGraph(n, base, slack_pct=slack)
    ref = oracle.OracleGraph(n, base[base[:, 0] != base[:, 1]], mode=oracle.SUPERIOR)
    x = rng.integers(0, n, (k, 2)).astype(np.int32)
    x[: k // 4, 0] = 5                                   # a vertex that many edges meet at
    x[k // 2: k // 2 + k // 8] = x[: k // 8, ::-1]       # repeats, reversed
    for r in range(7):
        assert g.insert_edges(x) == ref.insert_edges(x)
        assert g.insert_edges(x) == 0
        assert g.stats()["applied"] == 0
        assert g.delete_edges(x[k // 3:]) == ref.delete_edges(x[k // 3:])
        if r == 3:
            _same(g, ref)
    _same(g, ref)
    g.close()


@pytest.mark.parametrize("k", [1, 40, 1024, 1500])
def test_invalid_ids_change_nothing(cm, k):
    rng = np.random.default_rng(k)
    n = 300
    base = rng.integers(0, n, (900, 2)).astype(np.int32)
    g = cm.CoreGraph(n, base)
    g.delete_vertices([7])
    ref = oracle.OracleGraph(n, g.edges(), mode=oracle.SUPERIOR)
    good = rng.integers(8, n, (k, 2)).astype(np.int32)
    for bad in (n, -1, 7):
        x = good.copy()
        x[k // 2, 1] = bad
        for f in (g.insert_edges, g.delete_edges):
            with pytest.raises(cm.CoreMaintError) as e:
                f(x)
            assert e.value.code == cm.CM_ERR_INVALID and f"edge {k // 2} " in str(e.value)
    assert g.insert_edges(good) == ref.insert_edges(good)
    c = ref.cores()
    c[7] = -1
    assert (g.cores() == c).all()
    g.close()


def test_lists_compact_in_place(cm):
    """Edges that come and go at full lists need no new list space: the pool
    stays as it is over many rounds."""
    rng = np.random.default_rng(3)
    n = 400
    i, j = np.triu_indices(n, 1)
    pick = rng.permutation(len(i))[:8000]
    e = np.stack([i[pick], j[pick]], 1).astype(np.int32)
    asked = []

    class Counting(cm._TorchAllocator):
        def __init__(self):
            super().__init__()
            inner = self.alloc
            self.alloc = cm._ALLOC_FN(lambda size, stream, ctx: asked.append(size) or inner(size, stream, ctx))

    g = cm.CoreGraph(n, e[:6000], allocator=Counting())
    ref = oracle.bz(n, e[:6000])
    for k in (500, 2000):
        for r in range(60):
            assert g.insert_edges(e[6000: 6000 + k]) == k
            if r == 8:
                seen = len(asked)
            assert g.delete_edges(e[6000: 6000 + k]) == k
        assert len(asked) == seen
    assert (g.cores() == ref).all()
    g.close()
