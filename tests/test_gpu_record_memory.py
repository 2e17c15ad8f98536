"""The memory of the search records is optional: an allocator that refuses it
(all of it, or only large blocks) leaves every call working, deletions never
ask for it, and a handle that has been refused asks again once its graph has
grown.  Small graphs and graphs whose words alone exceed the block that every
handle has.  Iterations, cores and superior degrees against the oracle."""
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


class Limited:
    """Torch's caching allocator; requests above `limit` bytes get NULL, but for
    powers of two (the task queue and the hash sets, which a call needs)."""

    def __init__(self, cm):
        inner = cm._TorchAllocator()
        self.limit, self.asked = None, []

        def alloc(size, stream, ctx):
            self.asked.append(size)
            refuse = self.limit is not None and size > self.limit and size & (size - 1)
            return None if refuse else inner.alloc(size, stream, ctx)

        self.inner, self.free, self.alloc = inner, inner.free, cm._ALLOC_FN(alloc)


def _same(g, ref):
    cores = ref.cores()
    assert (g.cores() == cores).all()
    e = np.asarray(ref.edges())
    cu, cv = cores[e[:, 0]], cores[e[:, 1]]
    sd = np.bincount(e[:, 0][cv >= cu], minlength=len(cores)) + np.bincount(e[:, 1][cu >= cv], minlength=len(cores))
    assert (g.superior_degrees() == sd).all()


@pytest.mark.parametrize("limit", [100_000, 6 << 20, None], ids=["nothing", "6-MiB", "all"])
@pytest.mark.parametrize("n", [3000, 300_000])
def test_refused_records(cm, n, limit):
    import torch
    rng = np.random.default_rng(n)
    d = 3000
    p = np.repeat([0.8, 0.6, 0.35, 0.2], d // 4)          # a dense part: long lists, many iterations
    i, j = np.triu_indices(d, 1)
    keep = rng.random(len(i)) < p[i] * p[j]
    e = np.stack([i[keep], j[keep]], 1)
    if n > d:
        e = np.concatenate([e, np.stack([np.arange(d, n), rng.integers(0, np.arange(d, n))], 1)])
    e = rng.permutation(e).astype(np.int32)
    alloc = Limited(cm)
    g = cm.CoreGraph(n, torch.from_numpy(e).cuda(), allocator=alloc, block_mode_edges=-1, stream=torch.cuda.Stream())
    ref = oracle.OracleGraph(n, e, mode=oracle.SUPERIOR)
    alloc.limit = limit
    records = 8 * n + len(e)                                      # less than the records of the pool take
    before = len(alloc.asked)
    step = g.step(0, 1000)
    assert g.delete_edges(e[:900]) == ref.delete_edges(e[:900])
    step.run([0], e[:0], [900], e[900:1800])
    assert ref.delete_edges(e[900:1800]) == 900
    _same(g, ref)
    assert all(s <= records or s & (s - 1) == 0 for s in alloc.asked[before:])   # deletions ask for no records
    before = len(alloc.asked)
    hot = rng.choice(d, 30, replace=False)
    for b in range(3):
        x = np.stack([rng.choice(hot, 800), rng.integers(0, d, 800)], 1).astype(np.int32)
        x = x[x[:, 0] != x[:, 1]]
        for f, r in ((g.insert_edges, ref.insert_edges), (g.delete_edges, ref.delete_edges)):
            assert f(x) == r(x)
            assert g.stats()["iterations"] == ref.last_iterations()
            _same(g, ref)
    asked = alloc.asked[before:]
    assert asked and max(asked) > records and len(asked) <= 4     # once, not on every call
    # a captured step with both phases, and a graph that grows with memory at hand again
    both = g.step(1000, 1000)
    a, b = both.run([900], e[:900], [900], e[5000:5900])
    assert (int(a[0]), int(b[0])) == (ref.insert_edges(e[:900]), ref.delete_edges(e[5000:5900]))
    _same(g, ref)
    alloc.limit = None
    more = rng.integers(0, n, (len(e) // 2, 2)).astype(np.int32)
    more = more[more[:, 0] != more[:, 1]]
    m = g.m
    assert g.insert_edges(more) == g.m - m > len(more) // 4
    cur = g.edges()
    assert len(np.unique(np.sort(cur, 1), axis=0)) == g.m
    assert (g.cores() == oracle.bz(n, cur)).all()
    r = g.check()
    assert [r[k] for k in ("sd_mismatches", "key_mismatches", "degree_mismatches", "kcore_violations")] == [0] * 4
    both.close()
    step.close()
    g.close()
