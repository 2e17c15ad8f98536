"""The full decomposition, and the superior degrees computed after it, where their paths meet: cascades longer than a block
follows alone (paths, grids), more departures at once than a block's queue
holds (forests, stars), lists long enough to be shared in chunks, empty
levels, and lists that start anywhere in a caller's CSR.  Exact comparison
with the oracle's Batagelj-Zaversnik peeling."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cm():
    import torch
    from paper_1612_09368_gb300 import build
    build.build()
    import paper_1612_09368_gb300 as cm
    torch.cuda.set_device(0)
    return cm


def _pairs(a, b):
    return np.stack([np.asarray(a), np.asarray(b)], 1).astype(np.int32)


def _clique(lo, k):
    i, j = np.triu_indices(k, 1)
    return _pairs(lo + i, lo + j)


def _graph(kind):
    rng = np.random.default_rng(7)
    if kind == "path":            # one cascade of 25,000 steps from each end
        return 50000, _pairs(np.arange(49999), np.arange(1, 50000))
    if kind == "cycle-with-tail":
        return 40000, np.concatenate([_pairs(np.arange(20000), (np.arange(20000) + 1) % 20000),
                                      _pairs(np.arange(19999, 39999), np.arange(20000, 40000))])
    if kind == "stars":           # 40,000 leaves; hubs of 16,383 to 16,385 and a few slots
        sizes = [16383, 16384, 16385] + [3] * 2000
        hub = np.repeat(np.arange(len(sizes)), sizes)
        n = len(sizes) + len(hub)
        return n, np.concatenate([_pairs(hub, len(sizes) + np.arange(len(hub))), _clique(0, 40)])
    if kind == "tree":            # a random recursive tree: every departure at level 1
        v = np.arange(1, 60000)
        return 60000, _pairs((rng.random(len(v)) * v).astype(np.int64), v)
    if kind == "cliques":         # levels 3, 40 and 299 with nothing between
        return 500, np.concatenate([_clique(0, 4), _clique(10, 41), _clique(100, 300)])
    if kind == "bipartite":
        i, j = np.meshgrid(np.arange(70), np.arange(70, 40070), indexing="ij")
        return 40070, _pairs(i.ravel(), j.ravel())
    if kind == "grid":
        return 200 * 200, synth.grid(200, 300, synth.stream(7, 1))
    if kind == "rmat":
        return 1 << 14, synth.rmat(14, 24, synth.stream(7, 2))
    if kind == "31-vertices":
        return 31, _clique(3, 9)
    return 1, np.zeros((0, 2), np.int32)


def _sd(n, e, cores):
    """Neighbours with a core of at least the vertex's own; -1 for a dead vertex."""
    cu, cv = cores[e[:, 0]], cores[e[:, 1]]
    sd = np.bincount(e[:, 0][cv >= cu], minlength=n) + np.bincount(e[:, 1][cu >= cv], minlength=n)
    return np.where(cores < 0, -1, sd)


KINDS = ["path", "cycle-with-tail", "stars", "tree", "cliques", "bipartite", "grid", "rmat", "31-vertices", "single"]


@pytest.mark.parametrize("kind", KINDS)
def test_store(cm, kind):
    import torch
    n, e = _graph(kind)
    ref = oracle.bz(n, e)
    g = cm.CoreGraph(n, torch.from_numpy(e).cuda() if len(e) else e)
    assert (g.cores() == ref).all()
    assert (g.superior_degrees() == _sd(n, e, ref)).all()
    g.recompute_cores()
    assert (g.cores() == ref).all()
    assert (g.superior_degrees() == _sd(n, e, ref)).all()
    if n > 100:   # holes in the lists, dead vertices
        dead = np.arange(0, n, 97, dtype=np.int32)
        g.delete_vertices(dead)
        live = ~np.isin(e, dead).any(1)
        want = oracle.bz(n, e[live])
        want[dead] = -1
        g.apply_edges(cm.CM_OP_DELETE, e[live][:50])
        g.apply_edges(cm.CM_OP_INSERT, e[live][:50])
        g.recompute_cores()
        assert (g.cores() == want).all()
        assert (g.superior_degrees() == _sd(n, e[live], want)).all()
    g.close()


@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("kind", KINDS)
def test_csr(cm, kind, shift):
    import torch
    n, e = _graph(kind)
    src = np.concatenate([e[:, 0], e[:, 1]]).astype(np.int64)
    dst = np.concatenate([e[:, 1], e[:, 0]])
    order = np.argsort(src, kind="stable")
    row = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    # the ids start `shift` entries into a buffer, with out-of-range ids around them
    buf = np.full(len(dst) + shift + 4, n, np.int32)
    buf[shift: shift + len(dst)] = dst[order]
    f = cm.lib().cm_core_numbers_noalloc
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int32] + [ctypes.c_void_p] * 4
    d_row, d_buf = torch.from_numpy(row).cuda(), torch.from_numpy(buf).cuda()
    out = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    rc = f(n, d_row.data_ptr(), d_buf.data_ptr() + 4 * shift, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    assert (out.cpu().numpy() == oracle.bz(n, e)).all()
