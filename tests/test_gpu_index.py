"""The edge index under edges that come and go: inserted keys take the buckets
that deleted ones left, lookups still find every edge and no other, and the
host's count of dead buckets stays within what the table holds (a batch larger
than the free buckets still triggers the rebuild)."""
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


@pytest.mark.parametrize("step", [False, True])
@pytest.mark.parametrize("k", [1, 37, 700])
def test_same_edges_come_and_go(cm, k, step):
    import torch
    rng = np.random.default_rng(k)
    n = 500
    i, j = np.triu_indices(n, 1)
    pick = rng.permutation(len(i))
    base = np.stack([i, j], 1)[pick[:2000]].astype(np.int32)
    flux = np.stack([i, j], 1)[pick[2000: 2000 + 3 * k]].astype(np.int32)
    g = cm.CoreGraph(n, base, stream=torch.cuda.Stream())
    ref0 = oracle.bz(n, base)
    st = g.step(k, k) if step else None
    if st:
        st.run([k], flux[:k], [0], flux[:0])
    else:
        assert g.insert_edges(flux[:k]) == k
    for r in range(120):
        new, old = flux[k * ((r + 1) % 3): k * ((r + 1) % 3) + k], flux[k * (r % 3): k * (r % 3) + k]
        if st:
            a, b = st.run([k], new, [k], old)
            assert (int(a[0]), int(b[0])) == (k, k)
        else:
            assert g.insert_edges(new) == k
            assert g.insert_edges(new) == 0        # found again, whatever bucket it took
            assert g.delete_edges(old) == k
            assert g.delete_edges(old) == 0
    cur = np.concatenate([base, flux[k * (120 % 3): k * (120 % 3) + k]])
    assert (g.cores() == oracle.bz(n, cur)).all()
    got = np.sort(g.edges(), 1)
    assert set(map(tuple, got.tolist())) == set(map(tuple, np.sort(cur, 1).tolist()))
    # a large batch after all that: room is made where it is needed
    rest = np.stack([i, j], 1)[pick[2000 + 3 * k: 2000 + 3 * k + 30000]].astype(np.int32)
    assert g.insert_edges(rest) == 30000
    assert g.delete_edges(rest) == 30000
    assert g.delete_edges(cur[len(base):]) == k
    assert (g.cores() == ref0).all()
    r = g.check()
    assert r["sd_mismatches"] == r["degree_mismatches"] == r["bad_neighbour_ids"] == r["kcore_violations"] == 0
    g.close()
