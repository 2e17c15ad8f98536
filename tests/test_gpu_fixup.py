"""The grid-mode fix-up of superior degrees: few moved vertices (a warp each),
more of them than warps (short lists together), lists on both sides of the
short limit (256 slots) and of a chunk's end, deletions with and without a hub
(1024 slots), and more moved vertices than eight per warp.  Hubs with leaves
hang on a ring by one edge each and rise when a batch adds more edges to the
ring.  Core numbers and superior degrees are integers with one right answer:
exact comparison."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

EDGES = [3, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1537, 4095, 4096, 4097, 9000]
CASES = {
    "few": EDGES,
    "many": EDGES + [1 + i % 41 for i in range(5000)],
    "crowd": [300 + i for i in range(100)] + [2 + i % 4 for i in range(40000)],
}


@pytest.fixture(scope="module")
def cm():
    import torch
    from paper_1612_09368_gb300 import build
    build.build()
    import paper_1612_09368_gb300 as cm
    torch.cuda.set_device(0)
    return cm


def _sd(n, e, cores):
    cu, cv = cores[e[:, 0]], cores[e[:, 1]]
    return np.bincount(e[:, 0][cv >= cu], minlength=n) + np.bincount(e[:, 1][cu >= cv], minlength=n)


@pytest.mark.parametrize("opts", [{}, {"block_slots": 512, "block_slots_delete": 4096}], ids=["default", "chunks"])
@pytest.mark.parametrize("extra", [1, 2])
@pytest.mark.parametrize("case", list(CASES))
def test_moved_lists(cm, case, extra, opts):
    import torch
    lens = np.asarray(CASES[case])
    m, ring = len(lens), max(64, len(lens))
    hub = ring + np.arange(m)
    leaf = ring + m + np.arange(lens.sum())
    n = ring + m + len(leaf)
    r = np.arange(ring)
    e = np.concatenate([np.stack([r, (r + 1) % ring], 1), np.stack([np.arange(m), hub], 1),
                        np.stack([np.repeat(hub, lens), leaf], 1)]).astype(np.int32)
    new = np.concatenate([np.stack([(np.arange(m) + 2 + 7 * j) % ring, hub], 1) for j in range(extra)]).astype(np.int32)
    g = cm.CoreGraph(n, torch.from_numpy(e).cuda(), block_mode_edges=-1, **opts)
    both = np.concatenate([e, new])
    for _ in range(2):
        for cur, call in ((both, g.insert_edges), (e, g.delete_edges)):
            assert call(torch.from_numpy(new).cuda()) == len(new)
            ref = oracle.bz(n, cur)
            assert (g.cores() == ref).all()
            assert (g.superior_degrees() == _sd(n, cur, ref)).all()
            s = g.stats()
            assert s["grid_iterations"] == s["iterations"] and s["changed"] >= m
    g.close()
