"""Parts of the grid-mode search on prepared states: moments that a whole call
meets only by chance of timing.  Exact integers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def units(tmp_path_factory):
    import torch
    from paper_1612_09368_gb300 import build
    torch.cuda.set_device(0)
    lib = str(tmp_path_factory.mktemp("units") / "search_units.so")
    r = subprocess.run([build.nvcc(), *build.FLAGS, *build.ARCH, "-shared", os.path.join(HERE, "search_units.cu"),
                        "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("visited", [True, False], ids=["visited", "not-visited-yet"])
@pytest.mark.parametrize("hub_len", [0, 256], ids=["one-warp", "chunks"])
@pytest.mark.parametrize("length", [257, 512, 1300])
def test_eviction_from_an_earlier_iterations_record(units, length, hub_len, visited):
    """A vertex that an earlier iteration recorded is evicted: each candidate of
    the record loses one support in this iteration.  In the paper's order
    (expand_early -1) that can come before the vertex has visited its
    candidates, whose words then still belong to older iterations (a processed
    flag and a count just above the level among them)."""
    import torch
    k, e, e0, n = 5, 9, 3, length + 1
    nb = 1 + np.arange(length)
    words = np.zeros(n, np.uint64)
    old = np.where(nb % 3 == 0, (np.uint64(k + 1) << np.uint64(32)) | np.uint64((e - 2) << 2 | 3),
                   np.where(nb % 3 == 1, np.uint64((e - 5) << 2), np.uint64(0))).astype(np.uint64)
    words[1:] = (np.uint64(40) << np.uint64(32)) | np.uint64(e << 2 | 3) if visited else old
    words[0] = (np.uint64(k) << np.uint64(32)) | np.uint64(e << 2 | 3)
    key = np.full(n, 2 * k + 1, np.uint32)
    key[1::7] = 2 * k + 2                       # risen above the level since
    key[2::11] = 2 * k                          # its superior degree does not exceed the level
    hc = np.stack([key >> 1, (key >> 1) + (key & 1)], 1).astype(np.int32)
    off, end = np.zeros(n, np.int64), np.zeros(n, np.int32)
    end[0] = length
    rq, room = 4, length + 8
    quads = rq + 1 + (room + 3) // 4
    arena = np.zeros(4 * quads, np.int32)
    arena[4 * rq: 4 * rq + 4] = [length, room, 0, k]
    arena[4 * rq + 4: 4 * rq + 4 + length] = nb | np.where(nb % 2 == 0, -(1 << 31), 0)
    rec = np.zeros(n, np.uint64)
    rec[0] = (rq << 30) | (e - 1)
    ring, tqs = 1 << 11, 1 << 19
    t = [_dev(x.view(np.int64) if x.dtype == np.uint64 else x.view(np.int32) if x.dtype == np.uint32 else x)
         for x in (hc, words, key, off, end, np.append(nb, [-1] * 3).astype(np.int32), rec, arena)]
    tq = torch.empty(tqs, dtype=torch.int64, device="cuda")
    vq, eq = (torch.zeros(ring, dtype=torch.int32, device="cuda") for _ in range(2))
    hq = torch.zeros(units.unit_hub_ring() * 64, dtype=torch.uint8, device="cuda")
    ctl = torch.zeros(units.unit_ctl_bytes(), dtype=torch.uint8, device="cuda")
    counters = (ctypes.c_uint64 * 4)()
    rc = units.unit_evict(n, length, *[_p(x) for x in t], ctypes.c_uint64(quads), _p(tq), tqs, _p(vq), _p(eq), ring,
                          _p(hq), _p(ctl), 0 if visited else -1, hub_len, e, e0, counters)
    assert rc == 0 and counters[3] == 0
    chunks = -(-length // 512) if hub_len else 0
    assert list(counters)[:3] == [0, 1 + chunks, 1 if hub_len else 0]      # nobody else is evicted or visited
    got = t[1].cpu().numpy().view(np.uint64)
    cand = key == 2 * k + 1
    cand[0] = False
    want = words.copy()
    want[cand] = ((np.uint64(39) << np.uint64(32)) | np.uint64(e << 2 | 3)) if visited else \
        np.uint64(0xFFFFFFFF00000000) | np.uint64(e << 2)
    assert (got == want).all()


@pytest.mark.parametrize("wide", [0, 1])
def test_a_vertex_leaves_once_whatever_stamp_was_read(units, wide):
    """A deletion's neighbours as read with an old change stamp: one that has
    left level k + 1 meanwhile (its count is one below the threshold of level k)
    is not evicted again, the others leave when their count reaches it.  A
    word carries the low bits of its level."""
    import torch
    e, k, m = 9, 5, 128 if wide else 32
    i = np.arange(m)
    kind = i % 5            # 0 left meanwhile; 1 leaves now; 2, 4 stay; 3 leaves at the first touch
    sd = k + 2 + i % 7
    count = np.where((kind == 2) | (kind == 4), 0, sd - k)
    sd[kind == 3] = k
    thr = (sd - k + 1).astype(np.int32)
    level = np.where(kind == 0, k + 1, k).astype(np.uint64)
    word = (count.astype(np.uint64) << np.uint64(32)) | np.uint64(e << 2) | (level & np.uint64(3))
    word[(kind == 3) | (kind == 4)] = np.uint64(77) << np.uint64(32) | np.uint64((e - 1) << 2)
    read = np.full(m, e - 2, np.uint32)
    chg = np.where(kind == 0, e, e - 2).astype(np.uint32)
    d_word, d_chg = _dev(word.view(np.int64)), _dev(chg.view(np.int32))
    ring, tqs = 1 << 10, 1 << 19
    tq = torch.full((tqs,), -1, dtype=torch.int64, device="cuda")
    eq = torch.full((ring,), -1, dtype=torch.int32, device="cuda")
    ctl = torch.zeros(units.unit_ctl_bytes(), dtype=torch.uint8, device="cuda")
    args = [_dev(x) for x in (i.astype(np.int32), thr, word.view(np.int64), read.view(np.int32))]
    out = ctypes.c_uint64()
    rc = units.unit_delete(wide, m, _p(d_word), _p(d_chg), _p(tq), tqs, _p(eq), ring, _p(ctl), *[_p(x) for x in args], e,
                           k, ctypes.byref(out))
    assert rc == 0
    leave = np.flatnonzero((kind == 1) | (kind == 3))
    assert out.value == len(leave)
    assert (np.sort(eq.cpu().numpy()[: len(leave)]) == leave).all()
    want = chg.copy()
    want[leave] = e
    assert (d_chg.cpu().numpy().view(np.uint32) == want).all()
    got = d_word.cpu().numpy().view(np.uint64)
    first = np.uint64(1) << np.uint64(32) | np.uint64(e << 2 | k & 3)
    assert (got == np.where((kind == 3) | (kind == 4), first, word + (np.uint64(1) << np.uint64(32)))).all()
