"""Performance cases: the work that users have this library do, through its
public Python API, over the range of sizes that it is used at.

Kinds of a case:

  update   one handle; a batch of new edges goes in and a batch of existing
           edges goes out, the cores are read, then both batches are undone
           (so each pass does insertions and deletions and can be repeated);
  step     many independent graphs in one handle, each with its own insert
           and delete batch, applied as one captured update step and undone
           by the step of the opposite batches;
  serve    the request loop: two resident graphs, a burst of mixed requests
           from host memory, the cores of both graphs read, then the burst of
           the opposite requests;
  repeel   the full decomposition of a resident graph after its structure
           changed (apply_edges, recompute_cores, cores and superior
           degrees), then the change undone and the graph re-peeled;
  load     a graph built from an edge list (index, adjacency, decomposition),
           new vertices inserted, old ones deleted, cores read, handle closed;
  csr      the allocation-free decomposition of a caller's CSR graph.

Graph families (those of the paper's synthetic experiments and of this
repository's workloads): R-MAT (.57, .19, .19, .05) with permuted ids,
Erdos-Renyi, preferential attachment (Batagelj and Brandes' method) and a
square 4-neighbour grid with 1% random shortcuts.  New edges join uniform
vertices, or vertices in proportion to their degree (law "degree"); deleted
edges are uniform edges of the graph.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1612_09368_gb300 as cm

# ------------------------------------------------------------------ the cases


def listed():
    return [
        # A single friendship or citation arriving at a small graph: latency of
        # one call with host ids, launches and read-backs and no other work.
        dict(name="er10k-1", kind="update", family="er", n=10_000, degree=5, ins=1, dele=1, law="uniform", host=True),
        # The library's smallest configuration: G(10^4, 5*10^4), batches of 1,000
        # from host memory, as an interactive analysis applies them.
        dict(name="er10k-1000", kind="update", family="er", n=10_000, degree=5, ins=1000, dele=1000, law="uniform",
             host=True),
        # The rounds configuration: a social-network-like graph of 2^20 vertices
        # under a steady stream of 10^4 new and 10^4 retired edges per round.
        dict(name="rmat20-1e4", kind="update", family="rmat", n=1 << 20, degree=16, ins=10_000, dele=10_000,
             law="uniform", host=False),
        # A graph of one core level (all of a large Erdos-Renyi graph is one
        # shell or two): each batch searches a whole shell.
        dict(name="er2m-1e4", kind="update", family="er", n=2_000_003, degree=4, ins=10_007, dele=10_007,
             law="uniform", host=False),
        # The batch sweep on the largest graph: new edges between its dense,
        # busy vertices, few at a time ...
        dict(name="rmat24-deg-1e3", kind="update", family="rmat", n=1 << 24, degree=16, ins=1_000, dele=1_000,
             law="degree", host=False),
        # ... 10^5 uniform ones ...
        dict(name="rmat24-uni-1e5", kind="update", family="rmat", n=1 << 24, degree=16, ins=100_000, dele=100_000,
             law="uniform", host=False),
        # ... and the largest batch of the sweep, 10^6, in proportion to degree.
        dict(name="rmat24-deg-1e6", kind="update", family="rmat", n=1 << 24, degree=16, ins=1_000_000,
             dele=1_000_000, law="degree", host=False),
        # Many tenants: 64 preferential-attachment graphs of 10^3 to 10^6 vertices
        # with batches of 10 to 10^4 edges, 70% inserts, as one captured step.
        dict(name="ba64-step", kind="step", graphs=64, nmin=1_000, nmax=1_000_000, bmin=10, bmax=10_000),
        # Serving: the two resident graphs of the serving workload, a burst of 64
        # requests of log-normal size (median 200, 10 to 10^5), 70% inserts.
        dict(name="serve-rmat22-grid", kind="serve", n=1 << 22, degree=16, side=2048, requests=64, median=200),
        # Re-peeling the largest graph from scratch after 10^5 edges changed.
        dict(name="rmat24-repeel", kind="repeel", family="rmat", n=1 << 24, degree=16, ins=100_000),
        # Loading a graph, then growing and shrinking it by whole vertices.
        dict(name="rmat20-load", kind="load", family="rmat", n=1 << 20, degree=16, vins=100, vdeg=8, vdel=100),
        # A framework that owns the device memory asks for the cores of its CSR.
        dict(name="rmat20-csr", kind="csr", family="rmat", n=1 << 20, degree=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update"] * 6 + ["step", "serve", "repeel", "load", "csr"])
    if kind == "step":
        return dict(kind=kind, graphs=rng.randint(2, 64), nmin=1_000, nmax=_log(rng, 10_000, 1_000_000), bmin=10,
                    bmax=_log(rng, 30, 10_000))
    if kind == "serve":
        return dict(kind=kind, n=_log(rng, 10_000, 1 << 22), degree=rng.choice([8, 16]),
                    side=_log(rng, 60, 2048), requests=rng.randint(4, 64), median=_log(rng, 20, 400))
    family = rng.choice(["rmat", "rmat", "rmat", "er", "ba", "grid"])
    top = {"update": 1 << 24, "repeel": 1 << 24, "load": 1 << 21, "csr": 1 << 20}[kind]
    n = _log(rng, 10_000, top if family == "rmat" else min(top, 2_100_000))
    if family == "grid":
        n = math.isqrt(n) ** 2
    degree = {"rmat": rng.choice([8, 16]), "er": rng.choice([4, 5, 8]), "ba": rng.randint(4, 16), "grid": 2}[family]
    case = dict(kind=kind, family=family, n=n, degree=degree)
    if kind == "update":
        k = _log(rng, 1, n // 16)
        case.update(ins=k, dele=_log(rng, 1, n // 16) if rng.random() < 0.5 else k,
                    law=rng.choice(["uniform", "degree"]), host=rng.random() < 0.3)
    elif kind == "repeel":
        case.update(ins=_log(rng, 1, n // 16))
    elif kind == "load":
        case.update(vins=_log(rng, 1, 1000), vdeg=rng.randint(1, 16), vdel=_log(rng, 1, 1000))
    return case


# ------------------------------------------------------------------ graphs and batches


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rand(g, k, hi):
    return torch.randint(hi, (k,), generator=g, device="cuda")


def _rmat(g, n, samples):
    """Endpoints of R-MAT samples over 2^ceil(log2 n) vertices, ids permuted;
    samples that name a vertex >= n are dropped."""
    scale = max(1, (n - 1).bit_length())
    u = torch.zeros(samples, dtype=torch.int32, device="cuda")
    v = torch.zeros(samples, dtype=torch.int32, device="cuda")
    for _ in range(scale):
        r = torch.rand(samples, generator=g, device="cuda")
        bu = r >= 0.57 + 0.19
        u.mul_(2).add_(bu)
        v.mul_(2).add_(((r >= 0.57) & ~bu) | (r >= 0.57 + 0.19 + 0.19))
    del r, bu
    perm = torch.randperm(1 << scale, generator=g, device="cuda").int()
    u, v = perm[u], perm[v]
    if n < 1 << scale:
        keep = (u < n) & (v < n)
        u, v = u[keep], v[keep]
    return u, v


def _attach(g, n, degree):
    """Preferential attachment: every vertex brings `degree` edges, the other
    end of each a copy of a uniformly chosen earlier edge end."""
    m = n * degree
    ends = torch.arange(2 * m, device="cuda")
    r = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * (ends[1::2])).long()
    ends[1::2] = torch.minimum(r, ends[1::2] - 1)
    while bool((ends & 1).any()):
        ends = ends[ends]
    ends = ends // (2 * degree)
    return ends[0::2], ends[1::2]


def _graph(g, family, n, degree):
    """The graph's edges as sorted keys lo * n + hi, each edge once."""
    if family == "rmat":
        u, v = _rmat(g, n, n * degree)
    elif family == "er":
        u, v = _rand(g, n * degree, n), _rand(g, n * degree, n)
    elif family == "ba":
        u, v = _attach(g, n, degree)
    else:
        side = math.isqrt(n)
        at = torch.arange(n, device="cuda")
        right, down = at[at % side < side - 1], at[: n - side]
        k = max(1, (right.numel() + down.numel()) // 100)
        u = torch.cat([right, down, _rand(g, k, n)])
        v = torch.cat([right + 1, down + side, _rand(g, k, n)])
    return _keys(u, v, n)


def _keys(u, v, n):
    keep = u != v
    u, v = u[keep], v[keep]
    return torch.unique(torch.minimum(u, v).long() * n + torch.maximum(u, v))


def _pairs(keys, n):
    return torch.stack([keys // n, keys % n], 1).int()


def _new_edges(g, keys, n, k, law):
    """k distinct pairs that are no edges of the graph, in random order."""
    got = keys[:0]
    for _ in range(32):
        if got.numel() >= k:
            break
        t = 2 * k + 64
        if law == "degree":
            a, b = keys[_rand(g, t, keys.numel())], keys[_rand(g, t, keys.numel())]
            u = torch.where(_rand(g, t, 2) == 0, a // n, a % n)
            v = torch.where(_rand(g, t, 2) == 0, b // n, b % n)
        else:
            u, v = _rand(g, t, n), _rand(g, t, n)
        x = _keys(u, v, n)
        at = torch.searchsorted(keys, x).clamp_(max=keys.numel() - 1)
        got = torch.unique(torch.cat([got, x[keys[at] != x]]))
    return got[torch.randperm(got.numel(), generator=g, device="cuda")[:k]]


def _old_edges(g, keys, k):
    """k distinct uniform edges of the graph, in random order."""
    k = min(k, keys.numel())
    at = torch.unique(_rand(g, 2 * k + 64, keys.numel()))
    while at.numel() < k:
        at = torch.unique(torch.cat([at, _rand(g, 2 * k + 64, keys.numel())]))
    return keys[at[torch.randperm(at.numel(), generator=g, device="cuda")[:k]]]


def _tenants(case, seed):
    """Graphs of a step case.  The sizes follow from the case alone: n spread
    evenly over its logarithm, 4 to 16 edges per vertex, the batch size (70%
    of it new edges) spread likewise but in another order."""
    g = _gen(seed)
    c = case["graphs"]
    out = []
    for i in range(c):
        n = int(case["nmin"] * (case["nmax"] / case["nmin"]) ** ((i + 0.5) / c))
        b = int(case["bmin"] * (case["bmax"] / case["bmin"]) ** ((i * 0.618034) % 1.0))
        keys = _graph(g, "ba", n, 4 + 7 * i % 13)
        ki = round(0.7 * b)
        out.append((n, keys, _new_edges(g, keys, n, ki, "uniform"), _old_edges(g, keys, b - ki)))
    return out


def _requests(case, seed):
    """Two graphs and a burst of requests (graph, op, key range): new edges or
    existing edges, none shared between requests."""
    rng = np.random.default_rng(seed)
    g = _gen(seed)
    graphs = [(case["n"], _graph(g, "rmat", case["n"], case["degree"])),
              (case["side"] ** 2, _graph(g, "grid", case["side"] ** 2, 2))]
    size = np.clip(np.exp(rng.normal(math.log(case["median"]), 1.5, case["requests"])), 10, 100_000)
    reqs = []
    for i in range(case["requests"]):
        gi, op = int(rng.integers(2)), int(rng.random() >= 0.7)
        reqs.append((gi, op, max(1, int(min(size[i], graphs[gi][0] // 64)))))
    pools = {}
    for gi, (n, keys) in enumerate(graphs):
        for op in (0, 1):
            k = max(1, sum(r[2] for r in reqs if r[:2] == (gi, op)))
            pools[gi, op] = _new_edges(g, keys, n, k, "uniform") if op == 0 else _old_edges(g, keys, k)
    at = dict.fromkeys(pools, 0)
    burst = []
    for gi, op, k in reqs:
        a = at[gi, op]
        at[gi, op] = a + k
        if pools[gi, op][a:a + k].numel():
            burst.append((gi, op, pools[gi, op][a:a + k]))
    return graphs, burst


def _one(case, seed):
    """Graph and batches of the single-graph kinds."""
    g = _gen(seed)
    n = case["n"]
    keys = _graph(g, case["family"], n, case["degree"])
    ins = _new_edges(g, keys, n, case["ins"], case.get("law", "uniform")) if "ins" in case else keys[:0]
    dele = _old_edges(g, keys, case["dele"]) if "dele" in case else keys[:0]
    return n, keys, ins, dele


def _vertices(case, seed):
    """Neighbour lists of new vertices, and the old vertices to delete."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    lists = [rng.choice(n, case["vdeg"], replace=False).astype(np.int32) for _ in range(case["vins"])]
    return lists, rng.choice(n, case["vdel"], replace=False).astype(np.int32)


def _csr(n, keys):
    u, v = keys // n, keys % n
    both = torch.sort(torch.cat([u * n + v, v * n + u]))[0]
    row = torch.searchsorted(both, torch.arange(n + 1, device="cuda") * n)
    return row, (both % n).int()


# ------------------------------------------------------------------ prepare and run


def prepare(case, seed):
    s = {"kind": case["kind"]}
    if case["kind"] in ("update", "repeel"):
        n, keys, ins, dele = _one(case, seed)
        s["graph"] = cm.CoreGraph(n, _pairs(keys, n))
        batches = [_pairs(ins, n), _pairs(dele, n)]
        s["ins"], s["dele"] = [b.cpu().numpy() for b in batches] if case.get("host") else batches
        s["out"] = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)]
    elif case["kind"] == "step":
        ts = _tenants(case, seed)
        stream = torch.cuda.Stream()
        edges, ins, dele = (torch.cat([_pairs(t[i], t[0]) for t in ts]) for i in (1, 2, 3))
        torch.cuda.synchronize()
        s["graph"] = cm.CoreGraph(None, edges, multi=([t[0] for t in ts], [t[1].numel() for t in ts]), stream=stream)
        s["ins"], s["dele"] = ins, dele
        s["kins"], s["kdel"] = (np.array([t[i].numel() for t in ts], np.int64) for i in (2, 3))
        s["step"] = s["graph"].step(max(1, len(ins)), max(1, len(dele)))
        s["undo"] = s["graph"].step(max(1, len(dele)), max(1, len(ins)))
        s["out"] = [torch.empty(s["graph"].n, dtype=torch.int32, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
    elif case["kind"] == "serve":
        graphs, burst = _requests(case, seed)
        edges = [_pairs(keys, n) for n, keys in graphs]
        torch.cuda.synchronize()
        half = torch.cuda.get_device_properties(0).multi_processor_count // 2
        s["burst"] = [(gi, op, _pairs(k, graphs[gi][0]).cpu().numpy()) for gi, op, k in burst]
        s["graphs"] = [cm.CoreGraph(n, e, stream=torch.cuda.Stream(), max_sms=half)
                       for (n, _), e in zip(graphs, edges)]
        s["server"] = cm.Server(s["graphs"], 1 << 26)
    elif case["kind"] == "load":
        n, keys, _, _ = _one(case, seed)
        s["n"], s["edges"] = n, _pairs(keys, n)
        s["lists"], s["ids"] = _vertices(case, seed)
        s["out"] = [torch.empty(n + case["vins"], dtype=torch.int32, device="cuda") for _ in range(2)]
    else:
        n, keys, _, _ = _one(case, seed)
        s["n"], (s["row"], s["adj"]) = n, _csr(n, keys)
        s["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
        f = cm.lib().cm_core_numbers_noalloc
        f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int32] + [ctypes.c_void_p] * 4
        s["f"] = f
    return s


def run(s):
    if s["kind"] == "update":
        g = s["graph"]
        applied = [g.insert_edges(s["ins"]), g.delete_edges(s["dele"])]
        g.cores(s["out"][0])
        applied += [g.insert_edges(s["dele"]), g.delete_edges(s["ins"])]
        g.cores(s["out"][1])
        return {"applied": applied, "cores": s["out"][0], "undone": s["out"][1]}
    if s["kind"] == "step":
        a = s["step"].run(s["kins"], s["ins"], s["kdel"], s["dele"])
        s["graph"].cores(s["out"][0])
        b = s["undo"].run(s["kdel"], s["dele"], s["kins"], s["ins"])
        s["graph"].cores(s["out"][1])
        return {"applied": [*a, *b], "cores": s["out"][0], "undone": s["out"][1]}
    if s["kind"] == "serve":
        srv = s["server"]
        for gi, op, e in s["burst"]:
            srv.submit(gi, op, e)
        status = [srv.drain()]
        cores = [srv.cores(0), srv.cores(1)]
        for gi, op, e in s["burst"]:
            srv.submit(gi, 1 - op, e)
        status.append(srv.drain())
        return {"status": status, "cores": cores}
    if s["kind"] == "repeel":
        g = s["graph"]
        applied = [g.apply_edges(cm.CM_OP_INSERT, s["ins"])]
        g.recompute_cores()
        g.cores(s["out"][0])
        g.superior_degrees(s["out"][1])
        applied.append(g.apply_edges(cm.CM_OP_DELETE, s["ins"]))
        g.recompute_cores()
        return {"applied": applied, "cores": s["out"][0], "sd": s["out"][1]}
    if s["kind"] == "load":
        with cm.CoreGraph(s["n"], s["edges"]) as g:
            first, added = g.insert_vertices(s["lists"])
            gone = g.delete_vertices(s["ids"])
            g.cores(s["out"][0])
            g.superior_degrees(s["out"][1])
        return {"applied": [first, added, gone], "cores": s["out"][0], "sd": s["out"][1]}
    rc = s["f"](s["n"], s["row"].data_ptr(), s["adj"].data_ptr(), s["out"].data_ptr(),
                torch.cuda.current_stream().cuda_stream)
    return {"status": rc, "cores": s["out"]}


# ------------------------------------------------------------------ work and exact results


def work(case):
    """Bytes alone (there is no floating-point work).  A graph is 8 bytes per
    undirected edge in a decomposition (each id once per direction); an update
    reads its batch and, once, the lists of the edges' ends with their
    neighbours' cores, and each read of the cores writes 4 bytes per vertex.
    The search that a batch starts depends on the graph and is left out."""
    if case["kind"] == "step":
        mean = lambda a, b: a if a == b else (b - a) / math.log(b / a)  # noqa: E731  of a log-uniform size
        n, b = case["graphs"] * mean(case["nmin"], case["nmax"]), case["graphs"] * mean(case["bmin"], case["bmax"])
        return {"bytes": 2 * b * (8 + 2 * 20 * 8) + 2 * 4 * n, "flops": 0}
    if case["kind"] == "serve":
        b = case["requests"] * min(3 * case["median"], 100_000)
        return {"bytes": 2 * b * (8 + 2 * case["degree"] * 8) + 4 * (case["n"] + case["side"] ** 2), "flops": 0}
    n, d = case["n"], case["degree"]
    if case["kind"] == "update":
        ends = min(2 * (case["ins"] + case["dele"]), n)
        return {"bytes": 2 * (8 * (case["ins"] + case["dele"]) + ends * 2 * d * 8) + 2 * 4 * n, "flops": 0}
    if case["kind"] == "repeel":
        return {"bytes": 2 * (8 * n * d + 8 * n + 8 * case["ins"]) + 2 * 4 * n, "flops": 0}
    if case["kind"] == "load":
        return {"bytes": 8 * n * d + 8 * n * d + 2 * 4 * n + 8 * case["vins"] * case["vdeg"], "flops": 0}
    return {"bytes": 8 * n * d + 8 * n + 4 * n, "flops": 0}


def _cores(n, keys):
    """Core numbers by peeling, in plain torch: drop the vertices of degree at
    most k until none is left, then raise k."""
    u, v = keys // n, keys % n
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    core = torch.zeros(n, dtype=torch.int64, device="cuda")
    alive = torch.ones(n, dtype=torch.bool, device="cuda")
    k = 0
    while True:
        gone = alive & (deg <= k)
        if not bool(gone.any()):
            if not bool(alive.any()):
                return core
            k = int(deg[alive].min())
            continue
        core[gone] = k
        alive &= ~gone
        keep = alive[u] & alive[v]
        cut = ~keep
        deg -= torch.bincount(torch.cat([u[cut], v[cut]]), minlength=n)
        u, v = u[keep], v[keep]


def _sd(n, keys, core):
    """Superior degrees: neighbours whose core is at least the vertex's own."""
    u, v = keys // n, keys % n
    return torch.bincount(torch.cat([u[core[v] >= core[u]], v[core[u] >= core[v]]]), minlength=n)


def _apply(keys, ins, dele):
    out = torch.unique(torch.cat([keys, ins]))
    return out[~torch.isin(out, dele)]


def exact(case, seed):
    if case["kind"] != "step" and case["n"] * case.get("degree", 1) > 1 << 25:
        return None  # peeling 10^8 edges in plain torch takes too long
    if case["kind"] == "step":
        ts = _tenants(case, seed)
        if sum(t[1].numel() for t in ts) > 1 << 25:
            return None
        kins, kdel = (np.array([t[i].numel() for t in ts], np.int64) for i in (2, 3))
        after = torch.cat([_cores(n, _apply(keys, ins, dele)) for n, keys, ins, dele in ts])
        before = torch.cat([_cores(n, keys) for n, keys, _, _ in ts])
        return {"applied": [kins, kdel, kdel, kins], "cores": after, "undone": before}
    if case["kind"] == "serve":
        graphs, burst = _requests(case, seed)
        cores = []
        for gi, (n, keys) in enumerate(graphs):
            ins, dele = (torch.cat([keys[:0]] + [k for b, o, k in burst if (b, o) == (gi, op)]) for op in (0, 1))
            cores.append(_cores(n, _apply(keys, ins, dele)))
        return {"status": [0, 0], "cores": cores}
    n, keys, ins, dele = _one(case, seed)
    if case["kind"] == "update":
        ki, kd = ins.numel(), dele.numel()
        return {"applied": [ki, kd, kd, ki], "cores": _cores(n, _apply(keys, ins, dele)), "undone": _cores(n, keys)}
    if case["kind"] == "repeel":
        new = _apply(keys, ins, dele)
        core = _cores(n, new)
        return {"applied": [ins.numel(), ins.numel()], "cores": core, "sd": _sd(n, new, core)}
    if case["kind"] == "csr":
        return {"status": 0, "cores": _cores(n, keys)}
    lists, ids = _vertices(case, seed)
    total = n + case["vins"]
    own = torch.repeat_interleave(torch.arange(n, total, device="cuda"), case["vdeg"])
    nbr = torch.from_numpy(np.concatenate(lists)).cuda().long()
    dead = torch.zeros(total, dtype=torch.bool, device="cuda")
    dead[torch.from_numpy(ids).cuda().long()] = True
    u, v = torch.cat([keys // n, nbr]), torch.cat([keys % n, own])
    cut = dead[u] | dead[v]
    new = _keys(u[~cut], v[~cut], total)
    core = _cores(total, new)
    sd = _sd(total, new, core)
    core[dead], sd[dead] = -1, -1
    return {"applied": [n, own.numel(), int(cut.sum())], "cores": core, "sd": sd}
