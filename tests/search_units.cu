// Drives parts of the grid-mode search on prepared states (built and called by
// test_gpu_search_units.py).  One block, bounded waits.
#include "../paper_1612_09368_gb300/csrc/cm_search.cuh"

using namespace cm;

// An insertion search whose queue holds one task, the eviction of vertex v.
__global__ void __launch_bounds__(32 * kGridWarps) evict_kernel(DevGraph g, Ctl* C, MaintainParams P, int v, uint32_t e,
                                                                uint32_t e0) {
    WarpBuf& B = reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5];
    if (lane_id() == 0) B.slab = B.slab_end = 0;
    if (lane_id() < 7) B.st[lane_id()] = 0;
    if (threadIdx.x == 0) {
        s_quiet = ~0u;
        s_search_t0 = gtimer();
        P.TQ[0] = mk_task(T_EVICT, (unsigned long long)(uint32_t)v);
        C->task_tail = 1;
        __threadfence();
    }
    __syncthreads();
    async_search<false>(g, C, P, e, e0, true);
}

// All arrays are device memory.  n vertices, vertex 0 with the list
// adj[0, len), the others without one.  rq: the first arena quad of vertex 0's
// record, made in iteration e - 1.  counters: frontier, queue and eviction
// totals, and the error word.
extern "C" int unit_evict(int n, int len, int2* hc, unsigned long long* hw, uint32_t* kc, int64_t* off, int32_t* end,
                          int32_t* adj, unsigned long long* rec, int32_t* arena, unsigned long long quads,
                          unsigned long long* tq, int tq_size, int32_t* vq, int32_t* eq, int ring, HubItem* hq, Ctl* ctl,
                          int expand_early, int hub_len, unsigned e, unsigned e0, unsigned long long* counters) {
    DevGraph g{};
    g.n = n;
    g.hc = hc;
    g.hw = hw;
    g.kc = kc;
    g.off = off;
    g.end = end;
    g.adj = adj;
    g.adj_cap = (len + 3) & ~3;
    MaintainParams P{};
    P.g = g;
    P.ctl = ctl;
    P.VQ = vq;
    P.EQ = eq;
    P.qmask = (unsigned long long)ring - 1;
    P.HQ = hq;
    P.TQ = tq;
    P.tqmask = (unsigned long long)tq_size - 1;
    P.rec = rec;
    P.rec_mask = -1;
    P.arena = arena;
    P.arena_quads = quads;
    P.slab_quads = 32;
    P.hub_len = hub_len;
    P.claim_max = 1;
    P.expand_early = expand_early;
    P.limit_ns = 1000000000ull;
    if (cudaMemset(ctl, 0, sizeof(Ctl)) != cudaSuccess || cudaMemset(tq, 0xFF, 8ull * tq_size) != cudaSuccess) return 1;
    evict_kernel<<<1, 32 * kGridWarps, kSearchSmem>>>(g, ctl, P, 0, e, e0);
    Ctl h;
    if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(&h, ctl, sizeof(Ctl), cudaMemcpyDeviceToHost) != cudaSuccess)
        return 2;
    counters[0] = h.tail[0];
    counters[1] = h.task_tail;
    counters[2] = h.hub_created;
    counters[3] = (unsigned long long)h.error;
    return 0;
}

// Lane l handles entries l, l + 32, ... of a deletion's core-k neighbours.
template <int J>
__global__ void delete_kernel(DevGraph g, Ctl* C, MaintainParams P, const int32_t* id, const int32_t* thr,
                              const unsigned long long* s, const uint32_t* ch, uint32_t e, int k) {
    WarpBuf& B = *reinterpret_cast<WarpBuf*>(s_search);
    Walker W{0, 1, false, 0};
    int i[J], t[J];
    unsigned long long w[J];
    uint32_t c[J], low[J];
#pragma unroll
    for (int j = 0; j < J; j++) {
        const int a = j * 32 + lane_id();
        i[j] = id[a];
        t[j] = thr[a];
        w[j] = s[a];
        c[j] = ch[a];
        low[j] = e << 2 | level_bits(k);
    }
    delete_words<J>(g, C, P, B, W, i, t, low, w, c, e);
}

// 32 entries (wide: 128) at level k.  evicted: those logged.
extern "C" int unit_delete(int wide, int n, unsigned long long* hw, uint32_t* chg, unsigned long long* tq, int tq_size,
                           int32_t* eq, int ring, Ctl* ctl, const int32_t* id, const int32_t* thr,
                           const unsigned long long* s, const uint32_t* ch, unsigned e, int k,
                           unsigned long long* evicted) {
    DevGraph g{};
    g.n = n;
    g.hw = hw;
    g.chg = chg;
    MaintainParams P{};
    P.g = g;
    P.ctl = ctl;
    P.EQ = eq;
    P.qmask = (unsigned long long)ring - 1;
    P.TQ = tq;
    P.tqmask = (unsigned long long)tq_size - 1;
    if (cudaMemset(ctl, 0, sizeof(Ctl)) != cudaSuccess) return 1;
    if (wide) delete_kernel<4><<<1, 32, kSearchSmem>>>(g, ctl, P, id, thr, s, ch, e, k);
    else delete_kernel<1><<<1, 32, kSearchSmem>>>(g, ctl, P, id, thr, s, ch, e, k);
    Ctl h;
    if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(&h, ctl, sizeof(Ctl), cudaMemcpyDeviceToHost) != cudaSuccess)
        return 2;
    *evicted = h.tail[1];
    return h.error ? 3 : 0;
}

extern "C" int unit_ctl_bytes() { return (int)sizeof(Ctl); }
extern "C" int unit_hub_ring() { return (int)kHubRing; }
