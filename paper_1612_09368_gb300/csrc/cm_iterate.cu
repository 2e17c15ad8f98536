// cm_iterate.cu -- the superior-edge-set iterations of one update batch.
//
// maintain_kernel<MODE> runs the iterations of SuperiorEdgeInsert
// (Algorithm 1) or SuperiorEdgeDelete (Algorithm 5) on the remaining edges
// of a batch.  MODE 0 is a cooperative launch filling the GPU, with grid-wide
// barriers; MODE 1 is one block of 512 threads with __syncthreads barriers,
// for the long tail of iterations that carry little work (a barrier there
// costs ~0.1 us instead of a few us).  Either kernel stops at an iteration
// boundary when the other mode suits the work better and records where to
// resume (Ctl::rs); the host queues a grid launch and a block launch back to
// back, so the handover needs no host round trip.
//
// Each iteration:
//   SELECT   a maximal superior edge set (Section IV, Definition 6 and the
//            union after it; Algorithm 2 made deterministic).  An edge's
//            constrained endpoints are those whose core equals the edge's
//            core number min(core(u), core(v)).  In claim rounds every
//            eligible edge writes its priority fmix64(key) into its
//            constrained endpoints with atomicMin and wins when it holds all
//            of them; winners take their endpoints and edges touching a taken
//            endpoint wait for the next iteration.  The result is the greedy
//            (lexicographically first) maximal set in priority order.
//   APPLY    insert / delete the selected edges in the slack CSR and move
//            SD (superior degree, Definition 7) of constrained endpoints.
//   insert:  positive and negative search of Algorithms 3-4, run as
//            breadth-first waves in which both progress together (single-
//            block mode) or as a task queue without level barriers (grid
//            mode, cm_search.cuh: the order of processing does not
//            change the result).  The
//            constrained endpoints are the first frontier.  Processing a
//            frontier vertex v adds CSD(v) (Definition 8) to its support
//            count, which already holds one decrement per evicted neighbour
//            (the paper's pre-decremented cd).  If the count exceeds k, v
//            visits its unvisited core-k neighbours with SD > k (the next
//            frontier); otherwise v is evicted (Lemma 8).  An evicted vertex
//            takes one from the count of every core-k neighbour with SD > k,
//            visited or not; a processed neighbour whose count falls to k is
//            evicted too (InsertRemove, Algorithm 4).  Frontier and evictions
//            of a wave run in the same phase, so evictions prune the search
//            as it grows.  COMMIT: processed vertices still above k rise by
//            one (the last step of Algorithm 1, Lemma 7).
//   delete:  EVICT in waves (or, grid-wide, as queued tasks) from the
//            constrained endpoints whose SD fell below k (Algorithm 6); an
//            evicted vertex drops by one and takes
//            one from the support (initially SD) of every core-k neighbour,
//            which leaves when its support falls below k (DeleteRemove,
//            Algorithm 7; the last step of Algorithm 5).
//   FIX-UP   recompute SD of moved vertices and adjust SD of unmoved
//            neighbours whose core equals the moved vertex's new core
//            (insert) or old core (delete).  It only writes SD, which the
//            next iteration first reads in APPLY, so it runs inside the next
//            iteration's first claim phase and costs no barrier of its own.
// All levels run together on the cores of the iteration's start: searches
// and evictions only ever follow neighbours of the vertex's own level.
//
// The per-vertex bodies and the per-iteration vertex word are in cm_vertex.cuh.
//
// In single-block mode a wave's vertices get one warp each (fetched
// dynamically); one with at least 256 slots is deferred and then processed by
// the whole block.  The grid's searches and fix-ups are in cm_search.cuh.
#include <type_traits>

#include "cm_common.cuh"
#include "cm_launch.h"
#include "cm_search.cuh"
#include "cm_vertex.cuh"

namespace cm {

constexpr int kBlockThreads = 512;    // single-block mode
// kGridThreads (cm_launch.h), with two blocks per SM: 80 registers a thread.  The search
// needs about 90; at 64 (512 threads) the spills, which are written through to
// L2, cost more than the warps gain.  512 / 448 / 384 / 320 threads, one pass
// of inserts and deletes: R-MAT scale 20 with 10^4 edges 3.4 / 3.2 / 3.0 / 3.1
// ms, Erdos-Renyi 2*10^6 with 10^4 4.2 / 4.1 / 4.0 / 3.9 ms, R-MAT scale 24
// with 10^3 degree-proportional - / 10.3 / 9.7 / 10.4 ms.
static_assert(kGridThreads / 32 == kGridWarps, "one search buffer per grid-mode warp");
constexpr int kMaxBig = 64;
constexpr int kBlockLenSingle = 256;   // single-block mode: the block scans lists from this size

// The iteration loop's state while a grid-wide search or fix-up runs.
struct LoopState {
    unsigned long long nrem, nrem_next, vq0, eq0, cq0, vq_t, eq_t, cq_t, fx_lo, fx_hi, fx_long;
    REdge *Rc, *Rn;
    unsigned long long t_last;
    long long remsum, iters0;
    uint32_t e, e0;
    int iters, rounds, waves;
};

template <int MODE>
struct Barrier {
    Ctl* c;
    uint32_t expect;
    unsigned long long limit;
    unsigned long long t_last;
    bool timer;
    __device__ bool operator()(int phase) {
        bool ok = MODE == 0 ? grid_sync(c, expect, limit) : block_sync(c);
        if (timer) {
            unsigned long long now = gtimer();
            c->ph[phase] += now - t_last;
            c->st[ST_BARRIERS] += 1;
            t_last = now;
        }
        return ok;
    }
};

// ---------------------------------------------------------------- vertex loop (waves)
// Single-block mode: runs body(v, Group) for every vertex of ring[lo, hi),
// one warp per vertex.  Each warp's first vertex is dealt by its warp index;
// the rest are fetched dynamically (counter *ctr, zeroed at every barrier).
// A vertex with at least kBlockLenSingle slots is deferred by the warp that
// fetched it and then processed by the whole block, so a long list does not
// hold a wave on one warp.  Every thread of the launch must call it.
template <class Body>
__device__ __forceinline__ void for_each_vertex(const DevGraph& g, unsigned long long* ctr, const int32_t* ring,
                                                unsigned long long qm, unsigned long long lo, unsigned long long hi,
                                                Body body) {
    const int lane = lane_id();
    __shared__ int s_big[kMaxBig];
    __shared__ int s_nbig;
    if (threadIdx.x == 0) s_nbig = 0;
    __syncthreads();
    constexpr unsigned nw = kBlockThreads / 32;
    const unsigned long long cnt = hi - lo;
    unsigned long long j = threadIdx.x >> 5;
    for (;;) {
        if (j >= cnt) break;
        const int v = ring[(lo + j) & qm];
        int defer = 0;
        if (lane == 0 && g.end[v] >= kBlockLenSingle) {
            int s = atomicAdd(&s_nbig, 1);
            if (s < kMaxBig) {
                s_big[s] = v;
                defer = 1;
            }
        }
        if (!__shfl_sync(0xffffffffu, defer, 0)) body(v, WarpGroup{});
        if (cnt <= nw) break;   // every vertex was dealt by index
        if (lane == 0) j = nw + atomicAdd(ctr, 1ull);
        j = __shfl_sync(0xffffffffu, j, 0);
    }
    __syncthreads();
    const int nb = min(s_nbig, kMaxBig);
    for (int b = 0; b < nb; b++) {
        body(s_big[b], BlockGroup<kBlockThreads>{});
        __syncthreads();
    }
}

// Single-block mode: adjacency slots of the vertices of ring ranges
// [lo0, hi0) and [lo1, hi1) (a wave about to run), summed by the block.
__device__ __forceinline__ long long wave_slots(const DevGraph& g, const int32_t* r0, unsigned long long lo0,
                                                unsigned long long hi0, const int32_t* r1, unsigned long long lo1,
                                                unsigned long long hi1, unsigned long long qm) {
    __shared__ long long s_sum;
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    long long part = 0;
    for (unsigned long long i = lo0 + threadIdx.x; i < hi0; i += blockDim.x) part += g.end[r0[i & qm]];
    for (unsigned long long i = lo1 + threadIdx.x; i < hi1; i += blockDim.x) part += g.end[r1[i & qm]];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane_id() == 0 && part) atomicAdd((unsigned long long*)&s_sum, (unsigned long long)part);
    __syncthreads();
    const long long total = s_sum;
    __syncthreads();
    return total;
}

// An edge's core number k = min(core(lo), core(hi)) and its constrained
// endpoints: those whose core is k (Definition 6), except pinned vertices.
// An insertion never has pinned vertices (they exist only while a vertex
// deletion removes their edges), so it reads the cores from the 4-byte keys.
__device__ __forceinline__ void edge_level(const DevGraph& g, const REdge& E, bool ins, int& k, bool& clo,
                                           bool& chi) {
    if (ins) {
        const int a = key_core(g.kc[E.lo]);
        const int b = key_core(g.kc[E.hi]);
        k = min(a, b);
        clo = a == k;
        chi = b == k;
        return;
    }
    const int2 a = g.hc[E.lo];
    const int2 b = g.hc[E.hi];
    k = min(a.x, b.x);
    clo = a.x == k && a.y < PIN_SD;
    chi = b.x == k && b.y < PIN_SD;
}

// An edge's selection priority (smaller wins): fmix64 of its canonical key,
// a bijection, or the key itself (lexicographic order of (lo, hi)).
__device__ __forceinline__ unsigned long long edge_prio(const REdge& E, bool by_key) {
    const unsigned long long key = ekey(E.lo, E.hi);
    return by_key ? key : fmix64(key);
}

// Selection, claim phase of round r.  An edge already selected or blocked
// that did not claim in round r-1 has nothing to do and gathers nothing.
__device__ __forceinline__ void claim_edge(const DevGraph& g, REdge* R, long long i, int r, uint32_t e, bool by_key,
                                           bool ins) {
    REdge E = R[i];
    const uint32_t f = E.flags;
    const bool claimed_last = r > 0 && (f >> 2) == (uint32_t)r;
    if ((f & (F_SEL | F_BLK)) && !claimed_last) return;
    int k; bool clo, chi;
    edge_level(g, E, ins, k, clo, chi);
    if (claimed_last) {   // claimed in round r-1: clear that buffer
        unsigned long long* cb = ((r - 1) & 1) ? g.claim1 : g.claim0;
        if (clo) cb[E.lo] = CLAIM_FREE;
        if (chi) cb[E.hi] = CLAIM_FREE;
    }
    if (f & (F_SEL | F_BLK)) return;
    if ((clo && g.taken[E.lo] == e) || (chi && g.taken[E.hi] == e)) {
        R[i].flags = f | F_BLK;
        return;
    }
    const unsigned long long prio = edge_prio(E, by_key);
    unsigned long long* cb = (r & 1) ? g.claim1 : g.claim0;
    if (clo) atomicMin(&cb[E.lo], prio);
    if (chi) atomicMin(&cb[E.hi], prio);
    R[i].flags = (f & 3u) | ((uint32_t)(r + 1) << 2);
}

// Selection, check phase of round r.  Returns 1 if the edge claimed and lost.
__device__ __forceinline__ int check_edge(const DevGraph& g, REdge* R, long long i, int r, uint32_t e,
                                          uint32_t& nsel, bool by_key, bool ins) {
    REdge E = R[i];
    if ((E.flags >> 2) != (uint32_t)(r + 1)) return 0;
    int k; bool clo, chi;
    edge_level(g, E, ins, k, clo, chi);
    const unsigned long long prio = edge_prio(E, by_key);
    const unsigned long long* cb = (r & 1) ? g.claim1 : g.claim0;
    bool win = (!clo || cb[E.lo] == prio) && (!chi || cb[E.hi] == prio);
    if (!win) return 1;
    R[i].flags = E.flags | F_SEL;
    if (clo) g.taken[E.lo] = e;
    if (chi) g.taken[E.hi] = e;
    nsel++;
    return 0;
}

constexpr unsigned long long kMaxPasses = 256;   // launch pairs per phase of a captured step

// Inside a captured update step the launch pairs (grid kernel, then
// single-block kernel) are the body of a conditional WHILE node: the
// single-block kernel ends every pass by setting the node's condition, so
// the loop runs until the call is done or failed with no host round trip.
__device__ __forceinline__ void loop_control(const MaintainParams& P, Ctl* C) {
    if (!P.use_cond || threadIdx.x != 0) return;
    const unsigned long long n = C->passes + 1;
    C->passes = n;
    int err = vload32(&C->error);
    const int done = *(volatile int*)&C->rs.done;
    if (!err && !done && n >= kMaxPasses) {
        atomicCAS(&C->error, 0, E_ITER_LIMIT);
        err = 1;
    }
    cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, (!err && !done) ? 1u : 0u);
}

// One kernel per mode and operation (OP 0 insert, 1 delete): each carries one
// search only, which keeps its registers and instructions within bounds.
template <int MODE, int OP>
__global__ void __launch_bounds__(MODE == 0 ? kGridThreads : kBlockThreads, MODE == 0 ? 2 : 1)
    maintain_kernel(MaintainParams P) {
    Ctl* C = P.ctl;
    const DevGraph g = P.g;
    // where to resume (the host or the other mode wrote it before this launch)
    const int done0 = *(volatile int*)&C->rs.done;
    const int want = *(volatile int*)&C->rs.want;
    if (done0 || want != MODE || vload32(&C->error)) {
        if (MODE == 1) loop_control(P, C);
        return;
    }
    const int lane = lane_id();
    if (MODE == 0) {   // shared memory starts undefined: no search is quiescent yet, no warp holds arena room
        if (threadIdx.x == 0) s_quiet = ~0u;
        WarpBuf& B = reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5];
        if (lane == 0) B.slab = B.slab_end = 0;
        if (lane < 7) B.st[lane] = 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) C->rec_top = 0;
        __syncthreads();
    }
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const unsigned long long qm = P.qmask;
    const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
    Barrier<MODE> sync{C, P.expect, P.limit_ns, gtimer(), leader};
    const uint32_t rsel0 = *(volatile uint32_t*)&C->rs.rsel;
    REdge* Rc = rsel0 ? P.R1 : P.R0;
    REdge* Rn = rsel0 ? P.R0 : P.R1;
    unsigned long long nrem = vload64(&C->rs.nrem);
    uint32_t e = *(volatile uint32_t*)&C->rs.epoch;
    uint32_t e0 = e;         // records of this launch carry stamps from here on
    long long iters0 = *(volatile long long*)&C->rs.iters;
    unsigned long long vq_t = vload64(&C->tail[0]), eq_t = vload64(&C->tail[1]), cq_t = vload64(&C->tail[2]);
    // grid mode: the task queue starts empty for every search
    auto reset_tasks = [&]() {
        if (leader) {
            C->task_head = 0;
            C->task_tail = P.phantom_task ? 1 : 0;   // a phantom is never queued: no quiescence
            C->task_done = 0;
            C->hub_created = 0;
            C->hub_finished = 0;
        }
    };
    LocalStats ls;
    int iters = 0, rounds = 0, waves = 0;   // per launch (a call is capped far below 2^31 iterations)
    long long remsum = 0;
    // resume inside the search waves of an iteration the single-block mode began
    bool mid = *(volatile int*)&C->rs.mid != 0;
    bool escalate = false;
    unsigned long long nrem_next = 0, vq0 = 0, eq0 = 0, cq0 = 0, flo = 0, fhi = 0, elo = 0, ehi = 0;
    if (mid) {
        nrem_next = nrem;                  // edges left for the next iteration, in buffer rsel
        REdge* t0 = Rc;
        Rc = Rn;
        Rn = t0;
        vq0 = vload64(&C->rs.vq0);
        eq0 = vload64(&C->rs.eq0);
        cq0 = vload64(&C->rs.cq0);
        flo = vload64(&C->rs.flo);
        fhi = vload64(&C->rs.fhi);
        elo = vload64(&C->rs.elo);
        ehi = vload64(&C->rs.ehi);
    }
    bool ok = true;
    // pending SD fix-up of the previous iteration
    bool fx = false;
    unsigned long long fx_lo = 0, fx_hi = 0;
    // a call whose ingest kept no edge (its count read on the device) is done at once
    int next_want = MODE, finished = (!mid && nrem == 0) ? 1 : 0;
    const int32_t* FXQ = OP == 0 ? P.CQ : P.EQ;
    [[maybe_unused]] unsigned long long fx_long = 0;   // insert: chunks of long lists queued for it; delete: hubs met

    // Runs a grid-wide search or fix-up with the loop's state parked in shared
    // memory meanwhile (every thread holds the same values): see flush_stats.
    [[maybe_unused]] auto parked = [&](auto work) {
        WarpBuf& B = reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5];
        flush_stats(B, ls);
        __shared__ LoopState S;
        __syncthreads();   // the last reader of S is done
        if (threadIdx.x == 0) {
            S = LoopState{nrem, nrem_next, vq0, eq0, cq0, vq_t, eq_t, cq_t, fx_lo, fx_hi, fx_long, Rc, Rn, sync.t_last,
                          remsum, iters0, e, e0, iters, rounds, waves};
            s_search_t0 = gtimer();
        }
        __syncthreads();
        const bool fine = work(S);
        nrem = S.nrem;
        nrem_next = S.nrem_next;
        vq0 = S.vq0;
        eq0 = S.eq0;
        cq0 = S.cq0;
        vq_t = S.vq_t;
        eq_t = S.eq_t;
        cq_t = S.cq_t;
        Rc = S.Rc;
        Rn = S.Rn;
        sync.t_last = S.t_last;
        remsum = S.remsum;
        iters0 = S.iters0;
        e = S.e;
        e0 = S.e0;
        iters = S.iters;
        rounds = S.rounds;
        waves = S.waves;
        return fine;
    };
    [[maybe_unused]] auto search = [&](auto del) {
        if constexpr (MODE == 0) {
            return parked([&](const LoopState& S) {
                return async_search<decltype(del)::value>(g, C, P, S.e, S.e0, OP == 0 && S.nrem_next > 0);
            });
        } else {
            return true;
        }
    };
    // the pending SD fix-up; false: a barrier failed
    auto fixup = [&]() {
        if constexpr (MODE == 0) {
            // An insertion queues the chunks of long lists as it commits; a
            // deletion here, at the price of a barrier (~4 us), if its search
            // met a hub or the vertices are many: with the line at one a warp
            // R-MAT scale 20 deletions of 10^4 edges took 0.19 ms, not 0.185.
            bool queued = true;
            if (OP == 1) {
                queued = fx_long > 0 || fx_hi - fx_lo > 8ull * (unsigned long long)nwarps;
                fx_long = 0;
                if (queued) {
                    for (unsigned long long i = fx_lo + gwarp * 32 + lane; i < fx_hi; i += nwarps * 32) {
                        const int v = __ldcg(FXQ + (i & qm));
                        list_long(g, C, P, v, g.end[v]);
                    }
                    if (!sync(PH_FIXUP)) return false;
                    fx_long = vload64(&C->spc[2]);
                }
            }
            return parked([&](const LoopState& S) {
                fixup_grid<OP>(g, C, P, FXQ, S.fx_lo, S.fx_hi, queued, S.fx_long, S.e - 1, S.e0, S.nrem > 0);
                return true;
            });
        } else {
            for_each_vertex(g, &C->pc[2], FXQ, qm, fx_lo, fx_hi,
                            [&](int v, auto grp) { fixup_vertex<decltype(grp)>(g, v, e - 1, OP, ls); });
            return true;
        }
    };

    while (mid || nrem > 0) {
      if (!mid) {
        if (iters0 + iters >= P.max_iters) {
            if (leader) atomicCAS(&C->error, 0, E_ITER_LIMIT);
            ok = false;
            break;
        }
        remsum += (long long)nrem;
        // ------------------------------------------------ SELECT
        int r = 0;
        const bool lone = nrem == 1 && !fx;
        if (lone) {   // one edge is the maximal set: no claim, no barrier (this thread applies it, too)
            if (MODE == 0) reset_tasks();
            if (leader) {
                Rc[0].flags = F_SEL;
                ls.sel++;
            }
            r = 1;
        }
        while (!lone) {
            if (r == 0 && fx) {
                if (!(ok = fixup())) break;
                fx = false;
            }
            if (MODE == 0 && r == 0) reset_tasks();   // nobody pushes tasks before APPLY
            for (long long base = gwarp * 32; base < (long long)nrem; base += nwarps * 32) {
                long long i = base + lane;
                if (i < (long long)nrem) claim_edge(g, Rc, i, r, e, P.sel_key != 0, OP == 0);
            }
            if (!(ok = sync(PH_CLAIM))) break;
            int lost = 0;
            for (long long base = gwarp * 32; base < (long long)nrem; base += nwarps * 32) {
                long long i = base + lane;
                if (i < (long long)nrem) lost += check_edge(g, Rc, i, r, e, ls.sel, P.sel_key != 0, OP == 0);
            }
            lost = warp_sum(lost);
            if (lane == 0 && lost) atomicAdd(&C->pc[0], (unsigned long long)lost);
            if (!(ok = sync(PH_CHECK))) break;
            r++;
            if (vload64(&C->spc[0]) == 0) break;           // no edge lost: the set is maximal
            if (P.sel_rounds > 0 && r >= P.sel_rounds) break;   // capped: a superior edge set all the same
        }
        if (!ok) break;
        rounds += r;
        // ------------------------------------------------ APPLY
        vq0 = vq_t;
        eq0 = eq_t;
        cq0 = cq_t;
        for (long long base = gwarp * 32; base < (long long)nrem; base += nwarps * 32) {
            long long i = base + lane;
            bool valid = i < (long long)nrem;
            REdge E = {0, 0, 0, 0};
            bool sel = false, s_lo = false, s_hi = false;
            if (valid) {
                E = Rc[i];
                int k = 0; bool clo = false, chi = false;
                // only a selected edge or one that claimed in the final round needs its level
                if ((E.flags & F_SEL) || (E.flags >> 2) == (uint32_t)r) edge_level(g, E, OP == 0, k, clo, chi);
                if ((E.flags >> 2) == (uint32_t)r) {     // claimed in the final round
                    unsigned long long* cb = ((r - 1) & 1) ? g.claim1 : g.claim0;
                    if (clo) cb[E.lo] = CLAIM_FREE;
                    if (chi) cb[E.hi] = CLAIM_FREE;
                }
                sel = (E.flags & F_SEL) != 0;
                if (sel) {
                    if constexpr (OP == 0) {
                        int pu = atomicAdd(&g.end[E.lo], 1), pv = atomicAdd(&g.end[E.hi], 1);
                        if (pu < g.cap[E.lo] && pv < g.cap[E.hi]) {
                            g.adj[g.off[E.lo] + pu] = E.hi;
                            g.adj[g.off[E.hi] + pv] = E.lo;
                            g.idx[E.bkt].slo = pu;
                            g.idx[E.bkt].shi = pv;
                        } else {
                            atomicCAS(&C->error, 0, E_CAPACITY);
                        }
                        atomicAdd(&g.deg[E.lo], 1);
                        atomicAdd(&g.deg[E.hi], 1);
                        // a constrained endpoint's SD rises; with SD > k it roots the search
                        // (one selected edge per constrained endpoint and level: this is the
                        // only SD change of the endpoint in APPLY, so its key bit follows it)
                        if (MODE == 0) {
                            if (clo) rec_link(P, e0, E.lo, k, E.hi, !chi);
                            if (chi) rec_link(P, e0, E.hi, k, E.lo, !clo);
                        }
                        if (clo) {
                            const int sd = atomicAdd(&g.hc[E.lo].y, 1) + 1;
                            if (sd > k) atomicOr(&g.kc[E.lo], 1u);
                            s_lo = sd > k && visit(g, C, E.lo, e);
                        }
                        if (chi) {
                            const int sd = atomicAdd(&g.hc[E.hi].y, 1) + 1;
                            if (sd > k) atomicOr(&g.kc[E.hi], 1u);
                            s_hi = sd > k && visit(g, C, E.hi, e);
                        }
                    } else {
                        Bucket b = g.idx[E.bkt];
                        if (b.slo >= 0 && b.slo < g.end[E.lo] && b.shi >= 0 && b.shi < g.end[E.hi]) {
                            g.adj[g.off[E.lo] + b.slo] = HOLE;
                            g.adj[g.off[E.hi] + b.shi] = HOLE;
                        } else {
                            atomicCAS(&C->error, 0, E_CAPACITY);
                        }
                        g.idx[E.bkt].key = KEY_TOMB;
                        atomicSub(&g.deg[E.lo], 1);
                        atomicSub(&g.deg[E.hi], 1);
                        if (clo) {
                            int m = atomicSub(&g.hc[E.lo].y, 1) - 1;
                            if (m <= k) atomicAnd(&g.kc[E.lo], ~1u);
                            if (m < k) { s_lo = true; g.chg[E.lo] = e; }
                        }
                        if (chi) {
                            int m = atomicSub(&g.hc[E.hi].y, 1) - 1;
                            if (m <= k) atomicAnd(&g.kc[E.hi], ~1u);
                            if (m < k) { s_hi = true; g.chg[E.hi] = e; }
                        }
                    }
                }
                E.flags = 0;
            }
            warp_push_edge(&C->pc[1], Rn, valid && !sel, E);
            // roots: frontier (insert) or evicted (delete) constrained endpoints
            push_vertex<MODE == 0>(C, P, s_lo, E.lo, OP == 0 ? 0 : 1);
            push_vertex<MODE == 0>(C, P, s_hi, E.hi, OP == 0 ? 0 : 1);
        }
        if (!(ok = sync(PH_APPLY))) break;
        nrem_next = vload64(&C->spc[1]);
        vq_t = vload64(&C->stail[0]);
        eq_t = vload64(&C->stail[1]);
        flo = vq0;
        fhi = vq_t;
        elo = eq0;
        ehi = eq_t;
      }
      const bool resumed = mid;
      mid = false;

        if constexpr (OP == 0) {
            // -------------------------------------------- SEARCH (insert): frontier + evictions
            if constexpr (MODE == 0) {
                if (resumed) {   // the single-block mode began this search
                    reset_tasks();
                    if (!(ok = sync(PH_APPLY))) break;
                    seed_tasks(C, P, P.VQ, flo, fhi, T_FRONT);
                    seed_tasks(C, P, P.EQ, elo, ehi, T_EVICT);
                    if (!(ok = sync(PH_APPLY))) break;
                }
                waves++;
                ok = search(std::false_type{});
                if (!(ok = sync(PH_DISCOVER) && ok)) break;
                fhi = vload64(&C->stail[0]);
                ehi = vload64(&C->stail[1]);
            } else {
                while (fhi > flo || ehi > elo) {
                    // a wave too big for one block (by vertices, or by the slots
                    // of its vertices' lists) goes to the grid
                    if ((fhi - flo) + (ehi - elo) > (unsigned long long)P.big_wave ||
                        wave_slots(g, P.VQ, flo, fhi, P.EQ, elo, ehi, qm) > P.big_slots) {
                        escalate = true;
                        break;
                    }
                    waves++;
                    for_each_vertex(g, &C->pc[2], P.VQ, qm, flo, fhi, [&](int v, auto grp) {
                        process_frontier<decltype(grp)>(g, C, P, v, load_vinfo(g, v), e, ls);
                    });
                    for_each_vertex(g, &C->pc[3], P.EQ, qm, elo, ehi, [&](int v, auto grp) {
                        evict_insert_vertex<decltype(grp)>(g, C, P, load_vinfo(g, v), e, ls);
                    });
                    if (!(ok = sync(PH_DISCOVER))) break;
                    flo = fhi;
                    fhi = vload64(&C->stail[0]);
                    elo = ehi;
                    ehi = vload64(&C->stail[1]);
                }
            }
            if (!ok || escalate) break;
            vq_t = fhi;
            eq_t = ehi;
            // -------------------------------------------- COMMIT (insert): survivors rise
            for (long long base = gwarp * 32; base < (long long)(vq_t - vq0); base += nwarps * 32) {
                long long i = base + lane;
                bool up = false;
                int v = 0, len = 0;
                if (i < (long long)(vq_t - vq0)) {
                    v = P.VQ[(vq0 + i) & qm];
                    const int core = g.hc[v].x;
                    const int support = ww(g.hw[v]);
                    if (support > core) {
                        if (MODE == 0) len = g.end[v];
                        g.hc[v].x = core + 1;
                        g.kc[v] = key_of(core + 1, 0);   // bit set by the SD fix-up
                        g.chg[v] = e;
                        up = true;
                    }
                }
                warp_push(&C->tail[2], P.CQ, qm, up, v);
                if constexpr (MODE == 0) list_long(g, C, P, v, len);
            }
            if (!(ok = sync(PH_COMMIT))) break;
            fx_long = vload64(&C->spc[2]);
            cq_t = vload64(&C->stail[2]);
            fx = cq_t > cq0;
            fx_lo = cq0;
            fx_hi = cq_t;
        } else {
            // -------------------------------------------- EVICT (delete); evicted vertices drop by one
            if constexpr (MODE == 0) {
                if (resumed) {
                    reset_tasks();
                    if (!(ok = sync(PH_APPLY))) break;
                    seed_tasks(C, P, P.EQ, elo, ehi, T_EVICT);
                    if (!(ok = sync(PH_APPLY))) break;
                }
                waves++;
                ok = search(std::true_type{});
                if (!(ok = sync(PH_EVICT) && ok)) break;
                ehi = vload64(&C->stail[1]);
                fx_long = vload64(&C->hub_created);
            } else {
                while (ehi > elo) {
                    if (ehi - elo > (unsigned long long)P.big_wave ||
                        wave_slots(g, P.EQ, elo, ehi, P.EQ, 0, 0, qm) > P.big_slots) {
                        escalate = true;
                        break;
                    }
                    waves++;
                    for_each_vertex(g, &C->pc[2], P.EQ, qm, elo, ehi, [&](int v, auto grp) {
                        evict_delete_vertex<decltype(grp)>(g, C, P, v, load_vinfo(g, v), e, ls);
                    });
                    if (!(ok = sync(PH_EVICT))) break;
                    elo = ehi;
                    ehi = vload64(&C->stail[1]);
                }
            }
            if (!ok || escalate) break;
            eq_t = ehi;
            fx = eq_t > eq0;
            fx_lo = eq0;
            fx_hi = eq_t;
        }
        // ------------------------------------------------ next iteration, or hand over
        const unsigned long long nsel = nrem - nrem_next;
        // (a grid-wide insertion logs no evictions: they are about as many as the visits)
        const unsigned long long work = (vq_t - vq0) * (MODE == 0 && OP == 0 ? 2 : 1) + (eq_t - eq0) +
                                        (cq_t - cq0) + nsel;
        REdge* t = Rc;
        Rc = Rn;
        Rn = t;
        nrem = nrem_next;
        e++;
        iters++;
        if (nrem == 0) {
            finished = 1;
            break;
        }
        if (P.yield_each) {   // debug: end the launch here (the fix-up below still runs); resume in this mode
            next_want = MODE;
            break;
        }
        if (MODE == 0 && nrem <= (unsigned long long)P.small_edges && work <= (unsigned long long)P.small_work) {
            next_want = 1;
            break;
        }
        if (MODE == 1 && work > (unsigned long long)P.big_work) {
            next_want = 0;
            break;
        }
    }
    if (ok && fx) {
        ok = fixup() && sync(PH_FIXUP);
    }
    // statistics: one atomic per warp
    uint32_t tot[7] = {ls.vis, ls.visl, ls.ev, ls.evl, ls.ch, ls.chl, ls.sel};
    const int slot[7] = {ST_VISITED, ST_VISSLOTS, ST_EVICTED, ST_EVSLOTS, ST_CHANGED, ST_CHSLOTS, ST_SELECTED};
#pragma unroll
    for (int i = 0; i < 7; i++) {
        unsigned long long t = __reduce_add_sync(0xffffffffu, tot[i]);
        if (MODE == 0) t += reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5].st[i];
        if (lane == 0 && t) atomicAdd(&C->st[slot[i]], t);
    }
    if (leader) {
        C->st[ST_ITERS] += (unsigned long long)iters;
        if (MODE == 0) C->st[ST_GRID_ITERS] += (unsigned long long)iters;
        C->st[ST_ROUNDS] += (unsigned long long)rounds;
        C->st[ST_WAVES] += (unsigned long long)waves;
        C->st[ST_REMSUM] += (unsigned long long)remsum;
        if (ok && escalate) {
            C->rs.nrem = nrem_next;
            C->rs.rsel = Rn == P.R1 ? 1u : 0u;
            C->rs.epoch = e;
            C->rs.iters = iters0 + iters;
            C->rs.done = 0;
            C->rs.want = 0;
            C->rs.mid = 1;
            C->rs.vq0 = vq0;
            C->rs.eq0 = eq0;
            C->rs.cq0 = cq0;
            C->rs.flo = flo;
            C->rs.fhi = fhi;
            C->rs.elo = elo;
            C->rs.ehi = ehi;
            __threadfence();
        } else if (ok) {
            C->rs.nrem = nrem;
            C->rs.rsel = Rc == P.R1 ? 1u : 0u;
            C->rs.epoch = e;
            C->rs.iters = iters0 + iters;
            C->rs.done = finished;
            C->rs.want = next_want;
            C->rs.mid = 0;
            __threadfence();
        }
    }
    if (MODE == 1) loop_control(P, C);   // thread 0 is the leader: its writes above come first
}

static const void* maintain_kernel(int mode, int op) {
    return mode == 0 ? (op == 0 ? (const void*)maintain_kernel<0, 0> : (const void*)maintain_kernel<0, 1>)
                     : (op == 0 ? (const void*)maintain_kernel<1, 0> : (const void*)maintain_kernel<1, 1>);
}

// Resident blocks per SM of the grid-mode kernels (both operations).  Their
// search buffers take 40 KB of shared memory per block; the attribute is only
// needed past 48 KB.
int maintain_blocks_per_sm(int threads) {
    int least = 0;
    for (int op = 0; op < 2; op++) {
        const void* f = maintain_kernel(0, op);
        int nb = 0;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSearchSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, threads, kSearchSmem) != cudaSuccess)
            return 0;
        least = op == 0 || nb < least ? nb : least;
    }
    return least;
}

// Cooperative (co-resident blocks, which the grid barrier needs); the
// attribute form also records into a graph under stream capture.
cudaError_t launch_maintain(const MaintainParams& p, int blocks, int threads, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = kSearchSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    MaintainParams q = p;
    void* args[] = {&q};
    return cudaLaunchKernelExC(&cfg, maintain_kernel(0, p.op), args);
}

cudaError_t launch_maintain_block(const MaintainParams& p, cudaStream_t s) {
    MaintainParams q = p;
    void* args[] = {&q};
    return cudaLaunchKernel(maintain_kernel(1, p.op), dim3(1), dim3(kBlockThreads), args, 0, s);
}

}  // namespace cm
