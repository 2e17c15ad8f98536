// cm_peel.cuh -- full decomposition by level-synchronous bucket peeling,
// shared by the graph store (cm_store.cu) and the allocation-free entry
// point on a caller's CSR (cm_noalloc.cu).
//
// The static O(m) decomposition the paper cites, run level by level: at
// level k every remaining vertex whose working degree is at most k gets core
// k and leaves; each departure takes one degree from every neighbour, and a
// neighbour that falls to k leaves at the same level.  Empty levels are
// skipped to the smallest remaining degree.
//
// What bounds it: a graph has hundreds of levels, and a level's work is
// small (10^3 to 10^4 departures), so the time is levels x (dependent round
// trips + barriers), not bytes; below that lies the rate of the random
// returning atomics of the decrements (about 130 G/s measured).  Hence:
//
//   * one grid barrier per level.  Every block owns a share of the remaining
//     vertices (groups of 32 ids dealt round robin, compacted in place), scans
//     it, and follows the cascades that its own decrements start in a queue in
//     shared memory, with block barriers only.  No barrier separates the scan
//     from the decrements: a vertex is claimed by a compare-and-swap on its
//     core, so a scan that sees a degree another block has just brought to k
//     does no harm.
//   * the lists of up to 1024 departing vertices are walked together, quad by
//     quad (four slots, one 16-byte load), in windows of 512 slots per warp
//     with 16 decrements per lane in flight, whatever the lists' lengths.
//   * what one block should not do alone goes to the whole grid: vertices
//     beyond the queue's room or beyond kPeelQuads of a round, cascades of
//     more than kPeelRounds rounds, and lists of more than kSpread slots (as
//     chunks) are written to shared lists that all blocks take after the
//     barrier; only such levels pay further barriers.
//   * the barrier is one atomic per block on a word that also carries the
//     level's totals (vertices kept, whether any left, whether anything was
//     shared), and the waiters poll that word: two trips.
//
// Measured (GB300, edge factor 16): R-MAT scale 24 (297 levels) 24.5 -> 15.3
// ms, R-MAT scale 20 from a CSR 17.1 -> 4.9 ms, against one barrier per wave,
// one warp per list of up to 2047 slots and a separate phase for longer ones
// (1,598 barriers of about 15 us at scale 24; now 417).  A level without
// departures takes 5 us, one with 10^3 about 15.
#pragma once
#include "cm_common.cuh"

namespace cm {

constexpr int kUnpeeled = -2;          // core of a vertex still in the graph
constexpr int kPeelThreads = 1024;     // one block per SM
constexpr int kPeelWarps = kPeelThreads / 32;
constexpr int kPeelQueue = 3072;       // departing vertices a block holds (twice)
constexpr int kPeelTile = 8;           // list entries per thread and scan step
constexpr int kSpread = 16384;         // lists longer than this are shared by the grid ...
constexpr int kSpreadChunk = 4096;     // ... in chunks of this many slots
// How much of a cascade one block follows before the grid takes over: rounds,
// and quads walked in a round (one window a warp).  Without the limits one
// block walked 7*10^6 slots of the densest core's collapse while the others
// waited (R-MAT scale 24 59 ms); 64 rounds and 16,384 quads 19.8, 16 and
// 16,384 19.4, 8 and 4,096 18.8, 4 and 4,096 19.1, 4 and 1,024 20.6 ms (with
// the SD pass that follows).
constexpr int kPeelRounds = 8;
constexpr int kPeelQuads = 4096;

struct PeelShared {
    int32_t x[2][kPeelQueue];          // departing vertices: this round's and the next's
    long long off[kPeelThreads];       // lists of the vertices being walked
    int32_t len[kPeelThreads];
    int32_t pre[kPeelThreads];         // running count of their quads
    int32_t wsum[kPeelWarps];
    int n[2];                          // entries of x (may count past its end)
    int keep, mx, peeled, shared_out, upto;
    unsigned long long word;
};

// The arrays a peel works on besides the graph.
struct PeelWork {
    Ctl* ctl;
    int32_t* dcur;                     // working degrees
    int32_t* list;                     // remaining vertices, a region per block
    int32_t* far;                      // vertices handed to the grid (each at most once)
    unsigned long long* chunks;        // chunks of long lists: vertex << 32 | chunk
    unsigned long long chunk_cap;
    uint32_t blocks;
    unsigned long long limit_ns;
};

// Totals of a level, in one 64-bit word: 10 bits of arrivals, 11 of blocks
// that peeled, 11 of blocks that shared work, 32 of vertices kept.
__device__ __forceinline__ unsigned long long peel_word(int keep, bool peeled, bool shared_out) {
    return 1ull | (peeled ? 1ull << 10 : 0ull) | (shared_out ? 1ull << 21 : 0ull) |
           ((unsigned long long)(uint32_t)keep << 32);
}

// Grid barrier number `gen`: adds `mine` to its word and waits until every
// block has; returns the sum, or 0 on an error.  Four words take turns; a
// word is cleared two barriers before its next use.  The wait is bounded.
__device__ __forceinline__ unsigned long long peel_barrier(const PeelWork& W, PeelShared& S, unsigned gen,
                                                           unsigned long long mine) {
    Ctl* c = W.ctl;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long* w = &c->pw[gen & 3u];
        unsigned long long got;
        asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(got) : "l"(w), "l"(mine) : "memory");
        got += mine;
        const unsigned long long t0 = gtimer();
        for (unsigned spins = 1; (got & 1023ull) != W.blocks; spins++) {
            if ((spins & 15u) == 0) {
                if (vload32(&c->error)) break;
                if (gtimer() - t0 > W.limit_ns) {
                    atomicCAS(&c->error, 0, E_BARRIER_TIMEOUT);
                    break;
                }
            }
            got = ld_acquire64(w);
        }
        if ((got & 1023ull) != W.blocks) got = 0;
        if (blockIdx.x == 0) {
            c->pw[(gen + 2) & 3u] = 0;
            c->pm[(gen + 2) & 3u] = 0;
        }
        S.word = got;
    }
    __syncthreads();
    return S.word;
}

// Appends the set bits' vertices to the block's next queue; what does not
// fit is claimed here and handed to the grid.  Warp-collective.
template <class G>
__device__ __forceinline__ void peel_push(const G& g, const PeelWork& W, PeelShared& S, int q, int k, unsigned mask,
                                          const int (&id)[16]) {
    if (!__any_sync(0xffffffffu, mask != 0)) return;
    const int lane = lane_id();
    const int cnt = __popc(mask);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    int base = 0;
    if (lane == 31) base = atomicAdd(&S.n[q], incl);
    base = __shfl_sync(0xffffffffu, base, 31);
    int at = base + incl - cnt;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        if (!((mask >> i) & 1u)) continue;
        if (at < kPeelQueue) {
            S.x[q][at] = id[i];
        } else if (atomicCAS(g.core(id[i]), kUnpeeled, k) == kUnpeeled) {
            W.far[atomicAdd(&W.ctl->tail[0], 1ull)] = id[i];
            S.shared_out = 1;
            S.peeled = 1;
        }
        at++;
    }
}

// Walks the lists that the block's threads hold (vertex v; len 0: none): one
// degree off every neighbour; the ones that fall to k go to queue q.  Lists
// that begin after `limit` quads go to the grid instead.  Every thread of the
// block calls it.
template <class G>
__device__ __forceinline__ void peel_walk(const G& g, const PeelWork& W, PeelShared& S, int q, int k, int v,
                                          long long off, int len, int limit, unsigned long long& slots) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) S.upto = 0x7FFFFFFF;
    const int nq = g.quads(off, len);
    int incl = nq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) S.wsum[warp] = incl;
    S.off[threadIdx.x] = off;
    S.len[threadIdx.x] = len;
    __syncthreads();
    int before = lane < warp ? S.wsum[lane] : 0;   // kPeelWarps == 32: one per lane
    before = warp_sum(before);
    incl += before;
    S.pre[threadIdx.x] = incl;
    if (incl - nq < limit) {
        if (incl >= limit) S.upto = incl;   // the last one walked here
        slots += (unsigned)len;
    } else if (len > 0) {
        W.far[atomicAdd(&W.ctl->tail[0], 1ull)] = v;
        S.shared_out = 1;
    }
    __syncthreads();
    const int total = min(S.upto, S.pre[kPeelThreads - 1]);
    for (int w0 = warp * 128; w0 < total; w0 += kPeelWarps * 128) {
        int id[16];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int qi = w0 + u * 32 + lane;
            int o = 0;   // the owner: the first entry whose running count exceeds qi
#pragma unroll
            for (int step = kPeelThreads / 2; step > 0; step >>= 1)
                if (S.pre[o + step - 1] <= qi) o += step;
            const int first = o ? S.pre[o - 1] : 0;
            int4 a = make_int4(HOLE, HOLE, HOLE, HOLE);
            if (qi < total) a = g.quad(S.off[o], S.len[o], qi - first);
            id[4 * u] = a.x;
            id[4 * u + 1] = a.y;
            id[4 * u + 2] = a.z;
            id[4 * u + 3] = a.w;
        }
        int r[16];
#pragma unroll
        for (int i = 0; i < 16; i++) r[i] = id[i] >= 0 ? atomicSub(&W.dcur[id[i]], 1) : 0;
        unsigned mask = 0;
#pragma unroll
        for (int i = 0; i < 16; i++) mask |= id[i] >= 0 && r[i] == k + 1 ? 1u << i : 0u;
        peel_push(g, W, S, q, k, mask, id);
    }
    __syncthreads();   // the lists' entries are free again, the queue is complete
}

// The list of vertex v, if it is to be walked here: a long one is handed to
// the grid in chunks (unless there is no room for them).
template <class G>
__device__ __forceinline__ void peel_take(const G& g, const PeelWork& W, PeelShared& S, int v, long long& off,
                                          int& len) {
    g.list(v, off, len);
    if (len <= kSpread) return;
    const unsigned long long nch = (unsigned long long)((len + kSpreadChunk - 1) / kSpreadChunk);
    const unsigned long long at = atomicAdd(&W.ctl->tail[1], nch);
    for (unsigned long long c = 0; c < nch && at + c < W.chunk_cap; c++)
        W.chunks[at + c] = at + nch <= W.chunk_cap ? ((unsigned long long)(uint32_t)v << 32) | c : ~0ull;
    if (at + nch <= W.chunk_cap) {
        S.shared_out = 1;
        len = 0;
    }
}

// Follows the block's cascade: rounds over the queue until it stays empty,
// or for kPeelRounds (a long thin cascade, as along a path, must not hold the
// others at the barrier past its bounded wait): the rest goes to the grid.
// `q` is the queue to start with; returns the (empty) one to use next.
template <class G>
__device__ __forceinline__ int peel_drain(const G& g, const PeelWork& W, PeelShared& S, int q, int k,
                                          unsigned long long& slots) {
    for (int round = 0;; round++) {
        __syncthreads();
        const int n = min(S.n[q], kPeelQueue);
        if (n == 0) return q;
        if (round == kPeelRounds) {
            for (int i = threadIdx.x; i < n; i += kPeelThreads) {
                const int v = S.x[q][i];
                if (atomicCAS(g.core(v), kUnpeeled, k) == kUnpeeled) {
                    W.far[atomicAdd(&W.ctl->tail[0], 1ull)] = v;
                    S.shared_out = 1;
                    S.peeled = 1;
                }
            }
            __syncthreads();
            if (threadIdx.x == 0) S.n[q] = 0;
            __syncthreads();
            return q;
        }
        for (int b = 0; b < n; b += kPeelThreads) {
            const int i = b + (int)threadIdx.x;
            long long off = 0;
            int len = 0, v = 0;
            if (i < n) {
                v = S.x[q][i];
                if (atomicCAS(g.core(v), kUnpeeled, k) == kUnpeeled) {
                    S.peeled = 1;
                    peel_take(g, W, S, v, off, len);
                }
            }
            peel_walk(g, W, S, q ^ 1, k, v, off, len, kPeelQuads, slots);
        }
        if (threadIdx.x == 0) S.n[q] = 0;
        q ^= 1;
    }
}

// The whole decomposition; every block of a cooperative launch of W.blocks
// blocks of kPeelThreads threads calls it.  The control block's launch zone
// is zero at the start.
template <class G>
__device__ __forceinline__ void peel_graph(const G& g, const PeelWork& W, PeelShared& S) {
    Ctl* C = W.ctl;
    const int lane = lane_id();
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned long long t = gtimer(), slots = 0, scanned = 0;
    long long levels = 0, waves = 0;
    unsigned gen = 0;
    const int groups = (g.n + 31) / 32, nb = (int)W.blocks, b = (int)blockIdx.x;
    int32_t* mine = W.list + 32ll * ((long long)b * (groups / nb) + min(b, groups % nb));
    if (threadIdx.x == 0) {
        S.n[0] = S.n[1] = 0;
        S.keep = S.mx = S.peeled = S.shared_out = 0;
    }
    __syncthreads();
    // live vertices of degree > 0 start in their block's list; the others are done
    const int my_groups = groups / nb + (b < groups % nb ? 1 : 0);
    for (int j0 = 0; j0 < my_groups; j0 += kPeelWarps) {
        const int j = j0 + (int)(threadIdx.x >> 5);
        const long long v = 32ll * ((long long)j * nb + b) + lane;
        bool in = false;
        int mx = 0;
        if (j < my_groups && v < g.n && g.live((int)v)) {
            const int d = g.degree((int)v);
            W.dcur[v] = d;
            *g.core((int)v) = d > 0 ? kUnpeeled : 0;
            in = d > 0;
            mx = in ? 0x7FFFFFFF - d : 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&S.keep, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) mine[at + __popc(m & ((1u << lane) - 1))] = (int32_t)v;
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0 && mx) atomicMax(&S.mx, mx);
    }
    __syncthreads();
    int nl = S.keep;
    if (threadIdx.x == 0 && S.mx) atomicMax(&C->pm[0], (unsigned long long)S.mx);
    unsigned long long word = peel_barrier(W, S, gen, peel_word(nl, false, false));
    if (!word) return;
    bool left = (word >> 32) != 0;
    int k = left ? 0x7FFFFFFF - (int)vload64(&C->pm[gen & 3u]) : 0;
    int q = 0;
    unsigned long long far_lo = 0, chunk_lo = 0;
    while (left) {
        gen++;
        // scan the block's share: above k stays, the others leave now (or
        // left at an earlier level: their claim fails)
        if (threadIdx.x == 0) {
            S.keep = 0;
            S.mx = 0;
            S.peeled = 0;
            S.shared_out = 0;
        }
        __syncthreads();
        scanned += threadIdx.x == 0 ? (unsigned long long)nl : 0ull;
        for (int t0 = 0; t0 < nl; t0 += kPeelTile * kPeelThreads) {
            int v[kPeelTile], d[kPeelTile];
#pragma unroll
            for (int j = 0; j < kPeelTile; j++) {
                const int i = t0 + j * kPeelThreads + (int)threadIdx.x;
                v[j] = i < nl ? mine[i] : -1;
            }
#pragma unroll
            for (int j = 0; j < kPeelTile; j++) d[j] = v[j] >= 0 ? __ldcg(W.dcur + v[j]) : 0;
            __syncthreads();   // the tile is read: entries before its end may be overwritten
            int keep = 0, out = 0, mx = 0;
#pragma unroll
            for (int j = 0; j < kPeelTile; j++) {
                if (v[j] < 0) continue;
                if (d[j] > k) {
                    keep++;
                    mx = max(mx, 0x7FFFFFFF - d[j]);
                } else {
                    out++;
                }
            }
            int both = keep | (out << 16);   // at most 256 of each per warp
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, both, o);
                if (lane >= o) both += x;
            }
            for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const int tot = __shfl_sync(0xffffffffu, both, 31);
            int kb = 0, ob = 0;
            if (lane == 0) {
                if (tot & 0xFFFF) kb = atomicAdd(&S.keep, tot & 0xFFFF);
                if (tot >> 16) ob = atomicAdd(&S.n[q], tot >> 16);
                if (mx) atomicMax(&S.mx, mx);
            }
            kb = __shfl_sync(0xffffffffu, kb, 0) + (both & 0xFFFF) - keep;
            ob = __shfl_sync(0xffffffffu, ob, 0) + (both >> 16) - out;
#pragma unroll
            for (int j = 0; j < kPeelTile; j++) {
                if (v[j] < 0) continue;
                if (d[j] > k) {
                    mine[kb++] = v[j];
                } else {
                    if (ob < kPeelQueue) {
                        S.x[q][ob] = v[j];
                    } else if (atomicCAS(g.core(v[j]), kUnpeeled, k) == kUnpeeled) {
                        W.far[atomicAdd(&C->tail[0], 1ull)] = v[j];
                        S.shared_out = 1;
                        S.peeled = 1;
                    }
                    ob++;
                }
            }
            q = peel_drain(g, W, S, q, k, slots);
        }
        __syncthreads();
        nl = S.keep;
        if (threadIdx.x == 0 && S.mx) atomicMax(&C->pm[gen & 3u], (unsigned long long)S.mx);
        word = peel_barrier(W, S, gen, peel_word(nl, S.peeled != 0, S.shared_out != 0));
        if (!word) return;
        const unsigned long long kept = word >> 32;
        const bool peeled = ((word >> 10) & 2047ull) != 0;
        const int low = 0x7FFFFFFF - (int)vload64(&C->pm[gen & 3u]);
        if (lead) {
            const unsigned long long now = gtimer();
            C->ph[0] += now - t;
            t = now;
        }
        // what was shared: every block takes its part, until nothing new is
        while ((word >> 21) & 2047ull) {
            const unsigned long long far_hi = vload64(&C->tail[0]);
            const unsigned long long chunk_hi = min(vload64(&C->tail[1]), W.chunk_cap);
            const unsigned long long nf = far_hi - far_lo, items = nf + (chunk_hi - chunk_lo);
            gen++;
            // nobody may add to the shared lists before every block has read their ends
            if (!peel_barrier(W, S, gen, 1ull)) return;
            gen++;
            if (threadIdx.x == 0) S.shared_out = 0;
            __syncthreads();
            const unsigned long long span = (unsigned long long)kPeelThreads * nb;
            for (unsigned long long i0 = 0; i0 < items; i0 += span) {
                const unsigned long long i = i0 + (unsigned long long)threadIdx.x * nb + b;
                long long off = 0;
                int len = 0;
                if (i < nf) {
                    peel_take(g, W, S, W.far[far_lo + i], off, len);
                } else if (i < items) {
                    const unsigned long long task = W.chunks[chunk_lo + (i - nf)];
                    if (task != ~0ull) {
                        const int s0 = (int)(task & 0xFFFFFFFFull) * kSpreadChunk;
                        g.list((int)(task >> 32), off, len);
                        off += s0;
                        len = min(len - s0, kSpreadChunk);
                    }
                }
                peel_walk(g, W, S, q, k, 0, off, len, 0x7FFFFFFF, slots);
                q = peel_drain(g, W, S, q, k, slots);
            }
            far_lo = far_hi;
            chunk_lo = chunk_hi;
            word = peel_barrier(W, S, gen, peel_word(0, false, S.shared_out != 0));
            if (!word) return;
            waves++;
            if (lead) {
                const unsigned long long now = gtimer();
                C->ph[1] += now - t;
                t = now;
            }
        }
        levels += peeled ? 1 : 0;
        left = kept != 0;
        k = peeled ? k + 1 : low;
    }
    if (lead) {
        C->st[ST_LEVELS] = (unsigned long long)levels;
        C->st[ST_WAVES] = (unsigned long long)(levels + waves);
        C->st[ST_BARRIERS] = gen + 1;
    }
    for (int o = 16; o > 0; o >>= 1) slots += __shfl_xor_sync(0xffffffffu, slots, o);
    if (lane == 0 && slots) atomicAdd(&C->st[ST_VISSLOTS], slots);
    if (threadIdx.x == 0 && scanned) atomicAdd(&C->st[ST_VISITED], scanned);
}

}  // namespace cm
