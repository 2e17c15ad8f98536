// cm_search.cuh -- grid mode: the search of one iteration as a task queue
// (included by cm_iterate.cu only).
//
// In grid mode the search of an iteration (insert: positive search and
// evictions; delete: evictions) runs without level barriers.  Every vertex
// that enters the frontier or is evicted also becomes a task in a queue, and
// warps claim tasks until the queue is quiescent: every task pushed has
// finished.  The proof of the interleaved search does not depend on the
// order in which vertices are processed, so the waves of the single-block
// mode and this order reach the same cores.
//
// What bounds it: not bytes but dependent round trips.  A list step is a
// chain list words -> the neighbours' keys -> the candidates' per-iteration
// words -> their atomics -> the queue push, each about a microsecond away,
// so the time is trips x steps, and the layout below puts as many slots as
// registers allow behind each trip:
//
//   * a scan step is a window of 512 slots (16 per lane): four 16-byte list
//     loads per lane, then 16 key gathers, all in flight together.  The
//     slots that matter (candidates: core k, and for an insertion SD > k)
//     are few; they are compacted into a per-warp shared buffer, and their
//     words and atomics are then handled 128 at a time, every lane busy.
//   * tasks are taken 32 at a time, one per lane.  The lists of those with
//     at most 256 slots are walked together, quad by quad (a quad is four
//     slots, one 16-byte load), up to 128 quads a window: lane l of a
//     window's load takes quad l whoever owns it.  (With one warp per vertex
//     a vertex of 9 slots used three lanes of 32 and cost a queue hand-off.)
//   * a frontier vertex whose support stays at or below k is evicted by the
//     task that found it out, from the candidates it still holds.
//   * the scan of a longer list leaves a record behind (an arena in device
//     memory): the neighbours of core k and how many are above, a tenth to a
//     quarter of the list.  The vertex is then walked from its record: when it
//     is evicted later in the same search, and in the following iterations of
//     the launch for as long as its core stays k (an insertion only raises
//     cores, so the neighbours counted above stay above; edges and neighbours
//     that join the level are appended, see rec_link).
//
// Measured search time (GB300, one warp per vertex and 128-slot steps -> this
// layout): Erdos-Renyi, 2*10^6 vertices of degree 8, 10^4 uniform inserts 6.5
// -> 1.5 ms; 64 Barabasi-Albert graphs (57 iterations) 27 -> 11 ms; R-MAT
// scale 24, 10^3 degree-proportional inserts (4*10^5 vertices visited,
// 3.8*10^8 slots) 7.5 -> 4.1 ms, of which the key gathers alone are 1.3 ms
// at the 300 G gathers/s (one lane per clock and SM) that a kernel doing
// nothing else reaches.
//
// A vertex with at least P.hub_len slots becomes a hub item instead, whose
// list is split into kChunk-slot chunk tasks that any warp may take:
//   HUB_FRONT / HUB_FRONT_SPEC / HUB_FRONT_REC: each chunk adds its share of
//     CSD to the item; the warp that finishes the last chunk adds the sum to the
//     support word at once (setting the processed flag, as a whole-list
//     scan would) and either queues an expansion item (support > k; the
//     SPEC and REC chunks have visited their candidates already) or evicts
//     the vertex;
//   HUB_EXPAND: each chunk visits its share of the core-k neighbours;
//   HUB_EVICT_INS / HUB_EVICT_DEL / HUB_EVICT_REC: each chunk evicts its
//     share (REC: of the record); the last one lowers the core
//     (delete) and counts the vertex.
// The support word tolerates the delay: decrements from evicted neighbours
// land before or after the CSD sum in any order, and a processed hub whose
// count later falls to k is evicted by the decrement that does it.
#pragma once
#include "cm_common.cuh"
#include "cm_launch.h"
#include "cm_vertex.cuh"

namespace cm {

constexpr int kGridWarps = 12;    // warps per grid-mode block
constexpr int kWindow = 512;      // slots of a scan step
// Lists up to this many slots are walked together (and not recorded).  64 /
// 128 / 256 / 512: the captured step of 64 Barabasi-Albert graphs 51 / 45 /
// 42 / 41 ms, R-MAT scale 20 with 10^4 edges 3.2 / 3.1 / 2.8 / 2.9 ms.
constexpr int kShort = 256;

// Per-warp scratch of the search (dynamic shared memory).
struct WarpBuf {
    int32_t id[kWindow];              // a window's candidates, and from the end its other core-k neighbours
    unsigned long long kept[32];      // tasks the warp keeps for itself
    unsigned long long rec_q[32];     // records made but not published
    int32_t rec_v[32];
    unsigned long long slab, slab_end;   // arena quads the warp holds (for the whole launch)
    uint32_t st[7];                   // statistics of the launch so far (N_*)
    int32_t csd[32];                  // CSD of the tasks walked together
    uint8_t own[kWindow];             // their candidates' tasks (lane numbers)
};
constexpr size_t kSearchSmem = sizeof(WarpBuf) * kGridWarps;
extern __shared__ __align__(16) unsigned char s_search[];

// Statistics kept per warp in shared memory: as registers they would be live
// across the whole search, which is short of registers (a spilled register
// is written through to L2: with the loop state and these spilled, local
// memory took three times the requests of the lists and keys).
enum { N_VIS = 0, N_VISL, N_EV, N_EVL, N_CH, N_CHL, N_SEL };
__device__ __forceinline__ void note(WarpBuf& B, int what, uint32_t n) {   // one lane of the warp
    B.st[what] += n;
}
__device__ __forceinline__ void flush_stats(WarpBuf& B, LocalStats& ls) {   // outside searches and fix-ups: selections
    const uint32_t t = __reduce_add_sync(0xffffffffu, ls.sel);
    if (lane_id() == 0) note(B, N_SEL, t);
    ls = LocalStats{};
    __syncwarp();
}

__device__ __forceinline__ int vload32i(const int* p) { return *(const volatile int*)p; }

// A vertex's record: the stamp of the iteration that wrote it (30 bits, as
// in the per-iteration word) and its first arena quad, in one 64-bit word,
// so a reader sees both or neither.  The first quad is the header {count,
// room, neighbours above k, k}; the ids follow, those that were candidates
// (SD > k) with the sign bit set.  A record is fresh if it was made in this
// launch (stamp >= e0, the launch's first iteration: the single-block mode
// does not keep records up to date), and stands for the list at level k if
// its k is that (-1: candidates only, for this iteration's evictions) and it
// did not overflow (count > room).
constexpr int32_t REC_CAND = (int32_t)0x80000000;
__device__ __forceinline__ unsigned long long rec_word(unsigned long long quad, uint32_t e) {
    return (quad << 30) | (unsigned long long)(e & 0x3FFFFFFFu);
}
__device__ __forceinline__ uint32_t rec_stamp(unsigned long long w) { return (uint32_t)(w & 0x3FFFFFFFull); }

// A neighbour at or above level k joins the list of vertex v at level k (a
// new edge, or a neighbour that has just risen to k): v's record counts it
// above, or appends it.  Runs between searches, when nobody reads records.
__device__ __forceinline__ void rec_link(const MaintainParams& P, uint32_t e0, int v, int k, int other,
                                         bool other_above) {
    const unsigned long long w = vload64(&P.rec[v & P.rec_mask]);
    if (rec_stamp(w) < e0) return;
    int32_t* r = P.arena + 4 * (w >> 30);
    const int room = vload32(&r[1]);
    if (vload32(&r[3]) != k) return;
    if (other_above) {
        atomicAdd(&r[2], 1);
        return;
    }
    const int at = atomicAdd(&r[0], 1);
    if (at < room) r[4 + at] = other;
}

// Room for the ids of a record of a vertex with superior degree sd and a
// list of len slots: its core-k neighbours number at most sd, and the rest is
// for those that join.
__device__ __forceinline__ int rec_room(int sd, int len) { return min(sd, len) + (sd >> 3) + 16; }

// What a warp carries through a search besides its buffer.
struct Walker {
    int nk;        // kept tasks
    int klim;      // most it may keep: 1 while warps wait for tasks, 32 while the queue is long
    bool more;     // iterations follow: records take the whole level, not the candidates alone
    int nrec;      // records made but not published
};

// Arena room for n quads behind what the warp holds: the first quad, or
// NO_QUAD.  A warp takes room in slabs, so few records touch the shared
// counter; the caller moves B.slab past what it uses.  Warp-uniform.
constexpr unsigned long long NO_QUAD = ~0ull;
__device__ __forceinline__ unsigned long long arena_reserve(Ctl* C, const MaintainParams& P, WarpBuf& B, unsigned n) {
    unsigned long long at = B.slab;
    if (B.slab_end - at >= n) return at;
    const unsigned long long q = n > P.slab_quads ? n : P.slab_quads;
    if (lane_id() == 0) at = atomicAdd(&C->rec_top, q);
    at = __shfl_sync(0xffffffffu, at, 0);
    if (at + q > P.arena_quads) return NO_QUAD;
    if (lane_id() == 0) {
        B.slab = at;
        B.slab_end = at + q;
    }
    __syncwarp();
    return at;
}

// ---------------------------------------------------------------- pushes
// Appends the vertices of the lanes' bit masks (bit j: id[j]) to the logs
// and the task queue: `fm` enter the frontier (insert), `em` are evicted (an
// insertion needs no log of its evictions).  One atomic per counter for the
// warp, issued by several lanes at once.  The
// first few stay with the warp (W.klim): it runs them next, which saves the
// hand-off through the queue.  A kept task is not counted in the queue's
// tail and not reported done; the task that produced it is reported only
// when the warp has run out of kept tasks, so quiescence still waits for it.
// Evictions are kept first: they prune the search.  Warp-collective.
template <bool DEL, int J>
__device__ __forceinline__ void push_new(Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W, unsigned fm,
                                         unsigned em, const int (&id)[J]) {
    if (!__any_sync(0xffffffffu, (fm | em) != 0)) return;
    const int lane = lane_id();
    const unsigned mine = (unsigned)__popc(fm) | ((unsigned)__popc(em) << 16);
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned tot = __shfl_sync(0xffffffffu, incl, 31);
    const int nf = (int)(tot & 0xFFFFu), ne = (int)(tot >> 16);
    const int kq = min(W.klim - W.nk > 0 ? W.klim - W.nk : 0, nf + ne);
    const unsigned long long nq = (unsigned long long)(nf + ne - kq);
    unsigned long long base = 0;
    if (lane < 3) {
        unsigned long long* p = lane == 0 ? &C->tail[0] : lane == 1 ? &C->tail[1] : &C->task_tail;
        const unsigned long long n = lane == 0 ? (unsigned long long)nf
                                     : lane == 1 ? (unsigned long long)(DEL ? ne : 0) : nq;
        if (n) base = atomicAdd(p, n);
    }
    const unsigned long long fb = __shfl_sync(0xffffffffu, base, 0);
    const unsigned long long eb = __shfl_sync(0xffffffffu, base, 1);
    const unsigned long long tb = __shfl_sync(0xffffffffu, base, 2);
    const bool room = nq == 0 || task_room(C, P, tb, nq);
    const unsigned excl = incl - mine;
    int fr = (int)(excl & 0xFFFFu), er = (int)(excl >> 16);
#pragma unroll
    for (int j = 0; j < J; j++) {
        const bool f = (fm >> j) & 1u, x = (em >> j) & 1u;
        if (!f && !x) continue;
        const int rank = x ? er : ne + fr;
        if (!x) P.VQ[(fb + fr++) & P.qmask] = id[j];
        else if (DEL) P.EQ[(eb + er++) & P.qmask] = id[j];
        else er++;
        const unsigned long long task = mk_task(x ? T_EVICT : T_FRONT, (unsigned long long)(uint32_t)id[j]);
        if (rank < kq) B.kept[W.nk + rank] = task;
        else if (room) vstore64(&P.TQ[(tb + (unsigned)(rank - kq)) & P.tqmask], task);
    }
    W.nk += kq;
    __syncwarp();
}

// ---------------------------------------------------------------- scan of one list
// Slots [s, min(s + 128 U, len)) of a list (from_rec: of a record's ids).
// The candidates go to the front of the buffer; returns their number.
//   S_INSERT: the core-k neighbours with SD > k; `part` gains this lane's
//             share of CSD (Definition 8: those and the neighbours above k),
//             and with `others` the remaining core-k neighbours go to the end
//             of the buffer, the last one first (their number: ne);
//   S_DELETE: the core-k neighbours;
//   S_ROSE, S_DROPPED: the neighbours of core k, whose SD counts a vertex
//             differently now that it has risen to k or dropped to k - 1;
//             `part` gains the share of that vertex's own SD.
// Lists start 16-byte aligned and their capacity is a multiple of 4; they
// are read evict-first so that L2 keeps the keys.  Warp-collective.
enum { S_INSERT = 0, S_DELETE = 1, S_ROSE = 2, S_DROPPED = 3 };
template <int KIND, int U = 4>
__device__ __forceinline__ int scan_window(const DevGraph& g, const int32_t* list, bool from_rec, int s, int len,
                                           int k, bool others, WarpBuf& B, int& part, int& ne) {
    const int lane = lane_id();
    int id[4 * U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int t = s + u * 128 + lane * 4;
        int4 a = make_int4(HOLE, HOLE, HOLE, HOLE);
        if (t < len) a = __ldcs(reinterpret_cast<const int4*>(list + t));
        if (KIND == S_INSERT && from_rec) {
            a.x &= ~REC_CAND;
            a.y &= ~REC_CAND;
            a.z &= ~REC_CAND;
            a.w &= ~REC_CAND;
        }
        id[4 * u] = t < len ? a.x : HOLE;
        id[4 * u + 1] = t + 1 < len ? a.y : HOLE;
        id[4 * u + 2] = t + 2 < len ? a.z : HOLE;
        id[4 * u + 3] = t + 3 < len ? a.w : HOLE;
    }
    uint32_t key[4 * U];
#pragma unroll
    for (int i = 0; i < 4 * U; i++) key[i] = id[i] >= 0 ? g.kc[id[i]] : KEY_DEAD;
    unsigned mask = 0, eq = 0;
#pragma unroll
    for (int i = 0; i < 4 * U; i++) {
        if (KIND == S_INSERT) {   // key order is (core, bit): above k or a candidate <=> key >= 2k + 1
            part += (int)key[i] >= 2 * k + 1;
            mask |= key[i] == (uint32_t)(2 * k + 1) ? 1u << i : 0u;
            eq |= key[i] == (uint32_t)(2 * k) ? 1u << i : 0u;
        } else {
            if (KIND != S_DELETE) part += key_core(key[i]) >= (KIND == S_ROSE ? k : k - 1);
            mask |= key_core(key[i]) == k ? 1u << i : 0u;
        }
    }
    if (KIND != S_INSERT || !others) eq = 0;
    ne = 0;
    if (!__any_sync(0xffffffffu, (mask | eq) != 0)) return 0;
    const int cnt = __popc(mask) | (__popc(eq) << 16);   // at most 512 of both together
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const int tot = __shfl_sync(0xffffffffu, incl, 31);
    int at = (incl - cnt) & 0xFFFF, end = kWindow - 1 - ((incl - cnt) >> 16);
#pragma unroll
    for (int i = 0; i < 4 * U; i++) {
        if ((mask >> i) & 1u) B.id[at++] = id[i];
        if (KIND == S_INSERT && ((eq >> i) & 1u)) B.id[end--] = id[i];
    }
    ne = tot >> 16;
    __syncwarp();
    return tot & 0xFFFF;
}

// ---------------------------------------------------------------- short lists together
// Quads [gbase, gend) (at most 128) of the lanes' lists laid end to end: a
// lane's list is at g.adj + off, has len slots and level k; nq is its number
// of quads and incl the running sum of those over the lanes.  The candidates
// go to the front of the buffer, with their owner's lane beside them, and
// the owners' shares (`part` of scan_window, by KIND) to B.csd.  Returns the
// number of candidates.  Warp-collective.
template <int KIND>
__device__ __forceinline__ int walk_short(const DevGraph& g, WarpBuf& B, long long off, int len, int k, int nq,
                                          int incl, int gbase, int gend) {
    const int lane = lane_id();
    int id[16];
    uint32_t key[16];
    unsigned owners = 0;
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const int q = gbase + u * 32 + lane;
        int o = 0;   // the owner: the first lane whose running quad count exceeds q
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= q) o += step;
        const long long ob = __shfl_sync(0xffffffffu, off, o);
        const int ol = __shfl_sync(0xffffffffu, len, o);
        const int t0 = (q - __shfl_sync(0xffffffffu, incl - nq, o)) * 4;
        owners |= (unsigned)o << (8 * u);
        int4 a = make_int4(HOLE, HOLE, HOLE, HOLE);
        if (q < gend) a = __ldcs(reinterpret_cast<const int4*>(g.adj + ob + t0));
        id[4 * u] = a.x;
        id[4 * u + 1] = t0 + 1 < ol ? a.y : HOLE;
        id[4 * u + 2] = t0 + 2 < ol ? a.z : HOLE;
        id[4 * u + 3] = t0 + 3 < ol ? a.w : HOLE;
    }
#pragma unroll
    for (int i = 0; i < 16; i++) key[i] = id[i] >= 0 ? g.kc[id[i]] : KEY_DEAD;
    unsigned mask = 0;
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const int o = (int)((owners >> (8 * u)) & 31u);
        const int kk = __shfl_sync(0xffffffffu, k, o);
        int part = 0;
#pragma unroll
        for (int i = 4 * u; i < 4 * u + 4; i++) {
            if (KIND == S_INSERT) {
                part += (int)key[i] >= 2 * kk + 1;
                mask |= key[i] == (uint32_t)(2 * kk + 1) ? 1u << i : 0u;
            } else {
                if (KIND != S_DELETE) part += key_core(key[i]) >= (KIND == S_ROSE ? kk : kk - 1);
                mask |= key_core(key[i]) == kk ? 1u << i : 0u;
            }
        }
        if (KIND != S_DELETE && part) atomicAdd(&B.csd[o], part);
    }
    const int cnt = __popc(mask);
    int cinc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, cinc, o);
        if (lane >= o) cinc += x;
    }
    const int nc = __shfl_sync(0xffffffffu, cinc, 31);
    int at = cinc - cnt;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        if ((mask >> i) & 1u) {
            B.id[at] = id[i];
            B.own[at++] = (uint8_t)((owners >> (8 * (i >> 2))) & 31u);
        }
    }
    __syncwarp();
    return nc;
}

// ---------------------------------------------------------------- candidates
// Candidates id[] (-1: none) of an insertion search, at levels kk[], with
// their per-iteration words as read: the ones with their bit of `vis` are
// visited (those not visited yet enter the frontier), the others lose one
// support (a processed one that falls to its level is evicted).
template <int J>
__device__ __forceinline__ void insert_words(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                             const int (&id)[J], const int (&kk)[J], const unsigned long long (&s)[J],
                                             unsigned vis, uint32_t e) {
    const unsigned long long dec = 0xFFFFFFFF00000000ull;   // one off the count
    unsigned long long r[J];
    unsigned go = 0, cur = 0;
#pragma unroll
    for (int j = 0; j < J; j++) {
        r[j] = 0;
        if (id[j] < 0) continue;
        const bool same = same_iter(wz(s[j]), e), v = (vis >> j) & 1u;
        if (same && (v ? (wz(s[j]) & kVisited) != 0 : (wz(s[j]) & kProcessed) && ww(s[j]) <= kk[j])) continue;
        go |= 1u << j;
        unsigned long long* p = iter_word(g, id[j]);
        if (!same) {
            r[j] = atomicCAS(p, s[j], (v ? (unsigned long long)kVisited : dec) | (unsigned long long)(e << 2));
        } else {
            cur |= 1u << j;
            r[j] = v ? atomicOr(p, (unsigned long long)kVisited) : atomicAdd(p, dec);
        }
    }
    unsigned fm = 0, em = 0;
#pragma unroll
    for (int j = 0; j < J; j++) {
        if (!((go >> j) & 1u)) continue;
        const bool v = (vis >> j) & 1u;
        if (!((cur >> j) & 1u)) {
            if (r[j] == s[j]) {           // first to touch it in this iteration
                fm |= v ? 1u << j : 0u;
                continue;
            }
            make_current(g, C, id[j], e, r[j]);
            r[j] = v ? atomicOr(iter_word(g, id[j]), (unsigned long long)kVisited)
                     : atomicAdd(iter_word(g, id[j]), dec);
        }
        if (v) fm |= (wz(r[j]) & kVisited) == 0 ? 1u << j : 0u;
        else em |= (wz(r[j]) & kProcessed) && ww(r[j]) == kk[j] + 1 ? 1u << j : 0u;
    }
    push_new<false, J>(C, P, B, W, fm, em, id);
}

// The nc buffered candidates of an insertion search, 32 J at a time: of a
// vertex whose support exceeds its level, visit (those not visited yet enter
// the frontier, Algorithm 3); of an evicted one, take one from the support,
// and a processed candidate whose support falls to k leaves too (Algorithm
// 4).  MANY: candidate i belongs to the task of lane B.own[i], with that
// lane's level k and bit of the mask that decide() returns (set: visit);
// otherwise all belong to one task, with level k and bit 0.  decide() runs
// once, after the first words are requested, so the support atomics that it
// waits for overlap them.  Warp-collective.
template <bool MANY, int J = 4, class Decide>
__device__ __forceinline__ void act_insert(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                           int nc, int k, uint32_t e, Decide decide) {
    const int lane = lane_id();
    unsigned vmask = 0;
    for (int b0 = 0; b0 == 0 || b0 < nc; b0 += 32 * J) {
        int id[J], kk[J], ow[J];
        unsigned long long s[J];
        unsigned vis = 0;
#pragma unroll
        for (int j = 0; j < J; j++) {
            const int i = b0 + j * 32 + lane;
            id[j] = i < nc ? B.id[i] : -1;
            ow[j] = MANY && i < nc ? B.own[i] : 0;
            kk[j] = MANY ? __shfl_sync(0xffffffffu, k, ow[j]) : k;
            s[j] = id[j] >= 0 ? __ldcg(iter_word(g, id[j])) : 0ull;
        }
        if (b0 == 0) vmask = decide();
#pragma unroll
        for (int j = 0; j < J; j++) vis |= ((vmask >> ow[j]) & 1u) << j;
        insert_words<J>(g, C, P, B, W, id, kk, s, vis, e);
    }
}

// The recorded ids [i0, i1) of an evicted vertex at level k.  Its expansion
// in this iteration has visited the candidates among them (run_batch sees to
// that), so their words carry the iteration's stamp and a plain add does.  all: the record is of an
// earlier iteration and its marks are out of date (ids have risen above k,
// SDs have grown), so the keys tell who is a candidate now.  Warp-collective.
__device__ __forceinline__ void act_recorded(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                             const int32_t* list, int i0, int i1, int k, bool all) {
    const int lane = lane_id();
    for (int b0 = i0; b0 < i1; b0 += 128) {
        int id[4];
        unsigned go = 0, em = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int i = b0 + j * 32 + lane;
            const int x = i < i1 ? __ldcg(list + i) : 0;
            id[j] = x & ~REC_CAND;
            go |= i < i1 && (all || x < 0) ? 1u << j : 0u;
        }
        if (all) {
            uint32_t key[4];
#pragma unroll
            for (int j = 0; j < 4; j++) key[j] = (go >> j) & 1u ? g.kc[id[j]] : KEY_DEAD;
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (key[j] != (uint32_t)(2 * k + 1)) go &= ~(1u << j);
        }
        unsigned long long r[4];
#pragma unroll
        for (int j = 0; j < 4; j++)
            r[j] = (go >> j) & 1u ? atomicAdd(iter_word(g, id[j]), 0xFFFFFFFF00000000ull) : 0ull;
#pragma unroll
        for (int j = 0; j < 4; j++)
            em |= ((go >> j) & 1u) && (wz(r[j]) & kProcessed) && ww(r[j]) == k + 1 ? 1u << j : 0u;
        push_new<false, 4>(C, P, B, W, 0u, em, id);
    }
}

// Core-k neighbours id[] (-1: none) of vertices evicted by a deletion, with
// their words, thresholds SD - k + 1 and change stamps as read; low[]: the low
// half of a current word counted at their level.  One that has left meanwhile
// and passes for level k (level_bits) may be counted once more, which does no
// harm, but not evicted again.
template <int J>
__device__ __forceinline__ void delete_words(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                             const int (&id)[J], const int (&thr)[J], const uint32_t (&low)[J],
                                             const unsigned long long (&s)[J], const uint32_t (&ch)[J], uint32_t e) {
    const unsigned long long inc = 1ull << 32;
    unsigned long long r[J];
    unsigned go = 0;
#pragma unroll
    for (int j = 0; j < J; j++) {
        r[j] = 0;
        const bool same = same_iter(wz(s[j]), e);
        if (id[j] < 0 || ch[j] == e || thr[j] <= 0 || (same && ww(s[j]) >= thr[j])) continue;
        go |= 1u << j;
        r[j] = same ? atomicAdd(iter_word(g, id[j]), inc) : atomicCAS(iter_word(g, id[j]), s[j], inc | low[j]);
    }
    unsigned em = 0;
#pragma unroll
    for (int j = 0; j < J; j++) {
        if (!((go >> j) & 1u)) continue;
        if (!same_iter(wz(s[j]), e)) {
            if (r[j] == s[j]) {   // first to touch it in this iteration
                r[j] = low[j];
            } else {              // someone did it first: restamp if needed, then add
                make_current(g, C, id[j], e, r[j], low[j] & 3u);
                r[j] = atomicAdd(iter_word(g, id[j]), inc);
            }
        }
        if (wz(r[j]) == low[j] && ww(r[j]) + 1 == thr[j]) {
            g.chg[id[j]] = e;
            em |= 1u << j;
        }
    }
    push_new<true, J>(C, P, B, W, 0u, em, id);
}

// The nc buffered candidates (core-k neighbours) of vertices evicted by a
// deletion: each loses one support, initially its SD, and leaves when its
// count of evicted neighbours reaches SD - k + 1 (Algorithm 7).  Evicted
// vertices (chg == e) are skipped: their cores already dropped, so one that
// fell from k + 1 would pass for level k (one that is missed: see level_bits).
template <bool MANY, int J = 4>
__device__ __forceinline__ void act_delete(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                           int nc, int k, uint32_t e) {
    const int lane = lane_id();
    for (int b0 = 0; b0 < nc; b0 += 32 * J) {
        int id[J], thr[J];
        unsigned long long s[J];
        uint32_t ch[J], low[J];
#pragma unroll
        for (int j = 0; j < J; j++) {
            const int i = b0 + j * 32 + lane;
            id[j] = i < nc ? B.id[i] : -1;
            const int o = MANY && i < nc ? B.own[i] : 0;
            const int kk = MANY ? __shfl_sync(0xffffffffu, k, o) : k;
            s[j] = id[j] >= 0 ? __ldcg(iter_word(g, id[j])) : 0ull;
            ch[j] = id[j] >= 0 ? __ldcg(g.chg + id[j]) : e;
            thr[j] = id[j] >= 0 ? g.hc[id[j]].y - kk + 1 : 0;
            low[j] = e << 2 | level_bits(kk);
        }
        delete_words<J>(g, C, P, B, W, id, thr, low, s, ch, e);
    }
}

// ---------------------------------------------------------------- hub items
// Creates a hub item and its chunk tasks (warp-collective); false if the
// item ring is full (the caller then walks the list itself).  acc0: what its
// sum starts from; room > 0: the item also reserves arena room for a record
// of that many ids.
__device__ __forceinline__ bool make_hub(Ctl* C, const MaintainParams& P, int v, int kind, int k, long long off,
                                         int len, int acc0, int room) {
    const int lane = lane_id();
    const int nch = (len + kChunk - 1) / kChunk;
    unsigned long long idx = 0, tb = 0;
    int ok = 0;
    if (lane == 0) {
        if (vload64(&C->hub_created) - vload64(&C->hub_finished) < kHubRingSafe) {
            idx = atomicAdd(&C->hub_created, 1ull);
            unsigned long long rb = 0;
            int rcap = 0;
            if (room > 0) {
                const unsigned long long q = 1ull + (unsigned long long)((room + 3) >> 2);
                rb = atomicAdd(&C->rec_top, q);
                if (rb + q <= P.arena_quads) rcap = room;
            }
            HubItem* it = &P.HQ[idx & (kHubRing - 1)];
            it->off = off;
            it->v = v;
            it->kind = kind;
            it->k = k;
            it->len = len;
            it->nch = nch;
            it->acc = acc0;
            it->done = 0u;
            it->rcur = 0;
            it->ncand = 0;
            it->rquad = rb;
            it->rcap = rcap;
            __threadfence();   // the item before its tasks
            tb = atomicAdd(&C->task_tail, (unsigned long long)nch);
            ok = 1;
        }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) return false;
    idx = __shfl_sync(0xffffffffu, idx, 0);
    tb = __shfl_sync(0xffffffffu, tb, 0);
    if (!task_room(C, P, tb, (unsigned long long)nch)) return true;   // error recorded; the search stops
    const unsigned long long base = ((idx & (kHubRing - 1)) << kTaskChunkBits);
    for (int j = lane; j < nch; j += 32)
        vstore64(&P.TQ[(tb + j) & P.tqmask], mk_task(T_CHUNK, base | (unsigned long long)j));
    return true;
}

// One vertex pushed by the warp (an evicted hub).
__device__ __forceinline__ void push_evicted(Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W, int v) {
    const int id[1] = {v};
    push_new<false, 1>(C, P, B, W, 0u, lane_id() == 0 ? 1u : 0u, id);
}

// Adds a frontier vertex's CSD to its support and sets its processed flag;
// returns the old word.  Whoever made it a frontier vertex stamped its word
// with this iteration, so a plain add does.
__device__ __forceinline__ unsigned long long add_csd(const DevGraph& g, int v, int csd) {
    return atomicAdd(iter_word(g, v), ((unsigned long long)(uint32_t)csd << 32) + (unsigned long long)kProcessed);
}

// ---------------------------------------------------------------- one list walked by a warp
// Slots [s0, s1) of a list (from_rec: of a record) of a vertex at level k,
// window by window: scan, copy what belongs into a record, act on the
// candidates.  The one place for all insertion walks of single lists (whole
// lists, records, chunks of hubs), so that its instructions stay cached.
enum { A_EVICT = 0, A_VISIT = 1, A_COUNT = 2 };
struct Walk {
    const int32_t* list;
    int s0, s1, k;
    bool from_rec;
    int act;
    int32_t* out;     // ids of the record being made (NULL: none)
    int room;         // ... and room for them; past it `nrec` counts on
    int* shared;      // ... a hub's: the ids so far, shared by its chunks
    // results
    int part, ncand, nrec;
};
__device__ __forceinline__ void walk_insert(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                            Walk& L, uint32_t e) {
    const int lane = lane_id();
    L.part = L.ncand = L.nrec = 0;
    for (int s = L.s0; s < L.s1; s += kWindow) {
        int ne = 0;
        const int nc = scan_window<S_INSERT>(g, L.list, L.from_rec, s, L.s1, L.k, L.out && W.more, B, L.part, ne);
        L.ncand += nc;
        if (L.out && nc + ne > 0) {
            int at = L.nrec;
            L.nrec += nc + ne;
            if (L.shared) {
                if (lane == 0) at = atomicAdd(L.shared, nc + ne);
                at = __shfl_sync(0xffffffffu, at, 0);
            }
            if (at + nc + ne <= L.room) {
                for (int i = lane; i < nc; i += 32) L.out[at + i] = B.id[i] | REC_CAND;
                for (int i = lane; i < ne; i += 32) L.out[at + nc + i] = B.id[kWindow - 1 - i];
            }
        }
        if (L.act != A_COUNT && nc > 0)
            act_insert<false>(g, C, P, B, W, nc, L.k, e, [&] { return (unsigned)L.act; });
        __syncwarp();   // the buffer is free again
    }
}

// Makes a record of the walk's ids at arena quad q (header; the ids are
// there), room for `room` of them.  One lane calls it.
__device__ __forceinline__ void rec_header(const MaintainParams& P, const Walker& W, unsigned long long q, int n,
                                           int room, int above, int k) {
    *reinterpret_cast<int4*>(P.arena + 4 * q) = make_int4(n, room, above, W.more ? k : -1);
}

// Publishes the records a warp has made (at most 32), with one
// fence for all of them.  A vertex that is evicted before its record is out
// has its list walked again.
__device__ __forceinline__ void publish_records(const MaintainParams& P, WarpBuf& B, Walker& W, uint32_t e) {
    if (W.nrec == 0) return;
    __syncwarp();
    __threadfence();
    if (lane_id() < W.nrec) vstore64(&P.rec[B.rec_v[lane_id()]], rec_word(B.rec_q[lane_id()], e));
    W.nrec = 0;
}

// A frontier vertex with more than kShort slots (Algorithm 3): support +=
// CSD; above k it visits its candidates, else it is evicted.  Nearly all of
// them survive, so the candidates are visited as they are found
// (expand_early); one that fails after all, or the paper's order, walks the
// list again.  A list is recorded; from_rec: `list` is the vertex's record,
// `above` the neighbours it counts above k.
__device__ __forceinline__ void long_front(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                           int v, int k, const int32_t* list, int len, bool from_rec, int above,
                                           int room, uint32_t e) {
    const int lane = lane_id();
    const bool early = expand_early(P);
    unsigned long long q = NO_QUAD;
    if (!from_rec) q = arena_reserve(C, P, B, 1u + (unsigned)((room + 3) >> 2));
    Walk L{list, 0, len, k, from_rec, early ? A_VISIT : A_COUNT, q != NO_QUAD ? P.arena + 4 * q + 4 : nullptr, room,
           nullptr, 0, 0, 0};
    for (;;) {
        walk_insert(g, C, P, B, W, L, e);
        if (L.act == A_EVICT || (L.act == A_VISIT && !early)) break;   // the second walk
        const int csd = warp_sum(L.part) + above;
        unsigned up = 0;
        if (lane == 0) {
            up = ww(add_csd(g, v, csd)) + csd > k ? 1u : 0u;
            note(B, N_VIS, 1);
            note(B, N_VISL, len);
            if (!up) note(B, N_EV, 1);
        }
        up = __shfl_sync(0xffffffffu, up, 0);
        if (L.out && L.nrec <= room) {
            const int keep = min(room, W.more ? L.nrec + (L.nrec >> 2) + 16 : L.nrec);
            if (lane == 0) {
                rec_header(P, W, q, L.nrec, keep, csd - L.ncand, k);
                B.slab = q + 1 + (unsigned)((keep + 3) >> 2);
            }
            __syncwarp();
            if (lane == 0) {
                B.rec_v[W.nrec] = v;
                B.rec_q[W.nrec] = q;
            }
            W.nrec++;
        }
        if (early && up) break;
        L.out = nullptr;
        L.act = up ? A_VISIT : A_EVICT;
    }
}

// One chunk task of a hub (warp-collective).
template <bool DEL>
__device__ __forceinline__ void run_chunk(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                          uint32_t e, unsigned long long payload) {
    const int lane = lane_id();
    HubItem* it = &P.HQ[payload >> kTaskChunkBits];
    const int ci = (int)(payload & ((1ull << kTaskChunkBits) - 1));
    // the item was written by another SM: read it from L2
    const int v = vload32i(&it->v), kind = vload32i(&it->kind), k = vload32i(&it->k);
    const int len = vload32i(&it->len), nch = vload32i(&it->nch), rcap = vload32i(&it->rcap);
    const long long off = (long long)vload64((const unsigned long long*)&it->off);
    const unsigned long long rquad = vload64(&it->rquad);
    const int s0 = ci * kChunk, s1 = min(s0 + kChunk, len);
    const bool front = kind == HUB_FRONT || kind == HUB_FRONT_SPEC || kind == HUB_FRONT_REC;
    int part = 0, ncand = 0;
    if constexpr (DEL) {
        int ne = 0;
        const int nc = scan_window<S_DELETE>(g, g.adj + off, false, s0, s1, k, false, B, part, ne);
        act_delete<false>(g, C, P, B, W, nc, k, e);
    } else if (kind == HUB_EVICT_REC) {
        act_recorded(g, C, P, B, W, P.arena + off, s0, s1, k, vload32i(&it->acc) != 0);
    } else {
        Walk L{(kind == HUB_FRONT_REC ? P.arena : g.adj) + off, s0, s1, k, kind == HUB_FRONT_REC,
               kind == HUB_FRONT ? A_COUNT : kind == HUB_EVICT_INS ? A_EVICT : A_VISIT,
               rcap > 0 ? P.arena + 4 * rquad + 4 : nullptr, rcap, &it->rcur, 0, 0, 0};
        walk_insert(g, C, P, B, W, L, e);
        ncand = L.ncand;
        part = warp_sum(L.part);
    }
    __syncwarp();
    int decide = 0;   // 1 expand, 2 evict
    if (lane == 0) {
        if (front) {
            atomicAdd(&it->acc, part);
            if (ncand) atomicAdd(&it->ncand, ncand);
        }
        __threadfence();
        if (atomicAdd(&it->done, 1u) == (uint32_t)(nch - 1)) {
            if (front) {
                __threadfence();
                const int acc = atomicAdd(&it->acc, 0);
                const int rcur = atomicAdd(&it->rcur, 0);
                if (rcap > 0 && rcur <= rcap) {   // the record before the flag that lets others evict v
                    rec_header(P, W, rquad, rcur, rcap, acc - atomicAdd(&it->ncand, 0), k);
                    __threadfence();
                    vstore64(&P.rec[v], rec_word(rquad, e));
                }
                decide = ww(add_csd(g, v, acc)) + acc > k ? 1 : 2;
                note(B, N_VIS, 1);
                note(B, N_VISL, len);
            } else if (kind != HUB_EXPAND) {
                if (DEL) {
                    g.hc[v].x = k - 1;
                    g.kc[v] = key_of(k - 1, 0);   // the SD fix-up of the next claim phase sets its bit
                }
                note(B, N_EV, 1);
                note(B, N_EVL, len);
            }
            atomicAdd(&C->hub_finished, 1ull);
        }
    }
    if constexpr (!DEL) {
        decide = __shfl_sync(0xffffffffu, decide, 0);
        if (decide == 1 && kind == HUB_FRONT && !make_hub(C, P, v, HUB_EXPAND, k, off, len, 0, 0)) {
            Walk L{g.adj + off, 0, len, k, false, A_VISIT, nullptr, 0, nullptr, 0, 0, 0};
            walk_insert(g, C, P, B, W, L, e);
        }
        if (decide == 2) push_evicted(C, P, B, W, v);
    }
}

// A vertex with more than kShort slots evicted by a deletion (Algorithm 7):
// it drops to k - 1.
__device__ __forceinline__ void long_evict_delete(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B,
                                                  Walker& W, int v, int k, const int32_t* list, int len,
                                                  uint32_t e) {
    int part = 0, ne = 0;
    for (int s = 0; s < len; s += kWindow) {
        const int nc = scan_window<S_DELETE>(g, list, false, s, len, k, false, B, part, ne);
        act_delete<false>(g, C, P, B, W, nc, k, e);
        __syncwarp();
    }
    if (lane_id() == 0) {
        g.hc[v].x = k - 1;
        g.kc[v] = key_of(k - 1, 0);   // bit set by the SD fix-up
        note(B, N_EV, 1);
        note(B, N_EVL, len);
    }
}

// A task with at most 128 slots that is alone in its batch: one scan
// step, and one candidate per lane where they fit (the walk of many short
// lists takes about three times the instructions, which is what a lone task's
// latency consists of once its words are in L2).
template <bool DEL>
__device__ __forceinline__ void lone_short(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                           int v, int k, const int32_t* list, int len, bool front, uint32_t e) {
    const int lane = lane_id();
    int part = 0, ne = 0;
    const int nc = scan_window<DEL ? S_DELETE : S_INSERT, 1>(g, list, false, 0, len, k, false, B, part, ne);
    if constexpr (DEL) {
        if (nc <= 32) act_delete<false, 1>(g, C, P, B, W, nc, k, e);
        else act_delete<false, 4>(g, C, P, B, W, nc, k, e);
        if (lane == 0) {
            g.hc[v].x = k - 1;
            g.kc[v] = key_of(k - 1, 0);   // bit set by the SD fix-up
            note(B, N_EV, 1);
            note(B, N_EVL, len);
        }
    } else {
        unsigned long long old = 0;
        int csd = 0;
        if (front) {
            csd = warp_sum(part);
            if (lane == 0) {
                old = add_csd(g, v, csd);
                note(B, N_VIS, 1);
                note(B, N_VISL, len);
            }
        } else if (lane == 0) {
            note(B, N_EV, 1);
            note(B, N_EVL, len);
        }
        auto decide = [&] {
            if (!front) return 0u;
            const unsigned up = __shfl_sync(0xffffffffu, ww(old) + csd > k ? 1u : 0u, 0);
            if (!up && lane == 0) note(B, N_EV, 1);
            return up;
        };
        if (nc <= 32) act_insert<false, 1>(g, C, P, B, W, nc, k, e, decide);
        else act_insert<false, 4>(g, C, P, B, W, nc, k, e, decide);
    }
}

// The same for at most 32 slots, one per lane: everything that may be needed
// of a neighbour is read together with its key, which takes one round trip
// off the chain (and the buffer and its prefix sums with it): 1,000 edges on
// a 10^4-vertex graph, two inserts and two deletes, 1.13 -> 1.06 ms.
template <bool DEL>
__device__ __forceinline__ void lone_tiny(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                          int v, int k, const int32_t* list, int len, bool front, uint32_t e) {
    const int lane = lane_id();
    const int x = lane < len ? __ldcs(list + lane) : HOLE;
    uint32_t key = KEY_DEAD;
    unsigned long long s[1] = {0};
    if (x >= 0) {
        key = g.kc[x];
        s[0] = __ldcg(iter_word(g, x));
    }
    if constexpr (DEL) {
        const uint32_t ch[1] = {x >= 0 ? __ldcg(g.chg + x) : e};
        const int thr[1] = {x >= 0 ? g.hc[x].y - k + 1 : 0};
        const int id[1] = {key_core(key) == k ? x : -1};
        const uint32_t low[1] = {e << 2 | level_bits(k)};
        delete_words<1>(g, C, P, B, W, id, thr, low, s, ch, e);
        if (lane == 0) {
            g.hc[v].x = k - 1;
            g.kc[v] = key_of(k - 1, 0);   // bit set by the SD fix-up
            note(B, N_EV, 1);
            note(B, N_EVL, len);
        }
    } else {
        const int csd = __popc(__ballot_sync(0xffffffffu, (int)key >= 2 * k + 1));
        unsigned up = 0;
        if (front) {
            if (lane == 0) {
                up = ww(add_csd(g, v, csd)) + csd > k ? 1u : 0u;
                note(B, N_VIS, 1);
                note(B, N_VISL, len);
                if (!up) note(B, N_EV, 1);
            }
            up = __shfl_sync(0xffffffffu, up, 0);
        } else if (lane == 0) {
            note(B, N_EV, 1);
            note(B, N_EVL, len);
        }
        const int id[1] = {key == (uint32_t)(2 * k + 1) ? x : -1};
        const int kk[1] = {k};
        insert_words<1>(g, C, P, B, W, id, kk, s, up, e);
    }
}

// ---------------------------------------------------------------- a batch of tasks
// Runs the tasks of the lanes with t != TASK_EMPTY (warp-collective).
template <bool DEL>
__device__ __forceinline__ void run_batch(const DevGraph& g, Ctl* C, const MaintainParams& P, WarpBuf& B, Walker& W,
                                          uint32_t e, uint32_t e0, unsigned long long t) {
    const int lane = lane_id();
    const bool have = t != TASK_EMPTY;
    const int type = have ? (int)(t >> 62) : -1;
    for (unsigned m = __ballot_sync(0xffffffffu, type == T_CHUNK); m; m &= m - 1) {
        const unsigned long long payload = __shfl_sync(0xffffffffu, t, __ffs(m) - 1) & ((1ull << 62) - 1);
        run_chunk<DEL>(g, C, P, B, W, e, payload);
    }
    const bool vert = type == T_FRONT || type == T_EVICT;
    if (!__any_sync(0xffffffffu, vert)) return;
    const bool front = !DEL && type == T_FRONT;
    int v = 0, k = 0, sd = 0, len = 0;
    long long off = 0;
    unsigned long long rec = 0;
    if (vert) {   // independent loads, issued together
        v = (int)(uint32_t)t;
        const int2 c = g.hc[v];
        off = g.off[v];
        len = g.end[v];
        if (!DEL) rec = ld_acquire64(&P.rec[v & P.rec_mask]);
        k = c.x;
        sd = c.y;
    }
    int4 hdr = make_int4(0, 0, 0, -1);
    if (!DEL && vert && len > kShort && rec_stamp(rec) >= e0)
        hdr = __ldcg(reinterpret_cast<const int4*>(P.arena + 4 * (rec >> 30)));
    // Whose record will do.  For a frontier vertex: one at its level k.  For an
    // evicted one: one made in this very iteration, which is published after
    // the walk that visited its candidates, or an earlier one at its level if
    // the vertex expanded early: the processed flag, without which nobody
    // evicts it, came after its visits then.  In the paper's order the flag
    // comes first, so an eviction can overtake the visits and meet words that
    // are still of older iterations, which act_recorded must not: the list.
    const bool now = rec_stamp(rec) == e;
    const bool fits = front ? hdr.w == k : now || (hdr.w == k && expand_early(P));
    const unsigned use = __ballot_sync(0xffffffffu, hdr.x <= hdr.y && hdr.y > 0 && fits);
    // lists of more than kShort slots, one after another
    for (unsigned m = __ballot_sync(0xffffffffu, vert && len > kShort); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int xv = __shfl_sync(0xffffffffu, v, src), xk = __shfl_sync(0xffffffffu, k, src);
        const int xlen = __shfl_sync(0xffffffffu, len, src);
        const long long xoff = __shfl_sync(0xffffffffu, off, src);
        const bool xfront = __shfl_sync(0xffffffffu, (int)front, src) != 0;
        const bool hub = P.hub_len > 0 && xlen >= P.hub_len;
        if constexpr (DEL) {
            if (!hub || !make_hub(C, P, xv, HUB_EVICT_DEL, xk, xoff, xlen, 0, 0))
                long_evict_delete(g, C, P, B, W, xv, xk, g.adj + xoff, xlen, e);
        } else {
            const bool from_rec = ((use >> src) & 1u) != 0;
            const long long ro = (long long)(4 * (__shfl_sync(0xffffffffu, rec, src) >> 30) + 4);
            const int cnt = from_rec ? __shfl_sync(0xffffffffu, hdr.x, src) : xlen;
            const bool big = from_rec ? P.hub_len > 0 && cnt >= P.hub_len : hub;
            if (xfront) {
                const int above = from_rec ? __shfl_sync(0xffffffffu, hdr.z, src) : 0;
                const int room = rec_room(__shfl_sync(0xffffffffu, sd, src), xlen);
                const bool spec = expand_early(P);
                if (!big || !make_hub(C, P, xv, from_rec ? HUB_FRONT_REC : spec ? HUB_FRONT_SPEC : HUB_FRONT, xk,
                                      from_rec ? ro : xoff, cnt, above, spec && !from_rec ? room : 0))
                    long_front(g, C, P, B, W, xv, xk, from_rec ? P.arena + ro : g.adj + xoff, cnt, from_rec, above,
                               room, e);
            } else {
                const int all = __shfl_sync(0xffffffffu, now ? 0 : 1, src);
                if (!big || !make_hub(C, P, xv, from_rec ? HUB_EVICT_REC : HUB_EVICT_INS, xk, from_rec ? ro : xoff,
                                      cnt, all, 0)) {
                    if (from_rec) {
                        act_recorded(g, C, P, B, W, P.arena + ro, 0, cnt, xk, all != 0);
                    } else {
                        Walk L{g.adj + xoff, 0, xlen, xk, false, A_EVICT, nullptr, 0, nullptr, 0, 0, 0};
                        walk_insert(g, C, P, B, W, L, e);
                    }
                    if (lane == 0) {
                        note(B, N_EV, 1);
                        note(B, N_EVL, cnt);
                    }
                }
            }
        }
    }
    publish_records(P, B, W, e);
    // the others together, up to 128 quads (512 slots) a window
    unsigned rest = __ballot_sync(0xffffffffu, vert && len <= kShort);
    if (!rest) return;
    if ((rest & (rest - 1)) == 0 && __shfl_sync(0xffffffffu, len, __ffs(rest) - 1) <= 128) {
        // one: searches spend their thin phases here, so take the fewest steps
        const int src = __ffs(rest) - 1;
        const int xv = __shfl_sync(0xffffffffu, v, src), xk = __shfl_sync(0xffffffffu, k, src);
        const int xlen = __shfl_sync(0xffffffffu, len, src);
        const int32_t* list = g.adj + __shfl_sync(0xffffffffu, off, src);
        const bool xfront = __shfl_sync(0xffffffffu, (int)front, src) != 0;
        if (xlen <= 32) lone_tiny<DEL>(g, C, P, B, W, xv, xk, list, xlen, xfront, e);
        else lone_short<DEL>(g, C, P, B, W, xv, xk, list, xlen, xfront, e);
        return;
    }
    const int nq = vert && len <= kShort ? (len + 3) >> 2 : 0;
    int incl = nq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    int gbase = 0;
    while (rest) {
        const bool in = ((rest >> lane) & 1u) && incl - gbase <= 128;   // at least one: a list has <= 64 quads
        const unsigned gm = __ballot_sync(0xffffffffu, in);
        const int gend = __shfl_sync(0xffffffffu, incl, 31 - __clz(gm));
        B.csd[lane] = 0;
        __syncwarp();
        const int nc = walk_short<DEL ? S_DELETE : S_INSERT>(g, B, off, len, k, nq, incl, gbase, gend);
        if (DEL) {
            act_delete<true>(g, C, P, B, W, nc, k, e);
            if (in) {
                g.hc[v].x = k - 1;
                g.kc[v] = key_of(k - 1, 0);   // bit set by the SD fix-up
            }
            const uint32_t el = __reduce_add_sync(0xffffffffu, in ? (unsigned)len : 0u);
            if (lane == 0) {
                note(B, N_EV, (uint32_t)__popc(gm));
                note(B, N_EVL, el);
            }
        } else {
            int csd = 0;
            unsigned long long old = 0;
            if (in && front) {
                csd = B.csd[lane];
                old = add_csd(g, v, csd);
            }
            const unsigned fronts = __ballot_sync(0xffffffffu, in && front);
            const uint32_t fl = __reduce_add_sync(0xffffffffu, in && front ? (unsigned)len : 0u);
            const uint32_t el = __reduce_add_sync(0xffffffffu, in && !front ? (unsigned)len : 0u);
            if (lane == 0) {
                note(B, N_VIS, (uint32_t)__popc(fronts));
                note(B, N_VISL, fl);
                note(B, N_EV, (uint32_t)__popc(gm & ~fronts));
                note(B, N_EVL, el);
            }
            act_insert<true>(g, C, P, B, W, nc, k, e, [&] {
                const unsigned up = __ballot_sync(0xffffffffu, in && front && ww(old) + csd > k);
                if (lane == 0) note(B, N_EV, (uint32_t)__popc(fronts & ~up));
                return up;
            });
        }
        __syncwarp();
        rest &= ~gm;
        gbase = gend;
    }
}

// Search (iteration number) whose queue the block knows to be quiescent.
__shared__ volatile uint32_t s_quiet;
__shared__ unsigned long long s_search_t0;   // when the search began (its waits are bounded)

// Drains the task queue (every warp of the grid).  Returns false on error.
// A warp claims slots for its lanes with one atomic and polls them together;
// it runs whatever is ready as one batch.  How many it claims follows the
// queue's backlog when it last claimed: one slot when tasks are scarce (a
// slot past the tail is waited for), its share when they are plenty, at most
// 32 (P.claim_max raises the share it takes; guided self-scheduling, so that
// the last tasks of a search still spread over all warps).  Finished tasks
// are reported in batches, always before the warp waits on an empty slot (so
// a waiting warp never holds back the quiescence test).  Inlined into the
// kernel: as a separate function it took the graph and the parameters by
// reference, which put both in local memory.
template <bool DEL>
__device__ __forceinline__ bool async_search(const DevGraph& g, Ctl* C, const MaintainParams& P, uint32_t e,
                                             uint32_t e0, bool more) {
    const int lane = lane_id();
    WarpBuf& B = reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5];
    const unsigned long long share = (unsigned long long)(P.claim_max > 1 ? P.claim_max : 1);
    unsigned long long idx = 0;
    unsigned ndone = 0;
    unsigned held = 0;   // lanes that hold a claimed slot
    int claim = 1;
    unsigned int nap = 32;
    Walker W{0, 1, more, 0};
    // One warp of the grid tests quiescence (a test reads two counters that
    // every claim and push needs, so hundreds of testers slow those down);
    // one warp per block watches the word it sets and tells the others
    // through shared memory.
    const bool watcher = threadIdx.x < 32, poller = watcher && blockIdx.x == 0;
    for (unsigned int spins = 0;; spins++) {
        unsigned long long t = TASK_EMPTY, h = 0, tl = 0;
        bool look = false;   // the backlog was read in this round
        if (W.nk > 0) {      // the tasks this warp kept
            if (lane < W.nk) t = B.kept[lane];
            __syncwarp();
            W.nk = 0;
            if (W.klim > 1) {
                look = true;
                h = lane == 0 ? vload64(&C->task_head) : 0ull;
                tl = lane == 1 ? vload64(&C->task_tail) : 0ull;
            }
        } else {
            if (!held) {
                if (lane == 0) h = atomicAdd(&C->task_head, (unsigned long long)claim);
                else if (lane == 1) tl = vload64(&C->task_tail);
                look = true;
                held = claim == 32 ? 0xffffffffu : (1u << claim) - 1u;
                idx = __shfl_sync(0xffffffffu, h, 0) + (unsigned long long)lane;
            }
            unsigned long long* slot = &P.TQ[idx & P.tqmask];
            const bool mine = (held >> lane) & 1u;
            if (mine) t = ld_acquire64(slot);
            const unsigned got = __ballot_sync(0xffffffffu, t != TASK_EMPTY);
            if (!got) {
                int quit = 0;
                if (lane == 0) {
                    if (ndone) {   // report before waiting
                        __threadfence();
                        atomicAdd(&C->task_done, (unsigned long long)ndone);
                    }
                    if (poller) {
                        // quiescent: every task pushed has finished (done read first)
                        const unsigned long long d = ld_acquire64(&C->task_done);   // read before the tail
                        if (d == vload64(&C->task_tail)) vstore64(&C->quiet, e);
                    }
                    if (watcher && (vload64(&C->quiet) == e || vload32(&C->error))) s_quiet = e;
                    if (s_quiet == e) quit = 1;
                    if (!quit && (spins & 3u) == 0 && gtimer() - s_search_t0 > P.limit_ns) {
                        atomicCAS(&C->error, 0, E_BARRIER_TIMEOUT);
                        quit = 1;
                    }
                }
                ndone = 0;
                if (__shfl_sync(0xffffffffu, quit, 0)) break;
                __nanosleep(nap);
                if (nap < 512) nap <<= 1;
                claim = 1;
                W.klim = 1;
                continue;
            }
            nap = 32;
            if (t != TASK_EMPTY) vstore64(slot, TASK_EMPTY);   // free for the next search
            held &= ~got;
            ndone += (unsigned)__popc(got);
        }
        // Tasks are stored without a release, so a poll orders nothing but the
        // task.  A vertex task needs no more: what it reads of its vertex is
        // fixed since the last barrier, counts and flags are changed by atomics
        // whose results their callers had before they stored a task, a record's
        // word is published behind a fence and read with acquire, and keys and
        // change stamps may lag (see level_bits; an insertion changes neither
        // during its search).  A chunk task needs its hub item, which is
        // written before a fence that this one meets.
        __syncwarp();
        if (__any_sync(0xffffffffu, t != TASK_EMPTY && (int)(t >> 62) == T_CHUNK)) __threadfence();
        run_batch<DEL>(g, C, P, B, W, e, e0, t);
        __syncwarp();
        if (look) {
            h = __shfl_sync(0xffffffffu, h, 0);
            tl = __shfl_sync(0xffffffffu, tl, 1);
            const unsigned long long backlog = tl > h ? tl - h : 0ull;
            const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
            const unsigned long long c = backlog * share / (2 * nwarps);
            claim = c < 1 ? 1 : c > 32 ? 32 : (int)c;
            W.klim = backlog > 2 * nwarps ? 32 : 1;
        }
    }
    return vload32(&C->error) == 0;
}

// Queues tasks for log entries [lo, hi) that are already in the log (a
// search resumed from the single-block mode).  Every warp calls it.
__device__ __forceinline__ void seed_tasks(Ctl* C, const MaintainParams& P, const int32_t* log, unsigned long long lo,
                                           unsigned long long hi, int type) {
    const int lane = lane_id();
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (unsigned long long base = lo + (unsigned long long)gwarp * 32; base < hi;
         base += (unsigned long long)nwarps * 32) {
        const unsigned long long cnt = min(32ull, hi - base);
        unsigned long long tb = 0;
        if (lane == 0) tb = atomicAdd(&C->task_tail, cnt);
        tb = __shfl_sync(0xffffffffu, tb, 0);
        if (task_room(C, P, tb, cnt) && (unsigned long long)lane < cnt)
            vstore64(&P.TQ[(tb + lane) & P.tqmask],
                     mk_task(type, (unsigned long long)(uint32_t)log[(base + lane) & P.qmask]));
    }
}

// ---------------------------------------------------------------- SD fix-up
// Grid mode's fixup_vertex (cm_vertex.cuh), of the vertices whose core moved
// in iteration fe: their SD, and that of their unmoved neighbours that count
// them differently now (kk: the neighbours' core).  Like a search step it is
// a chain of trips (list, keys, change stamps, SD atomics), so what counts is
// slots in flight and an even share for every warp: long lists in chunks,
// short ones together.  Measured (GB300) against a warp per list and a block
// per list of 4096 slots and more: claim phases, where the fix-ups run, of
// R-MAT scale 24 with 10^6 degree-proportional edges 12.1 -> 8.6 ms (insert)
// and 10.2 -> 6.6 ms (delete); captured step of 64 Barabasi-Albert graphs
// 41.6 -> 38.7 ms.  Few moved vertices gain nothing (Erdos-Renyi 10^4
// vertices, 10^3 edges: 1.06 -> 1.08 ms for four calls).
//
// The nc buffered neighbours: of the moved vertex v, or (MANY) of that of
// lane B.own[i].  link: iterations follow, so a neighbour at a riser's new
// level takes it into its record.  Warp-collective.
template <int OP, bool MANY>
__device__ __forceinline__ void fixup_near(const DevGraph& g, const MaintainParams& P, WarpBuf& B, int nc, int v,
                                           int kk, uint32_t fe, uint32_t e0, bool link) {
    const int lane = lane_id();
    for (int b0 = 0; b0 < nc; b0 += 128) {
        int id[4], ow[4];
        uint32_t ch[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int i = b0 + j * 32 + lane;
            id[j] = i < nc ? B.id[i] : -1;
            ow[j] = MANY && i < nc ? B.own[i] : 0;
            ch[j] = i < nc ? __ldcg(g.chg + id[j]) : fe;
        }
        // all of this phase's changes to a neighbour go the same way, so
        // only the update that crosses its core moves its key bit
        int old[4];
#pragma unroll
        for (int j = 0; j < 4; j++)
            old[j] = ch[j] != fe ? atomicAdd(&g.hc[id[j]].y, OP == 0 ? 1 : -1) : -1;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int xk = MANY ? __shfl_sync(0xffffffffu, kk, ow[j]) : kk;
            const int xv = MANY && OP == 0 ? __shfl_sync(0xffffffffu, v, ow[j]) : v;
            if (ch[j] == fe) continue;
            if (OP == 0) {
                if (old[j] == xk) atomicOr(&g.kc[id[j]], 1u);
                if (link) rec_link(P, e0, id[j], xk, xv, false);
            } else if (old[j] == xk + 1) {
                atomicAnd(&g.kc[id[j]], ~1u);
            }
        }
    }
    __syncwarp();
}

// Lists of more than kShort slots are queued in chunks that any warps take
// (the task ring is empty between searches; an entry is chunk << 32 | v).
// The vertex's per-iteration word, which nobody needs before its next
// iteration, collects its chunks' shares (low half) and arrivals (high half).
// With a block per list of 4096 slots and more, 40% of the warps' time went
// to the blocks' barriers and to waiting for the block that drew the longest
// lists (R-MAT scale 24, 10^6 degree-proportional edges: 1.5*10^9 slots, two
// thirds of them in 77,000 lists).  Chunks of 1024, 2048 or 4096 slots differ
// by less than 1%.
__device__ __forceinline__ int fix_chunk(const MaintainParams& P) { return max(P.block_len & ~(kWindow - 1), kWindow); }
__device__ __forceinline__ void list_long(const DevGraph& g, Ctl* C, const MaintainParams& P, int v, int len) {
    if (len <= kShort) return;
    const int n = (len - 1) / fix_chunk(P) + 1;
    *iter_word(g, v) = 0;
    const unsigned long long at = atomicAdd(&C->pc[2], (unsigned long long)n);
    for (int i = 0; i < n; i++) P.TQ[(at + i) & P.tqmask] = (unsigned long long)i << 32 | (unsigned)v;
}

// The fix-up of the moved vertices log[lo, hi).  queued: their long lists are
// nlong queued chunks, which come first; then the vertices, several to a warp
// when there are more of them than warps, their short lists walked together.
// Otherwise a warp walks any list.  A warp's first item is dealt by its
// index, the rest are fetched (C->pc[2], zeroed at every barrier).  Every
// warp of the launch must call it.
template <int OP>
__device__ __forceinline__ void fixup_grid(const DevGraph& g, Ctl* C, const MaintainParams& P, const int32_t* log,
                                           unsigned long long lo, unsigned long long hi, bool queued,
                                           unsigned long long nlong, uint32_t fe, uint32_t e0, bool link) {
    WarpBuf& B = reinterpret_cast<WarpBuf*>(s_search)[threadIdx.x >> 5];
    const int lane = lane_id();
    constexpr int up = OP == 0 ? 0 : 1;   // from the moved vertex's core to the neighbours'
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    const unsigned long long cnt = hi - lo;
    unsigned many = 1;   // vertices an item
    unsigned long long all = nlong + cnt;
    if (queued && cnt > nw) {
        many = min(((unsigned)cnt - 1) / (unsigned)nw + 1, 32u);
        all = nlong + ((unsigned)cnt - 1) / many + 1;
    }
    unsigned long long j = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    while (j < all) {
        const bool chunk = j < nlong;
        if (chunk || many == 1) {
            int v, s0 = 0;
            if (chunk) {
                const unsigned long long t = __ldcg(&P.TQ[j & P.tqmask]);
                v = (int)(uint32_t)t;
                s0 = (int)(t >> 32) * fix_chunk(P);
            } else {
                v = __ldcg(log + ((lo + (j - nlong)) & P.qmask));
            }
            const int len = g.end[v], kn = g.hc[v].x;
            const int32_t* list = g.adj + g.off[v];
            if (chunk || !queued || len <= kShort) {
                const int s1 = chunk ? min(s0 + fix_chunk(P), len) : len;
                int sd = 0, ne = 0;
                for (int s = s0; s < s1; s += kWindow) {
                    const int nc = scan_window<OP == 0 ? S_ROSE : S_DROPPED>(g, list, false, s, s1, kn + up, false, B,
                                                                            sd, ne);
                    fixup_near<OP, false>(g, P, B, nc, v, kn + up, fe, e0, link);
                }
                sd = __reduce_add_sync(0xffffffffu, sd);
                if (lane == 0) {
                    bool last = true;
                    if (chunk) vstore64(&P.TQ[j & P.tqmask], TASK_EMPTY);
                    if (s1 - s0 < len) {
                        const unsigned long long o = atomicAdd(iter_word(g, v), 1ull << 32 | (unsigned)sd);
                        sd += (int)(uint32_t)o;
                        last = (int)(o >> 32) == (len - 1) / fix_chunk(P);
                        if (last) *iter_word(g, v) = 0;   // the stamp of no iteration
                    }
                    if (last) {
                        g.hc[v].y = sd;
                        g.kc[v] = key_of(kn, sd);
                        note(B, N_CH, 1);
                        note(B, N_CHL, len);
                    }
                }
            }
        } else {
            const unsigned long long i = (j - nlong) * many + lane;
            bool mine = lane < (int)many && i < cnt;
            int v = 0, kn = 0, len = 0;
            long long off = 0;
            if (mine) {
                v = __ldcg(log + ((lo + i) & P.qmask));
                kn = g.hc[v].x;
                off = g.off[v];
                len = g.end[v];
                mine = len <= kShort;   // the others are queued
            }
            const int nq = mine ? (len + 3) >> 2 : 0;
            int incl = nq;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            int gbase = 0;
            for (unsigned rest = __ballot_sync(0xffffffffu, mine); rest;) {
                const bool in = ((rest >> lane) & 1u) && incl - gbase <= 128;   // at least one: a list has <= 64 quads
                const unsigned gm = __ballot_sync(0xffffffffu, in);
                const int gend = __shfl_sync(0xffffffffu, incl, 31 - __clz(gm));
                B.csd[lane] = 0;
                __syncwarp();
                const int nc = walk_short<OP == 0 ? S_ROSE : S_DROPPED>(g, B, off, len, kn + up, nq, incl, gbase,
                                                                       gend);
                if (in) {
                    const int sd = B.csd[lane];
                    g.hc[v].y = sd;
                    g.kc[v] = key_of(kn, sd);
                }
                const uint32_t sl = __reduce_add_sync(0xffffffffu, in ? (unsigned)len : 0u);
                if (lane == 0) {
                    note(B, N_CH, (uint32_t)__popc(gm));
                    note(B, N_CHL, sl);
                }
                fixup_near<OP, true>(g, P, B, nc, v, kn + up, fe, e0, link);
                rest &= ~gm;
                gbase = gend;
            }
        }
        if (all <= nw) break;   // every item was dealt by index
        if (lane == 0) j = nw + atomicAdd(&C->pc[2], 1ull);
        j = __shfl_sync(0xffffffffu, j, 0);
    }
    __syncwarp();
}

}  // namespace cm
