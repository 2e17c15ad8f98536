// cm_store.cu -- device graph store: construction, full decomposition by
// bucket peeling, superior degrees, vertex insertion/deletion helpers and
// export.
#include <cstddef>

#include "cm_common.cuh"
#include "cm_launch.h"
#include "cm_peel.cuh"

namespace cm {


static inline unsigned grid_for(long long n, int t, long long cap = 1 << 20) {
    long long b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

// ------------------------------------------------------------------ construction
// Validate ids, drop self-loops and repeats (first index insertion wins), and
// place each kept edge: its turn at either end is its slot in that end's
// list.  The turns are taken here, by the degree counts themselves, while the
// edge's index bucket is at hand: counting degrees, then placing the edges by
// a second round of counters and writing the slots into the index then, read
// the edges three times and every bucket twice (R-MAT scale 20, 15.7M edges:
// 2.06 -> 1.21 ms for the construction without the peel and the SD pass).
// at[i] = the two slots ({-1, -1}: dropped); Ctl::nrem counts the kept.
__global__ void build_index_kernel(const int32_t* __restrict__ E, long long m, DevGraph g, int2* at, Ctl* c) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool kept = false;
    if (i < m) {
        const int32_t u = E[2 * i], v = E[2 * i + 1];
        int2 p = make_int2(-1, -1);
        if (u < 0 || v < 0 || u >= g.n || v >= g.n) {
            atomicMin(&c->bad_index, i);
            atomicCAS(&c->error, 0, E_INVALID);
        } else if (u != v) {
            bool existed = false;
            const long long b = idx_insert(g.idx, g.idx_mask, ekey(u, v), &existed);
            if (b < 0) {
                atomicCAS(&c->error, 0, E_INDEX_FULL);
            } else if (!existed) {
                kept = true;
                p.x = atomicAdd(&g.deg[u], 1);
                p.y = atomicAdd(&g.deg[v], 1);
                // one 8-byte store: slot of the higher id in the lower one's list, and the reverse
                *reinterpret_cast<int2*>(&g.idx[b].slo) = u < v ? p : make_int2(p.y, p.x);
            }
        }
        at[i] = p;
    }
    const int n = __syncthreads_count(kept);
    if (threadIdx.x == 0 && n) atomicAdd(&c->nrem, (unsigned long long)n);
}
static_assert(offsetof(Bucket, slo) % 8 == 0 && offsetof(Bucket, shi) == offsetof(Bucket, slo) + 4,
              "a bucket's slots are one aligned 8-byte word");

// Sum of capacities (into c->reloc_need) when sum_only, else assign each
// vertex of [v0, v1) a slot range, its degree's worth of it used, by a
// warp-level scan and one pool allocation per warp.
__global__ void offsets_kernel(DevGraph g, int32_t v0, int32_t v1, Ctl* c, int sum_only) {
    long long base = (long long)v0 + (((long long)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll);
    long long stride = (long long)gridDim.x * blockDim.x;
    int lane = lane_id();
    for (; base < v1; base += stride) {
        long long v = base + lane;
        int cp = 0, d = 0;
        if (v < v1) {
            d = g.deg[v];
            cp = cap_for(d, g.slack_pct, g.min_cap);
        }
        int incl = cp;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        int tot = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long wb = 0;
        if (lane == 31) wb = atomicAdd(sum_only ? &c->reloc_need : &c->adj_top, (unsigned long long)tot);
        wb = __shfl_sync(0xffffffffu, wb, 31);
        if (!sum_only && v < v1) {
            g.off[v] = (int64_t)(wb + incl - cp);
            g.cap[v] = cp;
            g.end[v] = d;
        }
    }
}

__global__ void scatter_kernel(const int32_t* __restrict__ E, const int2* __restrict__ at, long long m, DevGraph g) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int2 p = at[i];
    if (p.x < 0) return;
    const int32_t u = E[2 * i], v = E[2 * i + 1];
    g.adj[g.off[u] + p.x] = v;
    g.adj[g.off[v] + p.y] = u;
}

// Given cores (a checkpoint): core -1 marks a deleted vertex, which gets the
// dead key; a live vertex's key bit is set by the SD pass that follows.
__global__ void set_cores_kernel(const int32_t* __restrict__ cores, DevGraph g) {
    long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= g.n) return;
    const int c = cores[v];
    g.hc[v].x = c;
    g.kc[v] = c < 0 ? KEY_DEAD : key_of(c, 0);
}

// SD(v), Definition 7: neighbours with core >= core(v).  The cores are read
// from a compact copy (4 bytes per vertex) instead of the 8-byte {core, SD}
// words.  A warp takes 32 vertices and walks their lists together, quad by
// quad (four slots, one 16-byte list load), 16 core gathers per lane in
// flight, whatever the lists' lengths: bound by the gathers (300 G/s at most).
// Lists of kSdHub slots or more go to a second kernel, a block each.  (One
// warp per vertex, four gathers per lane: R-MAT scale 20 0.42 ms, now 0.16;
// the re-peel of scale 24 with this pass 18.8 -> 17.6 ms.)
constexpr int kSdHub = 2048;
__global__ void copy_cores_kernel(DevGraph g, int32_t* core) {
    long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= g.n) return;
    core[v] = g.hc[v].x;
}

// This lane's count of the slots of `list` quad q (of a list of len slots)
// whose core is at least k.
__device__ __forceinline__ int sd_quad(const int32_t* __restrict__ core, const int4& a, int t0, int len, int k) {
    const int x[4] = {a.x, t0 + 1 < len ? a.y : HOLE, t0 + 2 < len ? a.z : HOLE, t0 + 3 < len ? a.w : HOLE};
    int n = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) n += x[q] >= 0 && core[x[q]] >= k;
    return n;
}

__global__ void __launch_bounds__(256) init_mcd_kernel(DevGraph g, int32_t v0, int32_t v1,
                                                       const int32_t* __restrict__ core, int32_t* hubs, Ctl* c) {
    __shared__ int s_sd[8][32];
    int* sum = s_sd[threadIdx.x >> 5];
    const int lane = lane_id();
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v0 + 32 * w < v1; w += nw) {
        const long long v = v0 + 32 * w + lane;
        int k = -1, len = 0;
        long long off = 0;
        if (v < v1) {
            k = core[v];
            off = g.off[v];
            len = k >= 0 ? g.end[v] : 0;
        }
        const bool hub = len >= kSdHub;
        if (hub) hubs[atomicAdd(&c->gather_n, 1ull)] = (int32_t)v;
        const int nq = hub ? 0 : (len + 3) >> 2;
        int incl = nq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        sum[lane] = 0;
        __syncwarp();
        for (int w0 = 0; w0 < total; w0 += 128) {
            int4 a[4];
            int own[4], t0[4], ol[4], ok[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int q = w0 + u * 32 + lane;
                int o = 0;   // the owner: the first lane whose running count exceeds q
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= q) o += step;
                own[u] = o;
                t0[u] = (q - __shfl_sync(0xffffffffu, incl - nq, o)) * 4;
                ol[u] = __shfl_sync(0xffffffffu, len, o);
                ok[u] = __shfl_sync(0xffffffffu, k, o);
                const long long oo = __shfl_sync(0xffffffffu, off, o);
                a[u] = make_int4(HOLE, HOLE, HOLE, HOLE);
                if (q < total) a[u] = __ldcs(reinterpret_cast<const int4*>(g.adj + oo + t0[u]));
            }
            int n[4];
#pragma unroll
            for (int u = 0; u < 4; u++) n[u] = sd_quad(core, a[u], t0[u], ol[u], ok[u]);
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (n[u]) atomicAdd(&sum[own[u]], n[u]);
        }
        __syncwarp();
        if (k >= 0 && !hub) {
            const int sd = sum[lane];
            g.hc[v].y = sd;
            g.kc[v] = key_of(k, sd);
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(256) init_mcd_hub_kernel(DevGraph g, const int32_t* __restrict__ core,
                                                           const int32_t* __restrict__ hubs, const Ctl* c) {
    const long long n = (long long)vload64(&c->gather_n);
    __shared__ int s_sd;
    for (long long i = blockIdx.x; i < n; i += gridDim.x) {
        const int v = hubs[i];
        const int k = core[v], len = g.end[v];
        const int32_t* list = g.adj + g.off[v];
        if (threadIdx.x == 0) s_sd = 0;
        __syncthreads();
        int sd = 0;
        for (int s = 0; s < len; s += 4096) {
            int4 a[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int t0 = s + u * 1024 + threadIdx.x * 4;
                a[u] = t0 < len ? __ldcs(reinterpret_cast<const int4*>(list + t0)) : make_int4(HOLE, HOLE, HOLE, HOLE);
            }
#pragma unroll
            for (int u = 0; u < 4; u++) sd += sd_quad(core, a[u], s + u * 1024 + threadIdx.x * 4, len, k);
        }
        sd = warp_sum(sd);
        if (lane_id() == 0) atomicAdd(&s_sd, sd);
        __syncthreads();
        if (threadIdx.x == 0) {
            g.hc[v].y = s_sd;
            g.kc[v] = key_of(k, s_sd);
        }
        __syncthreads();
    }
}

cudaError_t build_index(const int32_t* E, long long m, DevGraph g, int2* at, Ctl* c, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    build_index_kernel<<<grid_for(m, 256, 1ll << 31), 256, 0, s>>>(E, m, g, at, c);
    return cudaGetLastError();
}
cudaError_t assign_offsets(DevGraph g, int32_t v0, int32_t v1, Ctl* c, cudaStream_t s) {
    if (v1 <= v0) return cudaSuccess;
    offsets_kernel<<<grid_for(v1 - v0, 256, 65536), 256, 0, s>>>(g, v0, v1, c, 0);
    return cudaGetLastError();
}
cudaError_t scatter_edges(const int32_t* E, const int2* at, long long m, DevGraph g, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    scatter_kernel<<<grid_for(m, 256, 1ll << 31), 256, 0, s>>>(E, at, m, g);
    return cudaGetLastError();
}
cudaError_t set_cores(const int32_t* cores, DevGraph g, cudaStream_t s) {
    if (g.n <= 0) return cudaSuccess;
    set_cores_kernel<<<grid_for(g.n, 256, 1ll << 31), 256, 0, s>>>(cores, g);
    return cudaGetLastError();
}
cudaError_t init_mcd(DevGraph g, int32_t v0, int32_t v1, int32_t* core_scratch, int32_t* hub_scratch, Ctl* c,
                     cudaStream_t s) {
    if (v1 <= v0) return cudaSuccess;
    const cudaError_t e = cudaMemsetAsync(&c->gather_n, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    copy_cores_kernel<<<grid_for(g.n, 256, 1ll << 31), 256, 0, s>>>(g, core_scratch);
    init_mcd_kernel<<<grid_for(v1 - v0, 256, 65536), 256, 0, s>>>(g, v0, v1, core_scratch, hub_scratch, c);
    init_mcd_hub_kernel<<<1024, 256, 0, s>>>(g, core_scratch, hub_scratch, c);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ peeling
// The store as cm_peel.cuh reads it: lists start 16-byte aligned, their
// capacity is a multiple of 4 (so a quad never leaves the list's
// allocation) and deleted entries are holes.
struct PeelStore {
    DevGraph d;
    int n;
    __device__ bool live(int v) const { return d.hc[v].x != -1; }
    __device__ int degree(int v) const { return d.deg[v]; }
    __device__ int* core(int v) const { return &d.hc[v].x; }
    __device__ void list(int v, long long& off, int& len) const {
        off = d.off[v];
        len = d.end[v];
    }
    __device__ int quads(long long, int len) const { return (len + 3) >> 2; }
    __device__ int4 quad(long long off, int len, int j) const {
        int4 a = __ldcs(reinterpret_cast<const int4*>(d.adj + off + 4ll * j));
        if (4 * j + 1 >= len) a.y = HOLE;
        if (4 * j + 2 >= len) a.z = HOLE;
        if (4 * j + 3 >= len) a.w = HOLE;
        return a;
    }
};

__global__ void __launch_bounds__(kPeelThreads, 1) peel_kernel(PeelParams P) {
    __shared__ PeelShared S;
    const PeelStore g{P.g, P.g.n};
    const PeelWork W{P.ctl, P.dcur, P.list, P.far, P.chunks, P.chunk_cap, gridDim.x, P.limit_ns};
    peel_graph(g, W, S);
}

// Cooperative: at most one block per SM, which the grid barrier needs resident.
cudaError_t launch_peel(const PeelParams& p, int blocks, cudaStream_t s) {
    PeelParams q = p;
    void* args[] = {&q};
    return cudaLaunchCooperativeKernel((const void*)peel_kernel, dim3(blocks), dim3(kPeelThreads), args, 0, s);
}

// ------------------------------------------------------------------ index rehash
__global__ void rehash_kernel(const Bucket* __restrict__ old_idx, unsigned long long old_size, DevGraph g, Ctl* c) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)old_size) return;
    Bucket b = old_idx[i];
    if (b.key == KEY_EMPTY || b.key == KEY_TOMB) return;
    bool existed = false;
    long long nb = idx_insert(g.idx, g.idx_mask, b.key, &existed);
    if (nb < 0) { atomicCAS(&c->error, 0, E_INDEX_FULL); return; }
    g.idx[nb].slo = b.slo;
    g.idx[nb].shi = b.shi;
}

cudaError_t rehash(const Bucket* old_idx, unsigned long long old_size, DevGraph g, Ctl* c, cudaStream_t s) {
    if (old_size == 0) return cudaSuccess;
    rehash_kernel<<<grid_for((long long)old_size, 256, 1ll << 31), 256, 0, s>>>(old_idx, old_size, g, c);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ vertex insertion
// Neighbour lists of `count` new vertices (ids base..base+count-1): every
// neighbour is live or new, and not the vertex itself.  Warp per vertex.
__global__ void validate_vertices_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ nb, int32_t count,
                                         int32_t base, DevGraph g, Ctl* c) {
    long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    int lane = lane_id();
    for (; w < count; w += nw) {
        long long a = off[w], b = off[w + 1];
        if (a < 0 || b < a) {
            if (lane == 0) atomicCAS(&c->error, 0, E_INVALID);
            continue;
        }
        for (long long j = a + lane; j < b; j += 32) {
            int32_t x = nb[j];
            bool bad = x < 0 || x >= base + count || x == base + w || (x < base && g.hc[x].x < 0);
            if (bad) {
                atomicMin(&c->bad_index, j);
                atomicCAS(&c->error, 0, E_INVALID);
            }
        }
    }
}

__global__ void init_vertices_kernel(const int64_t* __restrict__ off, int32_t count, int32_t base, DevGraph g, Ctl* c) {
    long long b0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll;
    long long stride = (long long)gridDim.x * blockDim.x;
    int lane = lane_id();
    for (; b0 < count; b0 += stride) {
        long long i = b0 + lane;
        int cp = 0;
        if (i < count) cp = cap_for(off[i + 1] - off[i], g.slack_pct, g.min_cap);
        int incl = cp;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        int tot = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long wb = 0;
        if (lane == 31) wb = atomicAdd(&c->adj_top, (unsigned long long)tot);
        wb = __shfl_sync(0xffffffffu, wb, 31);
        if (i < count) {
            long long v = base + i;
            g.off[v] = (int64_t)(wb + incl - cp);
            g.cap[v] = cp;
            g.end[v] = 0;
            g.deg[v] = 0;
            g.hc[v] = make_int2(0, 0);
            g.kc[v] = key_of(0, 0);
            g.hw[v] = 0ull;
            g.chg[v] = 0;
            g.taken[v] = 0;
            g.claim0[v] = CLAIM_FREE;
            g.claim1[v] = CLAIM_FREE;
            g.need[v] = 0;
        }
    }
}

__global__ void expand_vertex_edges_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ nb,
                                           int32_t count, int32_t base, int32_t* E) {
    long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    int lane = lane_id();
    for (; w < count; w += nw) {
        for (long long j = off[w] + lane; j < off[w + 1]; j += 32) {
            E[2 * j] = base + (int32_t)w;
            E[2 * j + 1] = nb[j];
        }
    }
}

cudaError_t validate_vertices(const int64_t* nbr_off, const int32_t* nbrs, int32_t count, int32_t base, DevGraph g,
                              Ctl* c, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    validate_vertices_kernel<<<grid_for((long long)count * 32, 256, 65536), 256, 0, s>>>(nbr_off, nbrs, count, base, g, c);
    return cudaGetLastError();
}
cudaError_t init_vertices(const int64_t* nbr_off, int32_t count, int32_t base, DevGraph g, Ctl* c, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    init_vertices_kernel<<<grid_for(count, 256, 65536), 256, 0, s>>>(nbr_off, count, base, g, c);
    return cudaGetLastError();
}
cudaError_t expand_vertex_edges(const int64_t* nbr_off, const int32_t* nbrs, int32_t count, int32_t base, int32_t* E,
                                cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    expand_vertex_edges_kernel<<<grid_for((long long)count * 32, 256, 65536), 256, 0, s>>>(nbr_off, nbrs, count, base, E);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ vertex deletion
__global__ void validate_ids_kernel(const int32_t* __restrict__ ids, int32_t count, DevGraph g, Ctl* c) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    int32_t v = ids[i];
    if (v < 0 || v >= g.n || g.hc[v].x < 0) {
        atomicMin(&c->bad_index, i);
        atomicCAS(&c->error, 0, E_INVALID);
        return;
    }
    atomicAdd(&c->reloc_need, (unsigned long long)g.end[v]);   // upper bound on incident edges
}

__global__ void gather_incident_kernel(const int32_t* __restrict__ ids, int32_t count, DevGraph g, int2* E,
                                       long long cap, Ctl* c) {
    long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    int lane = lane_id();
    for (; w < count; w += nw) {
        int v = ids[w];
        long long o = g.off[v];
        int len = g.end[v];
        for (int t0 = 0; t0 < len; t0 += 32) {
            int t = t0 + lane;
            int x = t < len ? g.adj[o + t] : HOLE;
            bool live = x >= 0;
            unsigned int b = __ballot_sync(0xffffffffu, live);
            unsigned long long base = 0;
            if (lane == 0 && b) base = atomicAdd(&c->gather_n, (unsigned long long)__popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            long long p = (long long)base + __popc(b & ((1u << lane) - 1));
            if (live && p < cap) E[p] = make_int2(v, x);
        }
    }
}

__global__ void mark_dead_kernel(const int32_t* __restrict__ ids, int32_t count, DevGraph g) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    int32_t v = ids[i];
    g.hc[v] = make_int2(-1, 0);
    g.kc[v] = KEY_DEAD;
    g.hw[v] = 0ull;
    g.end[v] = 0;
    g.deg[v] = 0;
}

// Vertices being deleted keep their core for the rest of the call and count
// as fixed support for their neighbours while their edges go (PIN_SD).
__global__ void pin_vertices_kernel(const int32_t* __restrict__ ids, int32_t count, DevGraph g) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    g.hc[ids[i]].y = PIN_SD;
    atomicOr(&g.kc[ids[i]], 1u);
}

cudaError_t pin_vertices(const int32_t* ids, int32_t count, DevGraph g, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    pin_vertices_kernel<<<grid_for(count, 256), 256, 0, s>>>(ids, count, g);
    return cudaGetLastError();
}

cudaError_t validate_ids(const int32_t* ids, int32_t count, DevGraph g, Ctl* c, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    validate_ids_kernel<<<grid_for(count, 256), 256, 0, s>>>(ids, count, g, c);
    return cudaGetLastError();
}
cudaError_t gather_incident(const int32_t* ids, int32_t count, DevGraph g, int32_t* E, long long cap, Ctl* c,
                            cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    gather_incident_kernel<<<grid_for((long long)count * 32, 256, 65536), 256, 0, s>>>(ids, count, g, (int2*)E, cap, c);
    return cudaGetLastError();
}
cudaError_t mark_dead(const int32_t* ids, int32_t count, DevGraph g, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    mark_dead_kernel<<<grid_for(count, 256), 256, 0, s>>>(ids, count, g);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ export
__global__ void export_cores_kernel(DevGraph g, int32_t* out) {
    long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= g.n) return;
    out[v] = g.hc[v].x;
}

// SD (Definition 7) of every vertex; -1 for a deleted vertex.
__global__ void export_sd_kernel(DevGraph g, int32_t* out) {
    long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= g.n) return;
    const int2 h = g.hc[v];
    out[v] = h.x < 0 ? -1 : h.y;
}

__global__ void export_edges_kernel(DevGraph g, int2* out, Ctl* c) {
    long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    int lane = lane_id();
    for (; w < g.n; w += nw) {
        long long o = g.off[w];
        int len = g.end[w];
        for (int t0 = 0; t0 < len; t0 += 32) {
            int t = t0 + lane;
            int x = t < len ? g.adj[o + t] : HOLE;
            bool p = x > (int)w;
            unsigned int b = __ballot_sync(0xffffffffu, p);
            unsigned long long base = 0;
            if (lane == 0 && b) base = atomicAdd(&c->gather_n, (unsigned long long)__popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (p) out[base + __popc(b & ((1u << lane) - 1))] = make_int2((int)w, x);
        }
    }
}

// Consistency of the store with its own definitions (a debug check, run on
// request).  Per live vertex v, from its list: SD (Definition 7) recounted
// from the neighbours' cores against hc[v].y; the scan key against core and
// the stored SD; the live degree against the list's non-hole slots; every
// slot a hole or a live vertex id; and the k-core condition (at least
// core(v) neighbours of core >= core(v)).  A pinned vertex (vertex deletion
// in progress) keeps its pinned SD and is not compared on SD, key or the
// k-core condition.  A dead vertex must carry the dead key.  Warp per
// vertex; out[0..4] count the mismatches of the five checks, out[5] the
// vertices checked, out[6] the smallest vertex that failed a check.
__global__ void check_store_kernel(DevGraph g, unsigned long long* out) {
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id();
    for (long long v = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < g.n; v += nw) {
        const int2 h = g.hc[v];
        const uint32_t key = g.kc[v];
        if (h.x < 0) {
            if (lane == 0) {
                atomicAdd(&out[5], 1ull);
                if (key != KEY_DEAD) {
                    atomicAdd(&out[1], 1ull);
                    atomicMin(&out[6], (unsigned long long)v);
                }
            }
            continue;
        }
        const long long o = g.off[v];
        const int len = g.end[v];
        int sd = 0, live = 0, bad = 0;
        for (int t = lane; t < len; t += 32) {
            const int w = g.adj[o + t];
            if (w == HOLE) continue;
            if (w < 0 || w >= g.n) {
                bad++;
                continue;
            }
            const int cw = g.hc[w].x;
            if (cw < 0) {
                bad++;
                continue;
            }
            live++;
            sd += cw >= h.x;
        }
        sd = warp_sum(sd);
        live = warp_sum(live);
        bad = warp_sum(bad);
        if (lane == 0) {
            const bool pinned = h.y == PIN_SD;
            bool fail = false;
            if (!pinned && sd != h.y) {
                atomicAdd(&out[0], 1ull);
                fail = true;
            }
            if (!pinned && key != key_of(h.x, h.y)) {
                atomicAdd(&out[1], 1ull);
                fail = true;
            }
            if (live != g.deg[v]) {
                atomicAdd(&out[2], 1ull);
                fail = true;
            }
            if (bad) {
                atomicAdd(&out[3], (unsigned long long)bad);
                fail = true;
            }
            if (!pinned && sd < h.x) {
                atomicAdd(&out[4], 1ull);
                fail = true;
            }
            atomicAdd(&out[5], 1ull);
            if (fail) atomicMin(&out[6], (unsigned long long)v);
        }
    }
}

cudaError_t check_store(DevGraph g, unsigned long long* out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, 6 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(out + 6, 0xFF, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    if (g.n <= 0) return cudaSuccess;
    check_store_kernel<<<grid_for((long long)g.n * 32, 256, 65536), 256, 0, s>>>(g, out);
    return cudaGetLastError();
}

cudaError_t export_cores(DevGraph g, int32_t* out, cudaStream_t s) {
    if (g.n <= 0) return cudaSuccess;
    export_cores_kernel<<<grid_for(g.n, 256, 1ll << 31), 256, 0, s>>>(g, out);
    return cudaGetLastError();
}
cudaError_t export_sd(DevGraph g, int32_t* out, cudaStream_t s) {
    if (g.n <= 0) return cudaSuccess;
    export_sd_kernel<<<grid_for(g.n, 256, 1ll << 31), 256, 0, s>>>(g, out);
    return cudaGetLastError();
}
cudaError_t export_edges(DevGraph g, int32_t* out, Ctl* c, cudaStream_t s) {
    if (g.n <= 0) return cudaSuccess;
    export_edges_kernel<<<grid_for((long long)g.n * 32, 256, 65536), 256, 0, s>>>(g, (int2*)out, c);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ multi-graph helpers
// Local ids of a concatenated per-graph batch -> global ids.  prefix[i] is
// the first batch entry of graph i (ng+1 entries).
__global__ void localize_multi_kernel(int32_t* E, long long k, const unsigned long long* kp,
                                      const long long* __restrict__ prefix, const int32_t* __restrict__ bases,
                                      int32_t ng) {
    if (kp) k = (long long)vload64(kp);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += stride) {
        int lo = 0, hi = ng - 1;
        while (lo < hi) {                 // last graph whose prefix <= i
            int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= i) lo = mid; else hi = mid - 1;
        }
        int b = bases[lo];
        int nv = bases[lo + 1] - b;       // bases has ng+1 entries
        int32_t u = E[2 * i], v = E[2 * i + 1];
        // an id outside its graph stays invalid (negative) so ingest rejects it
        E[2 * i] = (u >= 0 && u < nv) ? u + b : -1;
        E[2 * i + 1] = (v >= 0 && v < nv) ? v + b : -1;
    }
}

__global__ void count_multi_kernel(const REdge* __restrict__ R, long long n, const unsigned long long* np,
                                   const int32_t* __restrict__ bases, int32_t ng, unsigned long long* per_graph) {
    if (np) n = (long long)vload64(np);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        int x = R[i].lo;
        int lo = 0, hi = ng - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (bases[mid] <= x) lo = mid; else hi = mid - 1;
        }
        atomicAdd(&per_graph[lo], 1ull);
    }
}

// Captured step: every id of a batch names a live vertex (checked for both
// batches before anything changes).  bad_index gets (phase << 40) | i.
__global__ void validate_pairs_kernel(const int32_t* __restrict__ E, long long k, const unsigned long long* kp,
                                      int phase, DevGraph g, Ctl* c) {
    if (kp) k = (long long)vload64(kp);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += stride) {
        int32_t u = E[2 * i], v = E[2 * i + 1];
        if (u < 0 || v < 0 || u >= g.n || v >= g.n || g.hc[u].x < 0 || g.hc[v].x < 0) {
            atomicMin(&c->bad_index, ((long long)phase << 40) | i);
            atomicCAS(&c->error, 0, E_INVALID);
        }
    }
}

cudaError_t localize_multi(int32_t* E, long long k, const unsigned long long* kp, const long long* prefix,
                           const int32_t* bases, int32_t ng, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    localize_multi_kernel<<<grid_for(k, 256, 8192), 256, 0, s>>>(E, k, kp, prefix, bases, ng);
    return cudaGetLastError();
}
cudaError_t count_multi(const REdge* R, long long n, const unsigned long long* np, const int32_t* bases, int32_t ng,
                        unsigned long long* per_graph, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_multi_kernel<<<grid_for(n, 256, 8192), 256, 0, s>>>(R, n, np, bases, ng, per_graph);
    return cudaGetLastError();
}
cudaError_t validate_pairs(const int32_t* E, long long k, const unsigned long long* kp, int phase, DevGraph g, Ctl* c,
                           cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    validate_pairs_kernel<<<grid_for(k, 256, 8192), 256, 0, s>>>(E, k, kp, phase, g, c);
    return cudaGetLastError();
}

// capacity totals for a vertex range: sum_only pass of offsets_kernel
cudaError_t sum_caps(DevGraph g, int32_t v0, int32_t v1, Ctl* c, cudaStream_t s) {
    if (v1 <= v0) return cudaSuccess;
    offsets_kernel<<<grid_for(v1 - v0, 256, 65536), 256, 0, s>>>(g, v0, v1, c, 1);
    return cudaGetLastError();
}

}  // namespace cm
