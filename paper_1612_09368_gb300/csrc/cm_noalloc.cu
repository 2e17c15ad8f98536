// cm_noalloc.cu -- core numbers of a caller-provided CSR graph without any
// device allocation (cm_core_numbers_noalloc).
//
// Who needs this: callers that cannot call cudaMalloc -- a process whose
// framework has already reserved the device memory for its own pool, or a
// latency-critical loop that must not wait on the allocator (cudaMalloc and
// cudaFree can synchronise the device).  Every other entry point of this
// library allocates its graph store; this one only reads the caller's CSR
// and writes the caller's output array.
//
// Its scratch lives in one file-scope __device__ array (kScratchBytes, sized
// for kMaxVertices vertices).  Every GPU that loads the library holds it
// until the process exits.  All calls share it: a call clears what must
// start at zero, and two calls whose work overlaps on the GPU (for example
// on two streams) race on it.  The device address of the array is looked
// up once per device, on the first call made with that device current;
// make that first call before any stream capture.  Every call waits for its
// stream (it reads the kernel's error word back) before it returns.
#include <mutex>

#include "../../include/coremaint.h"
#include "cm_common.cuh"
#include "cm_peel.cuh"

namespace cm {

constexpr int32_t kMaxVertices = 1 << 20;
constexpr size_t kCtlBytes = 4096;
constexpr unsigned long long kMaxChunks = 1 << 18;   // chunk tasks of long lists (more: their block walks them alone)
// Ctl, 3 int32 per vertex, then the chunk tasks
constexpr size_t kScratchBytes = kCtlBytes + 3ull * sizeof(int32_t) * kMaxVertices + kMaxChunks * 8;
static_assert(sizeof(Ctl) <= kCtlBytes, "control block does not fit");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct PeelCsrParams {
    int32_t n;
    const int64_t* row_off;
    const int32_t* adj;
    int32_t* cores;
    unsigned char* scratch;
    unsigned long long limit_ns;
};

// A caller's CSR as cm_peel.cuh reads it.  Its lists start anywhere, so a
// list's quads are those of the array: a quad inside the list is one 16-byte
// load, one that reaches past either end is read by the slot (never outside
// the list).  Ids outside [0, n) are skipped.
struct PeelCsr {
    int n;
    const int64_t* row_off;
    const int32_t* adj;
    int32_t* cores;
    bool aligned;   // adj starts on a 16-byte boundary
    __device__ bool live(int) const { return true; }
    __device__ int degree(int v) const { return (int)(row_off[v + 1] - row_off[v]); }
    __device__ int* core(int v) const { return cores + v; }
    __device__ void list(int v, long long& off, int& len) const {
        off = row_off[v];
        len = (int)(row_off[v + 1] - off);
    }
    __device__ int quads(long long off, int len) const {
        return len <= 0 ? 0 : (int)(((off & 3) + len + 3) >> 2);
    }
    __device__ int slot(long long p, long long lo, long long hi) const {
        const int w = p >= lo && p < hi ? adj[p] : HOLE;
        return w < n ? w : HOLE;
    }
    __device__ int4 quad(long long off, int len, int j) const {
        const long long p = (off & ~3ll) + 4ll * j;
        if (aligned && p >= off && p + 4 <= off + len) {
            const int4 a = __ldcs(reinterpret_cast<const int4*>(adj + p));
            return make_int4(a.x < n ? a.x : HOLE, a.y < n ? a.y : HOLE, a.z < n ? a.z : HOLE, a.w < n ? a.w : HOLE);
        }
        return make_int4(slot(p, off, off + len), slot(p + 1, off, off + len), slot(p + 2, off, off + len),
                         slot(p + 3, off, off + len));
    }
};

__global__ void __launch_bounds__(kPeelThreads, 1) peel_csr_kernel(PeelCsrParams P) {
    __shared__ PeelShared S;
    int32_t* dcur = reinterpret_cast<int32_t*>(P.scratch + kCtlBytes);
    int32_t* list = dcur + kMaxVertices;
    int32_t* far = list + kMaxVertices;
    const PeelCsr g{P.n, P.row_off, P.adj, P.cores, (reinterpret_cast<uintptr_t>(P.adj) & 15) == 0};
    const PeelWork W{reinterpret_cast<Ctl*>(P.scratch), dcur, list, far,
                     reinterpret_cast<unsigned long long*>(far + kMaxVertices), kMaxChunks, gridDim.x, P.limit_ns};
    peel_graph(g, W, S);
}

// Per-device address of the scratch array (looked up once per device).
static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[64] = {nullptr};

static int scratch_for_current_device(unsigned char** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return CM_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return CM_ERR_CUDA;
        }
        g_noalloc_ptr[dev] = p;
    }
    *out = static_cast<unsigned char*>(g_noalloc_ptr[dev]);
    return CM_OK;
}

static bool on_device(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// A failed runtime call: clear the error it left, so that a later
// cudaGetLastError of the caller (or of a framework) does not report it.
static int cuda_failed() {
    cudaGetLastError();
    return CM_ERR_CUDA;
}

}  // namespace cm

using namespace cm;

extern "C" int cm_core_numbers_noalloc(int32_t n, const int64_t* row_off, const int32_t* adj, int32_t* cores,
                                       void* stream) {
    if (n < 0) return CM_ERR_INVALID;
    if (n > kMaxVertices) return CM_ERR_CAPACITY;
    if (n == 0) return CM_OK;
    if (!row_off || !adj || !cores) return CM_ERR_INVALID;
    if (!on_device(row_off) || !on_device(adj) || !on_device(cores)) return CM_ERR_INVALID;
    unsigned char* scratch = nullptr;
    int rc = scratch_for_current_device(&scratch);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    // the control block must start at zero; the per-vertex arrays are written before they are read
    if (cudaMemsetAsync(scratch, 0, kCtlBytes, s) != cudaSuccess) return cuda_failed();
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cuda_failed();
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cuda_failed();
    // one block per SM; fewer for a small graph (a block scans at least 256 vertices)
    int blocks = sms < 1000 ? sms : 1000;
    const int want = (int)(((long long)n + 255) / 256);
    if (want < blocks) blocks = want > 0 ? want : 1;
    PeelCsrParams p{};
    p.n = n;
    p.row_off = row_off;
    p.adj = adj;
    p.cores = cores;
    p.scratch = scratch;
    p.limit_ns = 4000000000ull;
    void* args[] = {&p};
    if (cudaLaunchCooperativeKernel((const void*)peel_csr_kernel, dim3(blocks), dim3(kPeelThreads), args, 0, s) != cudaSuccess)
        return cuda_failed();
    int err = 0;
    if (cudaMemcpyAsync(&err, &reinterpret_cast<Ctl*>(scratch)->error, sizeof(int), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return cuda_failed();
    return err ? CM_ERR_LIMIT : CM_OK;
}
