// cc_noalloc.cu -- cc_components_noalloc: the connected-component split of
// a caller-held particle state with no device allocation at all.
//
// Who needs it: a caller whose device memory is owned by another allocator
// (a framework's caching pool that has reserved the GPU's memory, or a
// fixed budget handed out up front) cannot count on a cudaMalloc from this
// library succeeding, and a caller in a latency-critical loop cannot accept
// the device-wide synchronisation that cudaMalloc and cudaFree imply.  The
// context-based entry points allocate on the first use of every level, so
// this entry point instead keeps its union-find scratch in a fixed,
// file-scope device array: every GPU that loads libcc.so holds
// CC_NOALLOC_MAX_N * 8 bytes (512 KiB) of it until the process exits.
//
// The array's name in host code is a host-side stand-in, not a device
// address: kernels get the address from cudaGetSymbolAddress, looked up once
// per device (with that device current) on the first call made there.
#include <mutex>

#include "cc_internal.cuh"

namespace cc {

// parent[] and component sizes, then the component count, the finished
// blocks of the last kernel and the tau kernel's counters
constexpr int NA_WORDS = 64, NA_CTR_AT = 8;
static __device__ __align__(256) int32_t g_noalloc_scratch[2 * CC_NOALLOC_MAX_N + NA_WORDS];
static_assert(NA_CTR_AT * 4 + sizeof(DevCounters) <= NA_WORDS * 4, "counters in the scratch tail");

namespace {

constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mutex;
int32_t *g_na_ptr[NA_MAX_DEVICES] = {};

struct NaScratch {
    int32_t *parent, *cnt;
    int32_t *ncomp;
    unsigned *done;
    DevCounters *ctr;
};

NaScratch na_view(int32_t *base)
{
    NaScratch s;
    int32_t *tail = base + 2 * CC_NOALLOC_MAX_N;
    s.parent = base;
    s.cnt = base + CC_NOALLOC_MAX_N;
    s.ncomp = tail;
    s.done = (unsigned *)(tail + 1);
    s.ctr = (DevCounters *)(tail + NA_CTR_AT);
    return s;
}

}  // namespace

// every word this call reads must start fresh: the array keeps the previous
// call's contents
__global__ void k_na_init(NaScratch S, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) {
        S.parent[k] = k;
        S.cnt[k] = 0;
    }
    if (k == 0) {
        *S.ncomp = 0;
        *S.done = 0u;
        S.ctr->edges = 0ull;
        S.ctr->tau_fp64 = 0ull;
        S.ctr->err = 0u;
    }
}

// label = root = smallest index of the component; a component is counted when
// its second member arrives (one size update per root and warp); the last
// block writes the count
__global__ void k_na_compress(int n, NaScratch S, int32_t *labels, int64_t *n_comp_out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    int r = -1;
    if (k < n) {
        r = uf_find(S.parent, k);
        labels[k] = r;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, r);
    if (r >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) {
        const int add = __popc(peers), old = atomicAdd(&S.cnt[r], add);
        if (old < 2 && old + add >= 2) atomicAdd(S.ncomp, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(S.done, 1u) == gridDim.x - 1) *n_comp_out = atomicAdd(S.ncomp, 0);
    }
}

}  // namespace cc

using namespace cc;

// Can a kernel on the current device read and write `ptr`?  Device and
// managed memory, and pinned host memory mapped into the device's address
// space, can; pageable host memory is refused (a kernel touching it would
// fault instead of returning an error).
static bool device_reachable(const void *ptr)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return a.devicePointer != nullptr;
    if (a.type == cudaMemoryTypeHost) return a.devicePointer == ptr;
    return false;
}

// device address of the scratch array for the current device, looked up
// once per device (with that device current) and kept for the life of the
// process (a cudaDeviceReset invalidates it; calls after one are not
// supported)
static int na_scratch(int32_t **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
        cudaGetLastError();
        return CC_E_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        int32_t *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return CC_E_CUDA;
        }
        g_na_ptr[dev] = p;
    }
    *out = g_na_ptr[dev];
    return CC_OK;
}

extern "C" int cc_components_noalloc(const double *m, const double *x3, const double *v3, int64_t n,
                                     const cc_params *p, double h, int32_t *labels_out, int64_t *n_comp_out,
                                     void *stream)
{
    if (!m || !x3 || !v3 || !p || !labels_out || !n_comp_out || !(h > 0.0) || !isfinite(h) || n < 1)
        return CC_E_ARG;
    // the parameters cc_init accepts for the same threshold test
    if (!(p->G > 0.0) || !isfinite(p->G) || !(p->eps >= 0.0) || !isfinite(p->eps) || !(p->eta > 0.0) ||
        !isfinite(p->eta) || (p->eta_outside != 0 && p->eta_outside != 1))
        return CC_E_ARG;
    if (n > CC_NOALLOC_MAX_N) return CC_E_CAPACITY;  // beyond the fixed scratch array
    // every pointer is read or written by a kernel: refuse what it cannot reach
    const void *ptrs[5] = {m, x3, v3, labels_out, n_comp_out};
    for (const void *q : ptrs)
        if (!device_reachable(q)) return CC_E_ARG;
    int32_t *base = nullptr;
    if (na_scratch(&base)) return CC_E_CUDA;
    const cudaStream_t s = (cudaStream_t)stream;
    const NaScratch S = na_view(base);
    TauParams P;
    P.G = p->G;
    P.eps2 = p->eps * p->eps;
    P.eta = p->eta;
    P.eta_in = p->eta_outside ? 1.0 : p->eta;
    P.eta_outside = p->eta_outside;
    P.h = h;
    P.near_tol = 0.0;
    P.fault_test = 0;
    const int ni = (int)n, g = (ni + 255) / 256;
    k_na_init<<<g, 256, 0, s>>>(S, ni);
    launch_tau_raw(m, x3, v3, ni, P, S.parent, S.ctr, s);
    k_na_compress<<<g, 256, 0, s>>>(ni, S, labels_out, n_comp_out);
    CC_COUNT_LAUNCH(2);
    if (cudaPeekAtLastError() != cudaSuccess) {  // a launch was refused: nothing was written
        cudaGetLastError();
        return CC_E_CUDA;
    }
    unsigned err = 0;
    if (cudaMemcpyAsync(&err, &S.ctr->err, sizeof(unsigned), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return CC_E_CUDA;
    }
    return err ? CC_E_TIMEOUT : CC_OK;
}
