// Device and pinned memory of the library.
//
// A program that makes a context per frame paid cudaMalloc, cudaFree and the
// pinned counters' cudaMallocHost and cudaFreeHost for each: 743 us a frame of
// 20,000 pixels, 533 us with memory that earlier contexts left. That memory lies in
// a pool of the library's own on each device (cudaMemPool), which keeps up to
// kKeepBytes of it mapped; the pool and not this file knows its blocks. What is in
// the pool unused, the driver takes back by itself for any cudaMalloc of the process
// that would otherwise be out of memory (4 GB unused in a pool and 2 GB free: a
// cudaMalloc of 4 GB succeeds), and the library does so before it reports
// MS_ERR_OOM. Larger blocks are cudaMalloc's and cudaFree's.
//
// What is kept belongs to one CUDA context, by the context's id, which no later
// context of the process has: after a cudaDeviceReset nothing kept before it is
// touched again.
#include "ms_blocks.cuh"

#include <cuda.h>

#include <atomic>
#include <mutex>

namespace ms {
namespace {

constexpr size_t kKeepBytes = size_t(512) << 20;
constexpr int kMaxPools = 64;     // contexts with pools; the rest use cudaMalloc alone
constexpr int kKeepCounters = 16;

std::atomic<int32_t> g_fail_allocs{0};

// Id of the calling thread's CUDA context, 0 if it has none or it cannot be told.
unsigned long long context_id() {
    struct Fns {
        CUresult (*current)(CUcontext*) = nullptr;
        CUresult (*id)(CUcontext, unsigned long long*) = nullptr;
    };
    static const Fns fns = [] {
        Fns f;
        void *cur = nullptr, *id = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &cur, 4000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &id, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            f.current = reinterpret_cast<decltype(f.current)>(cur);
            f.id = reinterpret_cast<decltype(f.id)>(id);
        }
        return f;
    }();
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (!fns.id || fns.current(&c) != CUDA_SUCCESS || !c || fns.id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

struct Pools {
    unsigned long long ctx;
    cudaMemPool_t blocks, scratch;
};
std::mutex g_mu;
Pools g_pools[kMaxPools];
int g_n_pools = 0;

struct Pinned {
    unsigned long long ctx;
    void* p;
};
Pinned g_pinned[kKeepCounters];
int g_n_pinned = 0;

cudaError_t make_pool(int dev, uint64_t keep, cudaMemPool_t* pool) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    const cudaError_t e = cudaMemPoolCreate(pool, &props);
    if (e == cudaSuccess) cudaMemPoolSetAttribute(*pool, cudaMemPoolAttrReleaseThreshold, &keep);
    return e;
}

// The current context's pools, made at their first use; false without them.
bool current_pools(Pools* out) {
    const unsigned long long ctx = context_id();
    int dev = 0;
    if (ctx == 0 || cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    for (int i = 0; i < g_n_pools; ++i)
        if (g_pools[i].ctx == ctx) {
            *out = g_pools[i];
            return true;
        }
    Pools p{ctx, nullptr, nullptr};
    if (g_n_pools == kMaxPools || make_pool(dev, kKeepBytes, &p.blocks) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    // scratch: release threshold never, so calls that allocate a workspace per call
    // and synchronise do not re-map it each time
    if (make_pool(dev, UINT64_MAX, &p.scratch) != cudaSuccess) {
        cudaMemPoolDestroy(p.blocks);
        (void)cudaGetLastError();
        return false;
    }
    *out = g_pools[g_n_pools++] = p;
    return true;
}

// Unused memory of the current context's pools goes back to the device.
void give_back() {
    (void)cudaGetLastError();
    Pools p;
    if (!current_pools(&p)) return;
    cudaMemPoolTrimTo(p.blocks, 0);
    cudaMemPoolTrimTo(p.scratch, 0);
}

}  // namespace

bool injected_alloc_failure() {
    int32_t left = g_fail_allocs.load();
    while (left > 0 && !g_fail_allocs.compare_exchange_weak(left, left - 1)) {
    }
    return left > 0;
}

cudaError_t device_malloc(void** p, size_t bytes) {
    *p = nullptr;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    give_back();
    return cudaMalloc(p, bytes);
}

cudaError_t block_alloc(Block* b, size_t bytes, cudaStream_t st) {
    Pools pools;
    *b = Block{};
    if (bytes > kKeepBytes || !current_pools(&pools)) return device_malloc(&b->p, bytes);
    const cudaError_t e = cudaMallocFromPoolAsync(&b->p, bytes, pools.blocks, st);
    b->pooled = e == cudaSuccess;
    if (e != cudaErrorMemoryAllocation) return e;
    give_back();
    return cudaMalloc(&b->p, bytes);
}

// cudaFree hands a pool's block back to the pool without a wait, so the stream is
// waited for first; if that fails (a stream that was destroyed already), the device.
void block_free(const Block& b, cudaStream_t st) {
    if (!b.p) return;
    const bool idle = cudaStreamSynchronize(st) == cudaSuccess || cudaDeviceSynchronize() == cudaSuccess;
    if (idle || !b.pooled) cudaFree(b.p);
}

cudaError_t scratch_malloc_async(void** p, size_t bytes, cudaStream_t st) {
    Pools pools;
    *p = nullptr;
    if (!current_pools(&pools)) return cudaMallocAsync(p, bytes, st);
    const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pools.scratch, st);
    if (e != cudaErrorMemoryAllocation) return e;
    give_back();
    return cudaMallocFromPoolAsync(p, bytes, pools.scratch, st);
}

cudaError_t counters_alloc(DevCounters** p, size_t bytes) {
    const unsigned long long ctx = context_id();
    *p = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (int i = 0; ctx != 0 && i < g_n_pinned; ++i)
            if (g_pinned[i].ctx == ctx) {
                *p = static_cast<DevCounters*>(g_pinned[i].p);
                g_pinned[i] = g_pinned[--g_n_pinned];
                return cudaSuccess;
            }
    }
    return cudaMallocHost(reinterpret_cast<void**>(p), bytes);
}

void counters_free(DevCounters* p) {
    if (!p) return;
    const unsigned long long ctx = context_id();
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (ctx != 0 && g_n_pinned < kKeepCounters) {
            g_pinned[g_n_pinned++] = Pinned{ctx, p};
            return;
        }
    }
    cudaFreeHost(p);
}

}  // namespace ms

extern "C" __attribute__((visibility("default"))) void ms_inject_alloc_failure(int32_t count) {
    ms::g_fail_allocs.store(count > 0 ? count : 0);
}
