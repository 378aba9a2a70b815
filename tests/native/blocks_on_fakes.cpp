// ms_blocks.cu on fakes of the CUDA calls it makes (no GPU): a device of a stated
// size with memory pools that keep what is freed, up to three contexts' ids, and a
// count of calls that wait for the device or that touch memory of a dead context.
// Prints a line for each check that fails and returns their number.
#include <cuda.h>

#include <atomic>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#include "ms_blocks.cuh"

namespace {

struct Pool {
    size_t keep, unused;
};
struct Block {
    size_t bytes;
    Pool* pool;
    unsigned long long ctx;
};
std::mutex mu;
size_t device_free = size_t(1) << 30;
bool driver_trims = true;  // whether cudaMalloc takes unused pool memory by itself
unsigned long long ctx_now = 1;
std::map<void*, Block> live;
std::map<void*, unsigned long long> pinned;
std::vector<Pool*> pools;
std::map<Pool*, unsigned long long> pool_ctx;
uintptr_t next_addr = 0x1000;
bool capturing = false;  // the stream of the calls
std::atomic<int> stream_waits{0};
int device_waits = 0, dead_uses = 0, bad_frees = 0, mallocs = 0, host_mallocs = 0, errors_left = 0;

void trim(Pool* p, size_t to) {
    if (p->unused > to) {
        device_free += p->unused - to;
        p->unused = to;
    }
}
void reset() {  // cudaDeviceReset
    std::lock_guard<std::mutex> lk(mu);
    for (auto& b : live) device_free += b.second.bytes;
    for (Pool* p : pools) trim(p, 0);
    live.clear();
    pinned.clear();
    ++ctx_now;
}
CUresult get_current(CUcontext* c) {
    *c = reinterpret_cast<CUcontext>(uintptr_t(64));  // the same handle for every context, as a primary one's
    return CUDA_SUCCESS;
}
CUresult get_id(CUcontext, unsigned long long* id) {
    *id = ctx_now;
    return CUDA_SUCCESS;
}

}  // namespace

cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *fn = !strcmp(name, "cuCtxGetId") ? reinterpret_cast<void*>(&get_id) : reinterpret_cast<void*>(&get_current);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    errors_left = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    ++device_waits;
    return capturing ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    ++stream_waits;
    return capturing ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
    std::lock_guard<std::mutex> lk(mu);
    ++mallocs;
    if (bytes > device_free && driver_trims)
        for (Pool* q : pools) trim(q, 0);
    if (bytes > device_free) {
        errors_left = 1;
        return cudaErrorMemoryAllocation;
    }
    device_free -= bytes;
    *p = reinterpret_cast<void*>(next_addr += 0x1000);
    live[*p] = Block{bytes, nullptr, ctx_now};
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> lk(mu);
    auto it = live.find(p);
    if (it == live.end()) {
        ++bad_frees;
        return cudaErrorInvalidValue;
    }
    if (Pool* q = it->second.pool) {
        q->unused += it->second.bytes;
        trim(q, q->keep);
    } else {
        device_free += it->second.bytes;
    }
    live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps*) {
    std::lock_guard<std::mutex> lk(mu);
    pools.push_back(new Pool{0, 0});
    pool_ctx[pools.back()] = ctx_now;
    *pool = reinterpret_cast<cudaMemPool_t>(pools.back());
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t pool, cudaMemPoolAttr, void* v) {
    reinterpret_cast<Pool*>(pool)->keep = size_t(*static_cast<uint64_t*>(v));
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t to) {
    std::lock_guard<std::mutex> lk(mu);
    trim(reinterpret_cast<Pool*>(pool), to);
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t) {
    std::lock_guard<std::mutex> lk(mu);
    Pool* q = reinterpret_cast<Pool*>(pool);
    if (pool_ctx[q] != ctx_now) ++dead_uses;
    if (q->unused >= bytes) {
        q->unused -= bytes;
    } else {
        if (bytes - q->unused > device_free) {
            errors_left = 1;
            return cudaErrorMemoryAllocation;
        }
        device_free -= bytes - q->unused;
        q->unused = 0;
    }
    *p = reinterpret_cast<void*>(next_addr += 0x1000);
    live[*p] = Block{bytes, q, ctx_now};
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) { return cudaMalloc(p, bytes); }
cudaError_t cudaMallocHost(void** p, size_t) {
    std::lock_guard<std::mutex> lk(mu);
    ++host_mallocs;
    *p = reinterpret_cast<void*>(next_addr += 0x1000);
    pinned[*p] = ctx_now;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::lock_guard<std::mutex> lk(mu);
    if (!pinned.erase(p)) ++bad_frees;
    return cudaSuccess;
}

namespace {

int failed = 0;
void check(bool ok, const char* what) {
    if (!ok) {
        printf("FAILED: %s\n", what);
        ++failed;
    }
}
constexpr size_t MB = size_t(1) << 20;
bool take(ms::Block* p, size_t bytes) { return ms::block_alloc(p, bytes, nullptr) == cudaSuccess; }
void give(const ms::Block& b) {
    const int waits = stream_waits;
    ms::block_free(b, nullptr);
    check(stream_waits == waits + 1, "the stream is waited for");
}

}  // namespace

int main() {
    ms::Block a, b, c;
    void* m;
    void* m2;
    // kept within the bound, taken over, larger blocks not kept
    check(take(&a, 300 * MB) && take(&b, 300 * MB), "two blocks");
    give(a);
    give(b);
    check(device_free == 1024 * MB - 512 * MB, "512 MB are kept of 600");
    const size_t before = device_free;
    check(take(&a, 400 * MB) && device_free == before, "a block from what was left");
    give(a);
    check(take(&a, 513 * MB), "a block larger than what may be kept, where it fits only without the kept ones");
    give(a);
    check(device_free == 1024 * MB, "which is given back at once");

    // every allocation gets the kept memory, with a driver that takes it itself and one that does not
    for (int own = 0; own < 2; ++own) {
        driver_trims = own == 0;
        check(take(&a, 500 * MB), "a block");
        give(a);
        check(ms::device_malloc(&m, 900 * MB) == cudaSuccess && errors_left == 0, "a batch's workspace");
        cudaFree(m);
        check(take(&a, 500 * MB), "a block");
        give(a);
        check(ms::scratch_malloc_async(&m, 900 * MB, nullptr) == cudaSuccess && errors_left == 0, "scratch");
        cudaFree(m);  // the scratch pool keeps it
        check(device_free == 1024 * MB - 900 * MB, "scratch stays mapped");
        check(take(&a, 500 * MB) && errors_left == 0, "a block once the scratch is unused");
        check(!take(&c, 525 * MB) && take(&b, 500 * MB) && !take(&c, 100 * MB), "no more than there is");
        give(a);
        give(b);
        check(ms::device_malloc(&m, 1024 * MB) == cudaSuccess, "all of it");
        check(ms::device_malloc(&m2, MB) == cudaErrorMemoryAllocation, "out of memory is said");
        cudaFree(m);
    }
    driver_trims = true;

    // nothing kept crosses a device reset
    ms::DevCounters *h1, *h2;
    check(take(&a, 200 * MB) && ms::counters_alloc(&h1, 96) == cudaSuccess, "before the reset");
    give(a);
    ms::counters_free(h1);
    check(ms::counters_alloc(&h2, 96) == cudaSuccess && h2 == h1 && host_mallocs == 1, "counters are taken over");
    ms::counters_free(h2);
    reset();
    check(take(&a, 200 * MB) && ms::counters_alloc(&h2, 96) == cudaSuccess && host_mallocs == 2, "after the reset");
    check(h2 != h1 && dead_uses == 0, "nothing of the dead context");
    give(a);
    ms::counters_free(h2);

    // pinned counters are bounded
    std::vector<ms::DevCounters*> hs(40);
    for (auto& h : hs) ms::counters_alloc(&h, 96);
    for (auto& h : hs) ms::counters_free(h);
    check(pinned.size() <= 16, "at most 16 pinned buffers");

    // several threads
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([t] {
            for (int i = 0; i < 200; ++i) {
                ms::Block p;
                ms::DevCounters* h;
                if (take(&p, (1 + (t * 7 + i) % 20) * MB)) ms::block_free(p, nullptr);
                ms::counters_alloc(&h, 96);
                ms::counters_free(h);
            }
        });
    for (auto& t : ts) t.join();
    check(live.empty() && device_free >= 512 * MB, "threads leave no block");
    check(bad_frees == 0 && device_waits == 0, "no foreign free, no wait for the device");

    // a block whose stream is being captured is not handed out again, a larger one is freed
    check(take(&a, 100 * MB) && take(&b, 600 * MB), "blocks");
    capturing = true;
    ms::block_free(a, nullptr);
    ms::block_free(b, nullptr);
    capturing = false;
    check(live.size() == 1 && live.count(a.p) == 1, "the pool's block stays taken");
    return failed;
}
