// The library's allocations (ms_blocks.cu): host code only.
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

namespace ms {

struct DevCounters;

// True when a test asked for the next workspace allocation to fail
// (ms_inject_alloc_failure).
bool injected_alloc_failure();
// Device memory of a context or of ms_run_host, from what earlier ones left where
// it fits. Its first use follows on `st`.
struct Block {
    void* p = nullptr;
    bool pooled = false;
};
cudaError_t block_alloc(Block* b, size_t bytes, cudaStream_t st);
// Its return, once the work on `st` (all of the work on it) has ended. What cannot be
// waited for, on a stream that is being captured, is not handed out again.
void block_free(const Block& b, cudaStream_t st);
// cudaMalloc that gives back what the library keeps before it reports that the
// device is out of memory.
cudaError_t device_malloc(void** p, size_t bytes);
// Stream-ordered scratch from the library's own pool (kept mapped between calls);
// free with cudaFreeAsync.
cudaError_t scratch_malloc_async(void** p, size_t bytes, cudaStream_t st);
// Pinned counters of one context, and their return, no copy into them pending.
cudaError_t counters_alloc(DevCounters** p, size_t bytes);
void counters_free(DevCounters* p);

}  // namespace ms
