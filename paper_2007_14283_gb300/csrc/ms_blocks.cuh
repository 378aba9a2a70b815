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
// it fits. Its first use follows on `st`. Freed by block_free once no work on it is
// left.
cudaError_t block_alloc(void** p, size_t bytes, cudaStream_t st);
void block_free(void* p);
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
