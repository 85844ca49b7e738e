// Scratch of calls that allocate per call (FW-H integration, spectra): stream-
// ordered allocations from one memory pool per device context.  cudaMalloc and
// cudaFree cost 65 us a pair below 64 MB and 250 us at 256 MB, and cudaFree waits for
// the whole device; a pooled pair costs a few microseconds once the pool holds memory.
// The pool keeps at most POOL_KEEP bytes between calls (the driver releases what is
// above at the next synchronisation) and gives everything back when a context is
// loaded or destroyed (fr_pool_trim).  cudaDeviceReset ends a context and its pool;
// the next call makes another.  Safe with several threads and streams: the driver
// orders the reuse of a block after its last use.
#pragma once

#include <cuda_runtime.h>

constexpr unsigned long long POOL_KEEP = 256ull << 20;

// n bytes usable on stream s; false if the device has no pools or the pool cannot
// grow (the caller then allocates for itself)
bool fr_pool_alloc(void** p, size_t n, cudaStream_t s);
void fr_pool_free(void* p, cudaStream_t s);
// returns the unused memory of the current context's pool to the device
void fr_pool_trim();
