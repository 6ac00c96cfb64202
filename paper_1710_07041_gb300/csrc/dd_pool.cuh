// Cache of solver workspaces (dd_pool.cu): device buffers keyed by (device,
// size) and pinned host buffers. pool_dev_free / pool_host_free require that
// no queued GPU work still uses the buffer.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace dd {
void *pool_dev_alloc(size_t bytes);   // a cached buffer of exactly this size, else dev_malloc
void pool_dev_free(void *p, size_t bytes);
void *pool_host_alloc(size_t bytes);
void pool_host_free(void *p, size_t bytes);
size_t pool_cached_bytes();   // device bytes cached for the current device
// stream-ordered device memory for the work fields of one call (n bytes, freed
// with cudaFreeAsync on the same stream); nullptr where there is none
void *pool_stream_alloc(size_t n, cudaStream_t st);
void pool_release();          // free every cached buffer
// cudaMalloc for memory that an object keeps; where it fails, once more with
// everything cached here given back
cudaError_t dev_malloc_bytes(void **p, size_t n);
template <typename T> cudaError_t dev_malloc(T **p, size_t n) { return dev_malloc_bytes((void **)p, n); }
}  // namespace dd
