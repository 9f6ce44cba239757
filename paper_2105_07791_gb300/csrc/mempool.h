// The library's stream-ordered device pool and page-locked staging buffers
// (mempool.cpp).
#pragma once

#include <cstddef>

#include <cuda_runtime.h>

namespace ndhss {

// Stream-ordered allocation from the library's per-device pool (freed memory
// stays cached between calls); release with cudaFreeAsync.
cudaError_t pool_malloc_async(void** p, size_t bytes, cudaStream_t st);

constexpr size_t PINNED_BYTES = size_t(4) << 20;
struct PinnedBuf {
    unsigned char* p = nullptr;     // PINNED_BYTES of page-locked memory
    cudaEvent_t ev = nullptr;       // its last user's copies
    int dev = 0;
};
// A buffer no copy reads any more, or null (the caller then copies from
// pageable memory).  Release with the stream its copies were enqueued on.
PinnedBuf* pinned_acquire();
void pinned_release(PinnedBuf* b, cudaStream_t st);

}  // namespace ndhss
