// Device scratch memory of single calls.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace nm {

// Stream-ordered scratch from a memory pool of the library's own, one per
// device, which keeps up to kPoolKeep bytes over synchronisations (the default
// pool returns everything to the device at each one, and the next call maps it
// anew).  nm_release_cached_memory returns what is kept.  For any thread and
// stream; allocation nodes under capture.
constexpr uint64_t kPoolKeep = 512ull << 20;
cudaError_t stream_alloc(void** p, size_t bytes, cudaStream_t s);
cudaError_t stream_free(void* p, cudaStream_t s);

}  // namespace nm
