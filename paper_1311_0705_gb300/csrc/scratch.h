// Stream-ordered device scratch that survives the call.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace hg {

// A block of device memory from scratch_get.
struct Scratch {
    void *p = nullptr;
    size_t bytes = 0;
    cudaEvent_t done = nullptr;  // (kept blocks) the end of the block's last use
};

// At least `bytes` of device memory on the current device, to be used on `stream` (the contents are arbitrary).
cudaError_t scratch_get(Scratch &s, size_t bytes, cudaStream_t stream);
// Give a block back; `stream` is where its last use was enqueued.  Nothing happens for an empty block.
void scratch_put(Scratch &s, cudaStream_t stream);
// A grid or ray plan of a device came to life (+1) or was released (-1); with the last one the kept blocks
// are released.
void scratch_users(int device, int delta);
// cudaMalloc on the current device; when it fails, once more without the kept blocks.
cudaError_t device_malloc(void **p, size_t bytes);

}  // namespace hg
