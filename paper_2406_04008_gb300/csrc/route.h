// Which of the caller's buffers a kernel takes directly (host code, no CUDA calls).
#pragma once
#include <cuda_runtime_api.h>

namespace collage {

// type, device: the buffer's, as cudaPointerGetAttributes reports them; own: the handle's device.  Only
// memory that lies on the handle's device: a peer's needs access that nobody may have enabled, and
// what the runtime does not know (pageable host memory, a stray address) is its copy's to refuse.
inline bool kernel_route(cudaMemoryType type, int device, int own) {
  return type == cudaMemoryTypeDevice && device == own;
}

}  // namespace collage
