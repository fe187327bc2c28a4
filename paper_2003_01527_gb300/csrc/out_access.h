// Which result buffers of the caller the listing kernels store into
// themselves.  Host code only.  Not part of the public ABI.
#pragma once

#include <cstdint>

#include <cuda_runtime_api.h>

namespace gsm {

// Kernels of device `device` store rows through `out` only if it is memory of
// that very device (another device's memory needs a peer mapping that nobody
// has asked for, and managed memory would migrate) and takes their widest
// store, 16 bytes.  Everything else gets its rows by a copy, which reaches any
// memory.  `attr` are the attributes of `out`.
inline bool kernels_may_store(const cudaPointerAttributes &attr, const void *out, int device) {
  return attr.type == cudaMemoryTypeDevice && attr.device == device &&
         (reinterpret_cast<uintptr_t>(out) & 15) == 0;
}

}  // namespace gsm
