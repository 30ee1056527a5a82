// Which of the caller's buffers the network's kernels use themselves; the others are staged: inputs
// copied to the handle's buffers before the kernels, outputs copied from them afterwards.  Plain
// C++, no CUDA call.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace mlpbuf {

// device memory of the handle's own device, or managed memory, of whole words.  Memory of another
// device may not be mapped into this one, which a kernel would fault on; a copy can reach it.
inline bool in_place(bool device_memory, bool managed, int device, int own_device, uintptr_t addr) {
  return addr % 4 == 0 && (managed || (device_memory && device == own_device));
}

inline bool overlap(uintptr_t a, size_t na, uintptr_t b, size_t nb) { return a < b + nb && b < a + na; }

}  // namespace mlpbuf
