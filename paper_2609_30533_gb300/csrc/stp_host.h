// Host-side decisions about a caller's buffers (no CUDA types).
#pragma once

#include <cstddef>
#include <cstdint>

namespace stp {

// Whether two byte ranges share a byte (a null or empty range shares none).
inline bool ranges_meet(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return a && b && na > 0 && nb > 0 && x < y + nb && y < x + na;
}

// Whether memory is another GPU's than the one that is current: a copy reaches it
// all the same, a kernel only with peer access. gpu: the memory lies on a GPU.
inline bool on_other_gpu(bool gpu, int owner, int current) { return gpu && owner != current; }

}  // namespace stp
