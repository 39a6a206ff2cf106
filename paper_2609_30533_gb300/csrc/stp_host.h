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

}  // namespace stp
