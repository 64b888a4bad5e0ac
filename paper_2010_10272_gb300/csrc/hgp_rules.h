// Rules of the host code that need no CUDA (internal; plain C++, compiled on their own by the tests).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace hgp {

// [p, p + bytes) lies in [base, base + size)
inline bool range_inside(uintptr_t p, size_t bytes, uintptr_t base, size_t size)
{
    return p >= base && p - base <= size && bytes <= size - (p - base);
}

// entries of the chunk that starts at p0 <= end, of a list that ends at `end` (up to 2^31 - 1, where
// p0 + chunk would overflow)
#ifdef __CUDACC__
__host__ __device__
#endif
inline int32_t chunk_length(int32_t p0, int32_t end, int32_t chunk) { return end - p0 < chunk ? end - p0 : chunk; }

}  // namespace hgp
