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

}  // namespace hgp
