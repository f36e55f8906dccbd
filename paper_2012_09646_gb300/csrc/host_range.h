// Whether a memory range lies within an allocation (host code only).
#pragma once

#include <cstddef>
#include <cstdint>

namespace gdag {

// [p, p + bytes) within [start, start + size); sums that wrap are outside
inline bool range_holds(uint64_t start, uint64_t size, uint64_t p, uint64_t bytes)
{
    return p >= start && p - start <= size && bytes <= size - (p - start);
}

}  // namespace gdag
