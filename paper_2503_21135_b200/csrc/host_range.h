// Whether one range of addresses lies within another.  Plain C++, no CUDA.
#pragma once
#include <stdint.h>

namespace dyn {

// [p, p + bytes) within [start, start + size); sizes whose ends pass the last address are never within anything.
static inline bool range_covers(uint64_t start, uint64_t size, uint64_t p, uint64_t bytes) {
    return p >= start && bytes <= size && p - start <= size - bytes;
}

}  // namespace dyn
