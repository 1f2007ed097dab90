// Whether a block of memory holds a range.
#pragma once
#include <stdint.h>

namespace lddmm {

// [p, p + bytes) inside [base, base + size)?
inline bool span_holds(uint64_t base, uint64_t size, uint64_t p, uint64_t bytes) {
  return p >= base && p - base <= size && bytes <= size - (p - base);
}

}  // namespace lddmm
