// When a kernel may read or write a caller's array itself, in place of a copy.
#pragma once

#include <stddef.h>
#include <stdint.h>

// What the runtime says of a pointer: memory that a kernel on the current device reaches, and the allocation around it.
struct MemoryAt {
    bool reachable = false;
    uintptr_t base = 0;
    size_t size = 0;
};

// The whole array lies in such memory, aligned for its elements.  (A copy checks its range against the allocation and
// fails; a kernel that was given an array too short would read or write behind it.)
inline bool covers_array(const MemoryAt &m, uintptr_t p, size_t align, size_t bytes) {
    return p && p % align == 0 && m.reachable && p >= m.base && bytes <= m.size && p - m.base <= m.size - bytes;
}
