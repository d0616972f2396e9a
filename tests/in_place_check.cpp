// Host check of covers_array (in_place.h): arrays inside their allocation, and ones that reach out of it at either end.
#include <cstdio>
#include "in_place.h"
int main() {
    int bad = 0;
    MemoryAt m;
    m.reachable = true;
    m.base = 1 << 20;
    m.size = 24 * 1000;
    auto check = [&](uintptr_t p, size_t align, size_t bytes, bool want) {
        if (covers_array(m, p, align, bytes) != want && bad++ < 10) printf("%zx %zu %zu\n", (size_t)p, align, bytes);
    };
    check(m.base, 8, 24 * 1000, true);
    check(m.base, 8, 24 * 1000 + 1, false);       // one byte short
    check(m.base + 8, 8, 24 * 1000, false);       // begins later
    check(m.base + 24, 8, 24 * 999, true);
    check(m.base - 8, 8, 16, false);              // begins before
    check(m.base + m.size, 8, 8, false);
    check(m.base + m.size - 8, 8, 8, true);
    check(m.base, 8, ~(size_t)0, false);          // no wrap-around
    check(m.base + 16, 8, ~(size_t)0 - 8, false);
    check(m.base + 4, 8, 8, false);               // alignment
    check(m.base + 4, 4, 8, true);
    check(0, 8, 8, false);
    m.reachable = false;
    check(m.base, 8, 8, false);
    printf("bad %d\n", bad);
    return bad != 0;
}
