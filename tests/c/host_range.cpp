// range_holds over the cases around the ends of an allocation, and over ranges
// whose sums wrap.
#include "host_range.h"

#include <cstdio>

using gdag::range_holds;

int main()
{
    int bad = 0;
    auto is = [&](bool got, bool want, const char *what) {
        if (got != want) {
            std::printf("%s: %d\n", what, got);
            ++bad;
        }
    };
    const uint64_t a = 0x10000, n = 0x1000, top = ~0ull;
    is(range_holds(a, n, a, n), true, "all of it");
    is(range_holds(a, n, a, 1), true, "first byte");
    is(range_holds(a, n, a + n - 1, 1), true, "last byte");
    is(range_holds(a, n, a + 1, n - 2), true, "inside");
    is(range_holds(a, n, a, n + 1), false, "one byte past the end");
    is(range_holds(a, n, a + n - 1, 2), false, "last byte and the next");
    is(range_holds(a, n, a - 1, 2), false, "from before the start");
    is(range_holds(a, n, a - 1, n + 2), false, "around it");
    is(range_holds(a, n, a + n, 1), false, "right after it");
    is(range_holds(a, n, a + 2 * n, 1), false, "beyond");
    is(range_holds(a, n, a + 1, top), false, "a size that wraps");
    is(range_holds(0, 0, a, 1), false, "no allocation");
    is(range_holds(top - n, n, top - 1, 1), true, "at the top");
    is(range_holds(top - n, n, top - 1, 2), false, "past the top");
    return bad;
}
