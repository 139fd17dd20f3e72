// Check of the range test that decides whether the batch's export kernel may
// write a result buffer (store.h): exact fits, one byte more, both sides of
// the allocation, an unknown allocation, and sizes that wrap around.
#include <cstdio>

#include "store.h"

using admm_impl::range_holds;

#define CHECK(c)                                                        \
    do {                                                                \
        if (!(c)) {                                                     \
            std::fprintf(stderr, "check failed line %d: %s\n", __LINE__, #c); \
            return 1;                                                   \
        }                                                               \
    } while (0)

int main()
{
    const uintptr_t base = 0x7f0000000000ull, top = ~(uintptr_t)0;
    const size_t size = 4096, most = ~(size_t)0;
    CHECK(range_holds(base, size, base, size));
    CHECK(range_holds(base, size, base + 8, size - 8));
    CHECK(range_holds(base, size, base + size - 8, 8));
    CHECK(range_holds(base, size, base + size, 0));
    CHECK(!range_holds(base, size, base, size + 1));
    CHECK(!range_holds(base, size, base + 8, size));
    CHECK(!range_holds(base, size, base + size, 8));
    CHECK(!range_holds(base, size, base + size + 8, 0));
    CHECK(!range_holds(base, size, base - 8, 16));
    CHECK(!range_holds(0, 0, base, 8));
    CHECK(!range_holds(base, size, base + 8, most));
    CHECK(!range_holds(base, size, base + 8, most - 7));
    CHECK(!range_holds(top - 4095, 4096, top - 7, 16));
    CHECK(range_holds(top - 4095, 4096, top - 7, 8));
    std::puts("ranges ok");
    return 0;
}
