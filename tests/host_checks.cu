// Checks of the library's host-side rules that need no GPU: one check per
// name on the command line; a failed one prints its line and exits with 1.
#include <cstdio>
#include <cstring>

#include "ask_internal.h"

using namespace ask;

#define EXPECT(c)                                                   \
    do {                                                            \
        if (!(c)) {                                                 \
            std::printf("%s:%d: %s\n", __FILE__, __LINE__, #c);     \
            return 1;                                               \
        }                                                           \
    } while (0)

// The leaf-list entries of a leaf of the persistent kernel: bands that cover
// its rows once, in order, each of 1 to kQueueLeafPx pixels.
static int queue_leaf_entries()
{
    const uint32_t sides[] = {1, 2, 3, 63, 64, 1000, 1023, 1024, 1025, 32768, 65535, 65536};
    for (uint32_t w : sides)
        for (uint32_t h : sides) {
            const uint32_t rows = queue_leaf_rows(w), nb = queue_leaf_bands(w, h);
            uint64_t next = 0;
            for (uint32_t k = 0; k < nb; ++k) {
                const uint64_t y0 = (uint64_t)k * rows;
                EXPECT(y0 == next && y0 < h);
                const uint32_t bh = h - (uint32_t)y0 < rows ? h - (uint32_t)y0 : rows;
                EXPECT((uint64_t)w * bh >= 1 && (uint64_t)w * bh <= kQueueLeafPx);
                EXPECT(w * bh != 0u);  // the count that the kernel keeps
                next = y0 + bh;
            }
            EXPECT(next == h);
            EXPECT((uint64_t)w * h > kQueueLeafPx || nb == 1u);
        }
    return 0;
}

struct Check {
    const char *name;
    int (*fn)();
};
static const Check kChecks[] = {
    {"queue_leaf_entries", queue_leaf_entries},
};

int main(int argc, char **argv)
{
    for (const Check &c : kChecks)
        if (argc > 1 && std::strcmp(argv[1], c.name) == 0)
            return c.fn();
    std::printf("no check of that name\n");
    return 2;
}
