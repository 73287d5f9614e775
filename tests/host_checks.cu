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

// A counter that starts `before` tickets short of the last, drawn on by `warps`
// warps in turn: every ticket is handed out once, and every warp stops.
static int level_ticket_counter()
{
    const uint32_t warps = 4864;
    for (uint32_t tickets : {100u, 4864u, 4865u, 100000u, 0xffffffffu - 9728u, 0xffffffffu - 4864u, 0xfffffffeu}) {
        const uint32_t before = tickets > warps + 10u ? 10u : tickets > warps ? tickets - warps : 0u;
        uint32_t counter = (tickets > warps ? tickets - warps : 0u) - before, served = 0, stopped = 0;
        for (uint32_t draw = 0; draw < before + warps; ++draw) {
            const uint32_t t = warps + counter++;
            if (past_tickets(t, warps, tickets))
                ++stopped;
            else
                ++served;
        }
        EXPECT(served == before && stopped == warps);
    }
    for (uint32_t light : {0u, 1u, 7u, 8u, 9u, 0xfffffff0u, 0xfffffffeu})
        for (uint32_t take : {1u, 2u, 4u, 8u})
            EXPECT(level_tickets(0u, light, take) == ((uint64_t)light + take - 1u) / take);
    return 0;
}

// The leaf counter: every item and the call past the end that each warp makes
// fit 32 bits, or the list is refused; ordinary lists are not.
static int leaf_item_counter()
{
    const uint32_t warps = 4864;
    for (uint32_t leaves : {0u, 1u, 500u, 5000u, 1u << 20, 0x7fffffffu, 0x80000000u, 0xfffff000u, 0xfffffffeu})
        for (uint32_t side : {1u, 16u, 1024u, 65535u, 65536u}) {
            const uint32_t shift = leaf_item_shift(leaves, side, warps);
            const uint64_t items = (uint64_t)leaves << shift;
            EXPECT(leaf_items_fit(leaves, shift, warps) == (items + warps < (1ull << 32)));
            EXPECT(items >= (1ull << 31) || leaf_items_fit(leaves, shift, warps));
            EXPECT(side < 65536u || shift >= 1u);
        }
    return 0;
}

struct Check {
    const char *name;
    int (*fn)();
};
static const Check kChecks[] = {
    {"queue_leaf_entries", queue_leaf_entries},
    {"level_ticket_counter", level_ticket_counter},
    {"leaf_item_counter", leaf_item_counter},
};

int main(int argc, char **argv)
{
    for (const Check &c : kChecks)
        if (argc > 1 && std::strcmp(argv[1], c.name) == 0)
            return c.fn();
    std::printf("no check of that name\n");
    return 2;
}
