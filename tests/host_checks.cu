// Checks of the library's host-side rules that need no GPU: one check per
// name on the command line; a failed one prints its line and exits with 1.
//
// The host driver is compiled in with a CUDA runtime of our own in the place
// of the calls below, and with launches that do nothing but record.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

static size_t g_malloc_limit = ~(size_t)0;  // a larger allocation fails
static size_t g_malloc_refused = 0;         // and one of this size
static int g_malloc_failed = 0;
static cudaError_t g_last = cudaSuccess;

template <typename T>
static cudaError_t fake_malloc(T **p, size_t bytes)
{
    if (bytes > g_malloc_limit || bytes == g_malloc_refused) {
        ++g_malloc_failed;
        return g_last = cudaErrorMemoryAllocation;
    }
    *p = static_cast<T *>(std::malloc(bytes < 64 ? bytes : 64));  // never touched
    return cudaSuccess;
}
static cudaError_t fake_free(void *p)
{
    std::free(p);
    return cudaSuccess;
}
static cudaError_t fake_memset(void *, int, size_t) { return cudaSuccess; }
static cudaError_t fake_get_last_error()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
static int g_device = 0, g_occupancy[100], g_occupancy_asked = 0;  // 0: the query fails
static cudaError_t fake_get_device(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
template <typename K>
static cudaError_t fake_occupancy(int *per_sm, K, int, size_t)
{
    ++g_occupancy_asked;
    *per_sm = g_occupancy[g_device];
    return *per_sm ? cudaSuccess : (g_last = cudaErrorInvalidDevice);
}
static cudaError_t g_launch = cudaSuccess;
template <typename... A>
static cudaError_t fake_launch(const cudaLaunchConfig_t *, A...)
{
    if (g_launch != cudaSuccess)
        g_last = g_launch;
    return g_launch;
}
#define cudaLaunchKernelEx fake_launch
#define cudaGetDevice fake_get_device
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_occupancy
#define cudaMalloc fake_malloc
#define cudaFree fake_free
#define cudaMemset fake_memset
#define cudaGetLastError fake_get_last_error

#include "ask_api.cu"
#include "ask_launch.cuh"

namespace ask {
static LeafArgs g_leaf;  // of the last leaf launch
#define RECORDS_NOTHING(name, ...) \
    cudaError_t name(__VA_ARGS__) { return cudaSuccess; }
RECORDS_NOTHING(launch_exhaustive, uint32_t *, uint32_t, PixelMap, uint32_t, uint32_t, uint32_t, bool,
                DevCounters *, cudaStream_t)
RECORDS_NOTHING(launch_init, uint2 *, uint4 *, DevCounters *, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t,
                cudaStream_t, const PixelMap *)
RECORDS_NOTHING(launch_init_batch, uint4 *, uint4 *, DevCounters *, const FrameDesc *, uint32_t, uint32_t,
                cudaStream_t)
RECORDS_NOTHING(launch_level, const LevelArgs &, bool, bool, int, cudaStream_t)
RECORDS_NOTHING(launch_fill, const FillArgs &, bool, int, cudaStream_t)
RECORDS_NOTHING(launch_queue, const QueueArgs &, uint32_t, bool, int, cudaStream_t)
RECORDS_NOTHING(launch_cdp2, const CdpArgs &, uint32_t, uint32_t, uint32_t, uint32_t, cudaStream_t)
RECORDS_NOTHING(cdp2_set_pending_limit, size_t)
RECORDS_NOTHING(launch_level_region, const LevelArgs &, bool, bool, uint32_t, int, cudaStream_t)
RECORDS_NOTHING(launch_leaf_region, const LeafArgs &, uint32_t, uint32_t, bool, int, cudaStream_t)
RECORDS_NOTHING(launch_exhaustive64, uint32_t *, uint32_t, PixelMap64, uint32_t, uint32_t, uint32_t, bool, bool,
                DevCounters *, cudaStream_t)
RECORDS_NOTHING(launch_level64, const Level64Args &, bool, bool, int, cudaStream_t)
RECORDS_NOTHING(launch_leaf64, const Leaf64Args &, bool, bool, int, cudaStream_t)
cudaError_t launch_leaf(const LeafArgs &a, uint32_t, uint32_t, bool, bool, bool, int, cudaStream_t)
{
    g_leaf = a;
    return cudaSuccess;
}
}  // namespace ask

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

// A small batch on a device with no memory left for its survivor pool renders
// without one, and with one once a smaller batch's fits.
static int pool_does_not_fit()
{
    alignas(16) static uint32_t map[4];
    const ask_frame big = {{-1.5f, 0.5f, -1.0f, 1.0f}, 1500, 100, 8, 2, 32, 0, map};
    const ask_frame small = {{-1.5f, 0.5f, -1.0f, 1.0f}, 300, 100, 2, 2, 32, 0, map};
    ask_ctx ctx{};
    ctx.dev.sms = 152;
    BatchBuffers b;
    BatchPlan bp, bq;
    uint32_t launches = 0, with = 0;
    EXPECT(plan_batch(&ctx, &big, 1, 0, 0, bp) == ASK_OK && pool_need(bp.pixels) == 1500u * 1500u);
    EXPECT(plan_batch(&ctx, &small, 1, 0, 0, bq) == ASK_OK && pool_need(bq.pixels) == 300u * 300u);
    for (size_t entry : {sizeof(float4), sizeof(uint32_t)}) {
        g_malloc_refused = 1500 * 1500 * entry;
        g_malloc_failed = 0;
        for (int k = 0; k < 2; ++k) {  // the second call does not ask again
            EXPECT(reserve_batch(&ctx, b, bp, true) == ASK_OK);
            EXPECT(g_malloc_failed == 1 && g_last == cudaSuccess && ctx.err[0] == 0);
            EXPECT(enqueue_batch(&ctx, b, bp, 0, nullptr, &launches) == ASK_OK);
            EXPECT(g_leaf.pool == nullptr && g_leaf.pool_frame == nullptr && g_leaf.pool_cap == 0);
        }
        EXPECT(reserve_batch(&ctx, b, bq, true) == ASK_OK);
        EXPECT(enqueue_batch(&ctx, b, bq, 0, nullptr, &with) == ASK_OK);
        EXPECT(g_leaf.pool != nullptr && g_leaf.pool_frame != nullptr && g_leaf.pool_cap == 300u * 300u);
        EXPECT(enqueue_batch(&ctx, b, bp, 0, nullptr, &launches) == ASK_OK && g_leaf.pool == nullptr);
        free_batch(b, true);
    }
    g_malloc_refused = 0;
    // memory that the batch cannot do without is an error as ever
    g_malloc_limit = 64;
    EXPECT(reserve_batch(&ctx, b, bp, true) == ASK_ENOMEM);
    free_batch(b, true);
    // with memory enough
    g_malloc_limit = ~(size_t)0;
    EXPECT(reserve_batch(&ctx, b, bp, true) == ASK_OK);
    EXPECT(enqueue_batch(&ctx, b, bp, 0, nullptr, &with) == ASK_OK);
    EXPECT(g_leaf.pool == b.pool && g_leaf.pool_cap == 1500u * 1500u && with == launches + 1u);
    free_batch(b, true);
    return 0;
}

// Occupancy is each device's own, asked once, and a failed query is not kept.
static int occupancy_by_device()
{
    static PerDevice known;
    auto ask = [&](int dev) {
        g_device = dev;
        return resident_ctas((void (*)())nullptr, 256, 0, &known);
    };
    g_occupancy[0] = 3;
    g_occupancy[1] = 5;
    g_occupancy[99] = 7;  // beyond those whose answers are kept
    EXPECT(ask(0) == 3 && ask(1) == 5 && ask(0) == 3 && ask(1) == 5 && g_occupancy_asked == 2);
    EXPECT(ask(99) == 7 && ask(99) == 7);
    EXPECT(ask(2) == 1 && g_last == cudaSuccess);  // fails
    g_occupancy[2] = 4;
    EXPECT(ask(2) == 4);
    g_occupancy[2] = 0;
    EXPECT(ask(2) == 4);
    g_device = 0;
    EXPECT(resident_ctas((void (*)())nullptr, 256, 0) == 3);
    return 0;
}

// A refused launch is reported by its own return value and leaves no error
// behind; one that went well leaves an error of before alone.
static int chained_launch_error()
{
    g_last = cudaErrorInvalidValue;
    EXPECT(launch_chained((void (*)())nullptr, 1, 32, 0, nullptr) == cudaSuccess && g_last == cudaErrorInvalidValue);
    g_launch = cudaErrorLaunchOutOfResources;
    EXPECT(launch_chained((void (*)())nullptr, 1, 32, 0, nullptr) == cudaErrorLaunchOutOfResources);
    EXPECT(g_last == cudaSuccess);
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
    {"pool_does_not_fit", pool_does_not_fit},
    {"occupancy_by_device", occupancy_by_device},
    {"chained_launch_error", chained_launch_error},
};

int main(int argc, char **argv)
{
    for (const Check &c : kChecks)
        if (argc > 1 && std::strcmp(argv[1], c.name) == 0)
            return c.fn();
    std::printf("no check of that name\n");
    return 2;
}
