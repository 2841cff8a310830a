// csrc/route.cuh without CUDA: every placement that a call may hold, and whether a kernel that the call launches takes it.
#include "../paper_2509_06362_b200/csrc/route.cuh"

using namespace maaso;

static bool launched(const Route& r, const Launches& l, int bucket, uint32_t n) {
    if (r.pack && (bucket == kPack4 || bucket == kPack8)) return l.pack;
    if (bucket < 6) return l.groups;
    if (bucket < kThreadBucket0) return l.blocks;
    if (bucket < kWideBucket) return l.threads;
    if (bucket == kWideBucket) return l.wide_from != 0 && n >= l.wide_from;
    return bucket < kWalkBig0 ? l.walk : (bucket == kWalkBig0 ? l.big : l.far);
}

static Route make_route(uint32_t flags, uint32_t mapping, uint32_t rows, uint32_t models, uint32_t classes, uint64_t items, bool fits32, uint32_t thread_pool,
                        uint32_t thread_hot) {
    Route r = Route();
    r.flags = flags;
    r.mapping = mapping;
    r.n_rows = rows;
    r.n_models = models;
    r.n_classes = classes;
    r.thread_pool_units = thread_pool / 16u;
    r.thread_hot_units = thread_hot / 16u;
    if (mapping == MAASO_MAP_AUTO && !(flags & MAASO_FLAG_TBT_MAXGAP) && !thread_pool) route_walk(r, items, 8u * items, 148u, fits32);
    return r;
}

// Placements without a kernel; the first of them: rows, models, classes, instances, batch cap.
extern "C" uint32_t routes_unscored(uint32_t flags, uint32_t mapping, uint64_t items, uint32_t fits32, uint32_t thread_pool, uint32_t thread_hot, uint32_t* first) {
    const uint32_t classes[] = {1, 2, 3, 4, 71, 128, 176, 177, 208, 209, 255, 256};
    const uint32_t sizes[] = {0, 1, 2, 4, 5, 8, 9, 16, 31, 32, 33, 64, 96, 127, 128}, caps[] = {1, 8, 9, 63, 64};
    uint32_t missing = 0;
    for (uint32_t rows = 1; rows <= MAASO_MAX_ROWS; rows++)
        for (uint32_t models = 1; models <= MAASO_MAX_MODELS; models++) {
            if (rows % models) continue;
            for (uint32_t c : classes) {
                const Route r = make_route(flags, mapping, rows, models, c, items, fits32 != 0, thread_pool, thread_hot);
                for (uint32_t n : sizes) {
                    const Launches l = route_launches(r, n, false);
                    for (uint32_t cap : caps) {
                        PlacementSize s = {n, 0u, 0u, 0u};
                        for (uint32_t i = 0; i < n; i++) s.add(r, i % 32u == 31u ? (cap + 1u) / 2u : cap);
                        const Home h = route_home(r, s);
                        const bool ok = (h.group >= 0 || h.walk >= 0) && (h.group < 0 || launched(r, l, h.group, n)) && (h.walk < 0 || launched(r, l, h.walk, n));
                        if (!ok && missing++ == 0) {
                            const uint32_t f[5] = {rows, models, c, n, cap};
                            for (int i = 0; i < 5; i++) first[i] = f[i];
                        }
                    }
                }
            }
        }
    return missing;
}

// The fewest instances of a placement that goes to the one-warp kernel in a batch of many placements, 0 if that kernel is not launched.
extern "C" uint32_t routes_wide_from(uint32_t flags, uint32_t mapping, uint32_t rows, uint32_t models, uint32_t classes, uint64_t items, uint32_t fits32,
                                     uint32_t thread_pool, uint32_t thread_hot) {
    return route_launches(make_route(flags, mapping, rows, models, classes, items, fits32 != 0, thread_pool, thread_hot), 1u << 20, false).wide_from;
}

// Parts that a placement is replayed in with a queue in front of every instance.
extern "C" uint32_t routes_parts(uint32_t models, uint64_t items, uint64_t insts) {
    Route r = Route();
    r.flags = MAASO_FLAG_INSTANCE_QUEUES;
    r.n_rows = 10u * models;
    r.n_models = models;
    r.n_classes = 3;
    route_walk(r, items, insts, 148u, true);
    return r.walk_parts;
}
