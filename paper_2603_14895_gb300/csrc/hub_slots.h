// hub_slots.h -- the hub chunk tables a graph keeps (host code, no CUDA calls of its own).
#pragma once

#include <stdint.h>

#include <algorithm>

namespace fsgp {

struct HubTable {
    int32_t min_deg = -1;       // table built for this hub threshold and chunk size (-1: no table)
    int32_t chunk = -1;
    int32_t n_hubs = 0;
    int64_t n_chunks = 0;
    int64_t *d_chunk_base = nullptr;  // [n_hubs + 1] (hub rows are new ids 0 .. n_hubs-1)
};

// The table of (min_deg, chunk): a kept one, or one that build(table) makes in the place of
// the one used longest ago, which drop(table) releases.  Two are kept: models with different
// chunks may alternate.  A run without hub rows takes an empty table and leaves the kept ones
// alone.  A slot carries its key only while its table is whole, so that a build that failed
// is tried again.
template <class Drop, class Build>
int hub_slot(HubTable (&slots)[2], int32_t min_deg, int32_t chunk, int32_t n_hubs, Drop drop, Build build,
             const HubTable **out) {
    static const HubTable none{};
    *out = &none;
    if (n_hubs == 0) return 0;
    HubTable &oldest = slots[0], &newest = slots[1];
    if (oldest.min_deg == min_deg && oldest.chunk == chunk) std::swap(oldest, newest);
    if (newest.min_deg != min_deg || newest.chunk != chunk) {
        drop(oldest);
        oldest = HubTable{};
        oldest.n_hubs = n_hubs;
        const int rc = build(oldest);
        if (rc) {
            drop(oldest);
            oldest = HubTable{};
            return rc;
        }
        oldest.min_deg = min_deg;
        oldest.chunk = chunk;
        std::swap(oldest, newest);
    }
    *out = &newest;
    return 0;
}

}  // namespace fsgp
