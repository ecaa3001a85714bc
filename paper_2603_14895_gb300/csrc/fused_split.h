// fused_split.h -- how a small graph's step is shared out between its two row classes
// (host code).
#pragma once

#include <stdint.h>

#include <algorithm>

namespace fsgp {

struct FusedSplit {
    int32_t warp_rows;          // rows that get a warp each: the first of the degree order
    int grid_mid, grid_small;   // CTAs on the warp rows and on the team rows (either may be 0)
};

// bucket_start[b]: rows with 2^b in-arcs and more, for b <= team_bits; cap: CTAs that fit at
// once; the others: rows (times nslices work items each) of a class per CTA.
//
// The rows of 2^b in-arcs and more get a warp each (16-bit counters), the others a team
// (counters of team_bits).  A small graph's step lasts as long as its longest chain of
// gathers, so b is the smallest bound for which the warp rows take at most half of the warps
// that fit at once (60 graphs of 8k to 1M words: 1.16 times faster on average than all of
// them, as fast as a quarter), and at most team_bits.
//
// Where the rows of 2^team_bits in-arcs, which only a warp can take, want more than half of
// the CTAs, and the two classes together more than there are, the CTAs go by work: arcs, and
// 16 per row for its words.  (Given every CTA but one, the warp rows leave the team rows of an
// R-MAT graph to a single CTA.  20 steps, ms, so and now: SIR, n = 524k, R = 64: 217 and 2.5;
// weighted 582 and 4.6; SIS, n = 262k, R = 128: 216 and 4.2; ER, n = 10k, mean degree 256,
// R = 100: 16.5 and 0.86; every row a warp, in those cases: 12.7, 11.2, 10.9 and 0.89.)
inline FusedSplit fused_split(const int32_t *bucket_start, int32_t n, int64_t nnz, int nslices, int64_t cap,
                              int warp_rows_per_cta, int team_rows_per_cta, int team_bits) {
    FusedSplit f{};
    int b = 0;
    while (b < team_bits && 2 * (int64_t)bucket_start[b] * nslices > cap * warp_rows_per_cta) ++b;
    f.warp_rows = b == 0 ? n : bucket_start[b];
    const int32_t team_rows = n - f.warp_rows;
    const int64_t want_mid = ((int64_t)f.warp_rows * nslices + warp_rows_per_cta - 1) / warp_rows_per_cta;
    const int64_t want_small = ((int64_t)team_rows * nslices + team_rows_per_cta - 1) / team_rows_per_cta;
    int64_t mid = want_mid;
    if (b == team_bits && 2 * want_mid > cap && want_mid + want_small > cap && team_rows > 0) {
        double team = 0.0;   // arcs of the team rows: 3/4 of their bucket's bound each
        for (int i = 1; i <= b; ++i)
            team += 0.75 * (double)((int64_t)1 << i) * (double)(bucket_start[i - 1] - bucket_start[i]);
        const double warp = std::max((double)nnz - team, (double)f.warp_rows * (double)((int64_t)1 << b)) + 16.0 * f.warp_rows;
        team += 16.0 * team_rows;
        mid = std::min(want_mid, std::max<int64_t>(1, (int64_t)((double)cap * warp / (warp + team))));
    }
    mid = std::min(mid, team_rows > 0 ? std::max<int64_t>(cap - 1, 1) : cap);
    f.grid_mid = (int)mid;
    f.grid_small = (int)std::min(want_small, std::max<int64_t>(cap - mid, 1));
    return f;
}

}  // namespace fsgp
