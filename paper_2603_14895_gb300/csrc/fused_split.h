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

// bucket_start[b], b = 0..32: rows with 2^b in-arcs and more; cap: CTAs that fit at once in a
// launch per step, run_cap: in the kernel that will run; the others: rows (times nslices work
// items each) of a class per CTA.
//
// The rows of 2^b in-arcs and more get a warp each (16-bit counters), the others a team
// (counters of team_bits).  A small graph's step lasts as long as its longest chain of
// gathers, so b is the smallest bound for which the warp rows take at most half of the warps
// that fit at once (60 graphs of 8k to 1M words: 1.16 times faster on average than all of
// them, as fast as a quarter), and at most team_bits.  Where all rows are short (below 64
// in-arcs), a larger b that saves a round of CTAs is worth more than the shorter chains of
// warp rows (T = 40, us, before and so: ER n = 9k, R = 256, SIR 784 and 597; n = 19k, R = 142, SIS
// 1076 and 812, IC 1007 and 750; n = 3k, three sets of R = 221, LT 827 and 632).
//
// Two cases go by an estimate of a step's time, in rounds of eight gathered arcs: six per
// round of rows, and the longest row of each round (rows come in descending degree).
// - Rows of 2^team_bits in-arcs, which only a warp can take, want more than half of the CTAs,
//   and the two classes together more than there are: the warp rows get the CTAs of a whole
//   number of rounds, the one with the earliest end.  (Given every CTA but one, they leave the
//   team rows of an R-MAT graph to a single CTA: 20 steps, ms, so and now: SIR, n = 524k, R = 64:
//   217 and 3.3; weighted 581 and 6.7; SIS, n = 262k, R = 128: 216 and 3.7; ER, n = 10k, mean degree
//   256, R = 100: 16.5 and 0.66; every row a warp, in those cases: 12.7, 11.2, 10.9 and 0.89.)
// - Every row a warp ends at least a fifth earlier: dense graphs, where a team's chain is long
//   (30 steps, us, before and so: ER n = 2000, mean degree 200, R = 64, SIS 1078 and 619, IC 1767 and
//   562; n = 5000, 150, R = 64, SIS 928 and 792; n = 5000, 256, R = 200, SIS 1826 and 1109, when the
//   first case's condition counted the CTAs of a launch per step).
inline FusedSplit fused_split(const int32_t *bucket_start, int32_t n, int32_t max_deg, int nslices,
                              int64_t cap, int64_t run_cap, int warp_rows_per_cta, int team_rows_per_cta, int team_bits) {
    FusedSplit f{};
    auto warp_rows = [&](int b) { return b == 0 ? n : bucket_start[b]; };
    auto ctas = [&](int64_t rows, int per_cta) { return (rows * nslices + per_cta - 1) / per_cta; };
    auto rounds = [&](int b) {
        return (ctas(warp_rows(b), warp_rows_per_cta) + ctas(n - warp_rows(b), team_rows_per_cta) + run_cap - 1) / run_cap;
    };
    int b = 0;
    while (b < team_bits && 2 * (int64_t)bucket_start[b] * nslices > cap * warp_rows_per_cta) ++b;
    if (max_deg < 64)
        for (int c = b + 1; c <= team_bits; ++c)
            if (rounds(c) < rounds(b)) b = c;
    // estimated end of rows [r0, r1) of at most `longest` arcs on g CTAs, `teams` of whose
    // teams share a row
    auto ends = [&](int32_t r0, int32_t r1, int32_t longest, int64_t g, int per_cta, double teams) {
        if (r1 <= r0) return 0.0;
        const double per_round = std::max(1.0, (double)g * per_cta / nslices);   // rows
        double arcs = 0.0;   // of rows at their bucket's bound
        for (int k = 1; k <= 32; ++k) {
            const int32_t lo = std::max(r0, bucket_start[k]), hi = std::min(r1, bucket_start[k - 1]);
            if (hi > lo) arcs += (double)(hi - lo) * (double)std::min<int64_t>(((int64_t)1 << k) - 1, longest);
        }
        const double rnd = (double)((ctas(r1 - r0, per_cta) + g - 1) / g);
        return 6.0 * rnd + (longest + (rnd > 1.0 ? arcs / per_round : 0.0)) / (8.0 * teams);
    };
    const double teams = (double)team_rows_per_cta / warp_rows_per_cta;   // of a warp
    auto time = [&](int32_t w, int32_t team_longest, int64_t mid, int64_t small) {
        return std::max(ends(0, w, max_deg, mid, warp_rows_per_cta, teams), ends(w, n, team_longest, small, team_rows_per_cta, 1.0));
    };
    f.warp_rows = warp_rows(b);
    const int32_t team_rows = n - f.warp_rows;
    const int32_t team_longest = (int32_t)std::min<int64_t>(max_deg, ((int64_t)1 << b) - 1);
    const int64_t want_mid = ctas(f.warp_rows, warp_rows_per_cta), want_small = ctas(team_rows, team_rows_per_cta);
    int64_t mid = want_mid;
    double end;
    if (b == team_bits && 2 * want_mid > cap && want_mid + want_small > run_cap && team_rows > 0) {
        cap = run_cap;
        end = 1e300;
        for (int64_t r = 1; r <= want_mid; ++r) {
            const int64_t m = std::min((want_mid + r - 1) / r, std::max<int64_t>(cap - 1, 1));
            const double t = time(f.warp_rows, team_longest, m, std::max<int64_t>(1, std::min(want_small, cap - m)));
            if (t < end) {
                end = t;
                mid = m;
            }
            if (m == 1 || ends(0, f.warp_rows, max_deg, m, warp_rows_per_cta, teams) > end) break;
        }
    } else {
        mid = std::min(mid, team_rows > 0 ? std::max<int64_t>(cap - 1, 1) : cap);
        const int64_t small = std::min(want_small, std::max<int64_t>(cap - mid, 1));
        const double scale = std::min(1.0, (double)run_cap / (double)(mid + small));   // (the persistent loop's grid)
        end = time(f.warp_rows, team_longest, std::max<int64_t>(1, (int64_t)(scale * mid)),
                   std::max<int64_t>(1, (int64_t)(scale * small)));
    }
    const int64_t all = std::min(ctas(n, warp_rows_per_cta), cap);
    if (team_rows > 0 && 5.0 * time(n, 0, std::min(all, run_cap), 0) < 4.0 * end) {
        f.warp_rows = n;
        f.grid_mid = (int)all;
        return f;
    }
    mid = std::min(mid, team_rows > 0 ? std::max<int64_t>(cap - 1, 1) : cap);
    f.grid_mid = (int)mid;
    f.grid_small = (int)std::min(want_small, std::max<int64_t>(cap - mid, 1));
    return f;
}

}  // namespace fsgp
