// rows.cuh -- the row kernels of one propagation step (gather + count + decide + write),
// templated on the model, the words per thread V and the team width TEAM.  Included by
// one translation unit per model so that the instantiations compile in parallel.
#pragma once

#include <algorithm>
#include <atomic>

#include "step.cuh"
#include "tile.cuh"

namespace fsgp {

template <int V>
struct Vec {
    uint32_t w[V];
};

template <int V>
__device__ __forceinline__ Vec<V> ldg_vec(const uint32_t *p) {
    Vec<V> r;
    if constexpr (V == 4) {
        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p));
        r.w[0] = q.x; r.w[1] = q.y; r.w[2] = q.z; r.w[3] = q.w;
    } else if constexpr (V == 2) {
        const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
        r.w[0] = q.x; r.w[1] = q.y;
    } else {
        r.w[0] = __ldg(p);
    }
    return r;
}

// State loads of a kernel that reads planes written earlier in the same launch (the
// persistent step loop): through L2 only (ld.global.cg), never the non-coherent path.
template <int V, bool CG>
__device__ __forceinline__ Vec<V> ld_vec(const uint32_t *p) {
    if constexpr (!CG) {
        return ldg_vec<V>(p);
    } else {
        Vec<V> r;
        if constexpr (V == 4) {
            const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(p));
            r.w[0] = q.x; r.w[1] = q.y; r.w[2] = q.z; r.w[3] = q.w;
        } else if constexpr (V == 2) {
            const uint2 q = __ldcg(reinterpret_cast<const uint2 *>(p));
            r.w[0] = q.x; r.w[1] = q.y;
        } else {
            r.w[0] = __ldcg(p);
        }
        return r;
    }
}

template <bool CG>
__device__ __forceinline__ uint32_t ld_word(const uint32_t *p) {
    if constexpr (CG) return __ldcg(p);
    else return __ldg(p);
}

template <int V>
__device__ __forceinline__ void st_vec(uint32_t *p, const uint32_t (&w)[V]) {
    if constexpr (V == 4) {
        *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    } else if constexpr (V == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
    } else {
        *p = w[0];
    }
}

template <int MODEL>
struct ModelTraits {
    // SIR: I, R.  SIS: I.  IC, LT: A, F.  SEIR: I, R, E.  SEIS: I, E.  SWIR: I, R, W.
    // Weighted SIR / SIS: as SIR / SIS.
    static constexpr int planes = (MODEL == FSGP_SIS || MODEL == kSisW)
                                      ? 1
                                      : ((MODEL == FSGP_SEIR || MODEL == FSGP_SWIR) ? 3 : 2);
    // plane gathered from in-neighbours: I (epidemic models), F (IC), A (LT)
    static constexpr int src_plane = MODEL == FSGP_IC ? 1 : 0;
    // per-arc draws (live-lane masks) instead of in-arc counts: IC and weighted graphs
    static constexpr bool weighted = MODEL == kSirW || MODEL == kSisW;
    static constexpr bool counts = MODEL != FSGP_IC && !weighted;
    // the state's source lanes are plane 1 (F) for IC / LT, plane 0 (I) otherwise
    static constexpr bool cascade = MODEL == FSGP_IC || MODEL == FSGP_LT;
    // hub rows may stop reading once every susceptible lane reaches K_sat
    static constexpr bool saturates = MODEL == FSGP_SIR || MODEL == FSGP_SIS || MODEL == FSGP_SEIR ||
                                      MODEL == FSGP_SEIS;
    // words decided through the warp tile (SWIR's second draw depends on its first one and
    // stays on the per-thread update)
    static constexpr bool tiled = MODEL != FSGP_SWIR;
    // fixed-threshold draws per word: recovery, and the latent exit of SEIR / SEIS
    static constexpr int fixed_draws = (MODEL == FSGP_SEIR || MODEL == FSGP_SEIS) ? 2 : (cascade ? 0 : 1);
};

// Lanes that can change through their in-arcs: susceptible (SWIR: also weakened) or
// inactive lanes.
template <int MODEL>
__device__ __forceinline__ uint32_t need_of(uint32_t vm, uint32_t s0, uint32_t s1, uint32_t s2) {
    if constexpr (MODEL == FSGP_SIR || MODEL == kSirW || MODEL == FSGP_SEIS || MODEL == FSGP_SWIR)
        return vm & ~s0 & ~s1;
    else if constexpr (MODEL == FSGP_SEIR) return vm & ~s0 & ~s1 & ~s2;
    else return vm & ~s0;
}

// One word of the synchronous update (Eq. updata) from the in-arc counts c (IC: the
// lanes made active by a live arc, `newly`).
template <int MODEL, int B>
__device__ __forceinline__ WordOut update_word(const StepArgs &A, uint32_t node, const WordCtx &x, uint32_t s0,
                                               uint32_t s1, uint32_t s2, int32_t d, const uint32_t (&c)[B],
                                               uint32_t newly) {
    WordOut o;
    if constexpr (MODEL == FSGP_SIR || MODEL == FSGP_SIS) {
        o = update_sir_word<MODEL, B>(A, node, x, s0, s1, d, c);
    } else if constexpr (MODEL == FSGP_IC) {
        o.n0 = s0 | newly;
        o.n1 = newly;
        o.n2 = 0u;
    } else if constexpr (ModelTraits<MODEL>::weighted) {
        // infected: a susceptible lane some infectious in-arc transmitted to; recovery
        // as in SIR / SIS
        const uint32_t infect = newly & need_of<MODEL>(x.vm, s0, s1, 0u);
        const uint32_t rec = lanes_u_less(s0 & x.vm, __ldg(&A.sp[x.s].g_rec), node, A.t, x.g, TAG_RECOVER,
                                          x.k0, x.k1);
        o.n0 = (s0 & ~rec) | infect;
        o.n1 = MODEL == kSirW ? (s1 | rec) : 0u;
        o.n2 = 0u;
    } else if constexpr (MODEL == FSGP_LT) {
        o = update_lt_word<B>(A, node, x, s0, d, c);
    } else if constexpr (MODEL == FSGP_SWIR) {
        o = update_swir_word<B>(A, node, x, s0, s1, s2, d, c);
    } else {
        o = update_seir_word<MODEL, B>(A, node, x, s0, s1, s2, d, c);
    }
    return o;
}

// Row flags of a decided word: bit 0 the new state has source lanes (its out-neighbours
// are pressed next step), bit 1 the row changed or can change on its own next step
// (an exposed lane: SEIR / SEIS).
template <int MODEL>
__device__ __forceinline__ uint32_t word_flags(const WordOut &o, uint32_t s0, uint32_t s1, uint32_t s2) {
    uint32_t fl = 0u;
    if (o.n0 != s0 || o.n1 != s1 || o.n2 != s2) fl |= 2u;
    if (ModelTraits<MODEL>::cascade ? (o.n1 != 0u) : (o.n0 != 0u)) fl |= 1u;
    if constexpr (MODEL == FSGP_SEIR) if (o.n2) fl |= 2u;
    if constexpr (MODEL == FSGP_SEIS) if (o.n1) fl |= 2u;
    return fl;
}

// IC live-arc threshold of a word: weighted cascade (live iff u * d < 2^32, i.e.
// u < floor((2^32 - 1) / d) + 1) or the set's constant probability.
__device__ __forceinline__ uint64_t ic_threshold(const StepArgs &A, int s, int32_t d) {
    if (A.ic_mode == FSGP_IC_WEIGHTED_CASCADE) return d > 0 ? (TWO32 - 1ull) / (uint64_t)d + 1ull : 0ull;
    return __ldg(&A.sp[s].p_const);
}

// Gather the `rem` in-arcs at col[first ..] of a row into bit-sliced counters (count
// models; rem <= 0: none).  PARTS teams of the warp share the row and take 8 arcs each per
// round, the rounds `step` arcs apart (8 * PARTS when nobody else works on the row).  The
// next round's column indices are loaded while the state words of this one are in flight.
//   One team per row: its lanes load the round's indices side by side and hand them out by
//   shuffles (a load per arc and thread would touch one cache line per row of the warp for
//   every arc); every lane of the warp takes part until no row has arcs left.
//   Several teams per row: the indices the warp needs lie in two or three lines anyway, and
//   the plain loads are cheaper than the shuffles (rows of 256 to 8191 arcs, R-MAT, SIS,
//   R = 256: 0.36 against 0.46 ms per step at n = 8M).
template <int MODEL, int V, int B, int TEAM, int PARTS, bool CG = false>
__device__ __forceinline__ void gather_counts(const StepArgs &A, int64_t first, int32_t rem, int32_t step, int w0,
                                              int lane, uint32_t (&c)[V][B]) {
    const uint32_t *src = A.cur + (size_t)ModelTraits<MODEL>::src_plane * A.plane_words + w0;
    const uint32_t Wn = (uint32_t)A.Wn;
    if constexpr (PARTS == 1 && TEAM > 1) {
        constexpr int NQ = TEAM >= 8 ? 1 : 8 / TEAM;  // indices each lane of the team loads
        const int tl = lane % TEAM, g0 = lane - tl;
        const int32_t *cp = A.col + first + tl;
        const bool loads = TEAM <= 8 || tl < 8;
        int32_t mine[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) mine[q] = loads && q * TEAM + tl < rem ? __ldg(cp + q * TEAM) : -1;
        while (__any_sync(0xffffffffu, rem > 0)) {
            Vec<V> xs[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int32_t u = __shfl_sync(0xffffffffu, mine[TEAM >= 8 ? 0 : j / TEAM], g0 + (TEAM >= 8 ? j : j % TEAM));
                xs[j] = Vec<V>{};
                if (u >= 0) xs[j] = ld_vec<V, CG>(src + (uint64_t)(uint32_t)u * Wn);
            }
            cp += step;
            rem -= step;
#pragma unroll
            for (int q = 0; q < NQ; ++q) mine[q] = loads && q * TEAM + tl < rem ? __ldg(cp + q * TEAM) : -1;
#pragma unroll
            for (int i = 0; i < V; ++i)
                add8<B>(c[i], xs[0].w[i], xs[1].w[i], xs[2].w[i], xs[3].w[i], xs[4].w[i], xs[5].w[i], xs[6].w[i],
                        xs[7].w[i]);
        }
    } else {
        const int part = lane / TEAM % PARTS;
        const int32_t *cp = A.col + first + 8 * part;
        rem -= 8 * part;
        int32_t u[8];
        if (rem >= 8) {
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = __ldg(cp + j);
        }
        while (rem >= 8) {
            Vec<V> xs[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) xs[j] = ld_vec<V, CG>(src + (uint64_t)(uint32_t)u[j] * Wn);
            cp += step;
            rem -= step;
            if (rem >= 8) {
#pragma unroll
                for (int j = 0; j < 8; ++j) u[j] = __ldg(cp + j);
            }
#pragma unroll
            for (int i = 0; i < V; ++i)
                add8<B>(c[i], xs[0].w[i], xs[1].w[i], xs[2].w[i], xs[3].w[i], xs[4].w[i], xs[5].w[i], xs[6].w[i],
                        xs[7].w[i]);
        }
        // the row's last, partial group
#pragma unroll 1
        for (; rem > 0; rem -= 4, cp += 4) {
            Vec<V> xs[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                xs[j] = Vec<V>{};
                if (j < rem) xs[j] = ld_vec<V, CG>(src + (uint64_t)(uint32_t)__ldg(cp + j) * Wn);
            }
#pragma unroll
            for (int i = 0; i < V; ++i) add4<B>(c[i], xs[0].w[i], xs[1].w[i], xs[2].w[i], xs[3].w[i]);
        }
        __syncwarp();
    }
}

// Gather the in-arcs [e_begin, e_end) with stride `step` (groups of 4 consecutive arcs)
// into live-lane masks (IC, weighted graphs).  Software pipelined like
// gather_counts.
// Draws are keyed by the arc's position in the caller's column array: arc e of the
// relabelled array is caller arc e + arcb.
template <int MODEL, int V>
__device__ __forceinline__ void gather_arcs(const StepArgs &A, int64_t e_begin, int64_t e_end,
                                            int64_t step, int64_t arcb, int w0, const uint32_t (&need)[V],
                                            const uint64_t (&ic_thr)[V], const WordCtx (&x)[V],
                                            uint32_t (&newly)[V]) {
    const uint32_t *src = A.cur + (size_t)ModelTraits<MODEL>::src_plane * A.plane_words + w0;
    const size_t Wn = (size_t)A.Wn;
    int32_t u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = e_begin + j < e_end ? __ldg(A.col + e_begin + j) : -1;
    for (int64_t e = e_begin; e < e_end; e += step) {
        Vec<V> xs[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            xs[j] = Vec<V>{};
            if (u[j] >= 0) xs[j] = ldg_vec<V>(src + (size_t)u[j] * Wn);
        }
        const int64_t en = e + step;
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = en + j < e_end ? __ldg(A.col + en + j) : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const uint32_t m = xs[j].w[i] & need[i] & ~newly[i];
                if (m) {
                    constexpr bool W = ModelTraits<MODEL>::weighted;
                    const int64_t ep = e + j + arcb;   // the caller's arc position
                    const uint64_t thr = W ? arc_threshold(A, x[i].s, ep) : ic_thr[i];
                    newly[i] |= lanes_u_less(m, thr, (uint32_t)ep, A.t, x[i].g, W ? TAG_ARC_INFECT : TAG_IC_EDGE,
                                             x[i].k0, x[i].k1);
                }
            }
        }
    }
}

// Counter plane b of word i of a thread's V words, by selects (i is not a compile-time
// constant where this is used; indexing the array with it would move it to local memory).
template <int V, int B>
__device__ __forceinline__ uint32_t pick(const uint32_t (&c)[V][B], int i, int b) {
    uint32_t r = c[0][b];
#pragma unroll
    for (int q = 1; q < V; ++q) r = i == q ? c[q][b] : r;
    return r;
}

// Resident CTAs per SM the register allocation is bounded for: wider thread words hold
// more counters.  Three with one and two words per thread: their 80 registers hold the team
// rows but for 4 to 36 bytes of spill stores, the warp rows with 16 counter planes per word
// but for 28 to 104 (SIS and SIR); a fourth leaves 64 registers (R-MAT n = 8M, R = 256, a SIS
// step with two words: team rows 602 us with four, 541 with three, 669 with five; warp rows 333
// with three, 377 with two, 586 with four.  One word, R = 32, T = 40, ms with three, four,
// five: SIS, R-MAT n = 4.2M 24.6, 26.2, 28.1; LT 28.3, 29.5, 34.2; SIR, BA n = 2M 10.7, 11.1,
// 13.5).
template <int V>
constexpr int min_ctas() { return V == 4 ? 2 : 3; }

// Row kernel that decides every word in the thread that gathered it (SWIR, whose second draw
// depends on its first): one work item is one slice (TEAM*V words) of one row.
// WARP_ROW = false: one team per item; true: one warp per item.
// BT: counter bits of a team kernel, sized to its rows' in-degree bound (fewer planes =
// fewer registers and cheaper counting and grouping).
// which: 0 = small rows with 16..small_max in-arcs (and every small row of a frontier
// step), 1 = mid rows, 3 = rows with 4..15 in-arcs (dense steps only).
// CG: the state planes are read through L2 only (the persistent step loop, which reads
// in one launch the planes that other CTAs wrote at the previous step).
// B: counter bits.  AG: teams that share a team row's arcs.
// bid of nb: the CTA's place among those that work on these rows.
template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT, bool CG, int B, int AG>
__device__ __forceinline__ void rows_body(const StepArgs &A, int which, int32_t *s_lane, unsigned long long *s_pc,
                                          int bid, int nb) {
    static_assert(!ModelTraits<MODEL>::tiled && ModelTraits<MODEL>::planes == 3, "the other models go through the warp tile");
    static_assert(AG == 1 || (!WARP_ROW && V == 1 && TEAM * AG <= 32), "arc groups: team rows within a warp");
    constexpr int TPW = 32 / TEAM;
    constexpr int SW = TEAM * V;
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    const bool sparse = *(volatile const int32_t *)&C->sparse != 0;
    const int32_t *rows = nullptr;   // frontier steps: candidate rows; dense: a range
    int32_t r0 = 0;
    int64_t nrows;
    if (sparse) {
        if (which >= 2) return;
        rows = which ? A.cand_mid : A.cand_small;
        nrows = (int64_t)((volatile const uint32_t *)C->cand_n)[which];
    } else {
        r0 = which == 0 ? A.r_small : which == 1 ? A.r_mid : A.r_small4;
        nrows = which == 0 ? A.n_small : which == 1 ? A.n_mid : A.n_small4;
    }
    if (nrows == 0) return;
    const int nl = A.Wn * 32;
    const bool lanes_on = A.lane_cnt != nullptr;
    const bool build = list_wanted(A);
    if (lanes_on)
        for (int i = threadIdx.x; i < A.np * nl; i += blockDim.x) s_lane[i] = 0;
    set_acc_zero(s_pc, A.S);
    const int lane = threadIdx.x & 31;
    const int team = lane / TEAM;
    const int tl = lane % TEAM;
    const int64_t gwarp = ((int64_t)bid * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)nb * blockDim.x) >> 5;
    constexpr int RPI = WARP_ROW ? 1 : TPW / AG;
    const int list_slot = A.k & 1;
    const int64_t nitems = nrows * A.nslices;
    Accum acc;
    // The word contexts and the plane popcount changes belong to the thread's current
    // slice: recomputed / flushed to shared memory only when the slice changes (never,
    // when a row is a single slice).
    int ctx_slice = -1;
    WordCtx x[V];
    int32_t d0[V], d1[V], d2[V];
#pragma unroll
    for (int i = 0; i < V; ++i) d0[i] = d1[i] = d2[i] = 0;

    for (int64_t base = gwarp * RPI; base < nitems; base += nwarps * RPI) {
        const int64_t item = WARP_ROW ? base : base + team / AG;
        const bool has_row = item < nitems;
        const int64_t ridx = has_row ? div_slices(item, A.nslices, nitems) : 0;
        const int slice = has_row ? (int)(item - ridx * A.nslices) : 0;
        const int32_t v = has_row ? (rows ? __ldg(rows + ridx) : r0 + (int32_t)ridx) : 0;   // new id
        const uint32_t node = has_row ? node_of(A, v) : 0u;                                  // Philox subject
        const int w0 = slice * SW + tl * V;
        const size_t off = (size_t)v * A.Wn + w0;
        if (slice != ctx_slice) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                if (ctx_slice >= 0) set_acc_add(s_pc, x[i].s, d0[i], d1[i], d2[i]);
                d0[i] = d1[i] = d2[i] = 0;
                x[i] = word_ctx(A, w0 + i);
            }
            ctx_slice = slice;
        }
        // lanes that can change through their in-arcs
        uint32_t need[V];
        {
            const Vec<V> a = has_row ? ld_vec<V, CG>(A.cur + off) : Vec<V>{};
            const Vec<V> b = has_row ? ld_vec<V, CG>(A.cur + A.plane_words + off) : Vec<V>{};
#pragma unroll
            for (int i = 0; i < V; ++i) need[i] = need_of<MODEL>(has_row ? x[i].vm : 0u, a.w[i], b.w[i], 0u);
        }
        uint32_t any_need = 0u;
#pragma unroll
        for (int i = 0; i < V; ++i) any_need |= need[i];
#pragma unroll
        for (int o = 1; o < TEAM; o <<= 1) any_need |= __shfl_xor_sync(0xffffffffu, any_need, o);

        uint32_t c[V][B];
#pragma unroll
        for (int i = 0; i < V; ++i)
#pragma unroll
            for (int b = 0; b < B; ++b) c[i][b] = 0u;
        int32_t beg = 0, end = 0;
        if (has_row) {
            beg = __ldg(A.rp + v);
            end = __ldg(A.rp + v + 1);
        }
        constexpr int parts = WARP_ROW ? TPW : AG;   // teams that share a row
        gather_counts<MODEL, V, B, TEAM, parts, CG>(A, beg, any_need ? end - beg : 0, 8 * parts, w0, lane, c);
        constexpr bool SPLIT = WARP_ROW && TPW >= V;   // enough teams to give each word one
        if constexpr (SPLIT && V == 2) {
            // merge the teams' counters, reduce-scatter first: at the first butterfly level
            // the partners (teams 2j, 2j+1) swap halves and keep word (team & 1) each, so
            // the remaining levels add one word instead of two; team i < 2 ends up with
            // the warp total of word i, which it decides below
            const int par = team & 1;
            uint32_t d[B];
#pragma unroll
            for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, par ? c[0][b] : c[1][b], TEAM);
#pragma unroll
            for (int b = 0; b < B; ++b) c[0][b] = par ? c[1][b] : c[0][b];
            add_sliced<B>(c[0], d);
#pragma unroll
            for (int o = 2 * TEAM; o < 32; o <<= 1) {
#pragma unroll
                for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, c[0][b], o);
                add_sliced<B>(c[0], d);
            }
#pragma unroll
            for (int b = 0; b < B; ++b) c[1][b] = c[0][b];
        } else if constexpr (parts > 1) {
            // merge the teams' partial results (the warp is converged here)
#pragma unroll
            for (int o = TEAM; o < TEAM * parts; o <<= 1) {
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    uint32_t d[B];
#pragma unroll
                    for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, c[i][b], o);
                    add_sliced<B>(c[i], d);
                }
            }
        }
        uint32_t fl = 0u;
        bool writer;
        if constexpr (SPLIT) {
            // every team holds the merged counts of the same words: team i < V decides the
            // i-th word of each thread's V words, so the decisions of a row run V-wide
            // instead of V-deep
            writer = has_row && team < V;
            if (writer) {
                const int i = team;
                uint32_t cw[B];
#pragma unroll
                for (int b = 0; b < B; ++b) cw[b] = pick<V, B>(c, i, b);
                WordCtx xw = x[0];
#pragma unroll
                for (int q = 1; q < V; ++q)
                    if (i == q) xw = x[q];
                const uint32_t s0 = ld_word<CG>(A.cur + off + i);
                const uint32_t s1 = ld_word<CG>(A.cur + A.plane_words + off + i);
                const uint32_t s2 = ld_word<CG>(A.cur + 2 * A.plane_words + off + i);
                const WordOut o = update_word<MODEL, B>(A, node, xw, s0, s1, s2, end - beg, cw, 0u);
                A.nxt[off + i] = o.n0;
                A.nxt[A.plane_words + off + i] = o.n1;
                A.nxt[2 * A.plane_words + off + i] = o.n2;
#pragma unroll
                for (int q = 0; q < V; ++q) {
                    if (i == q) {
                        d0[q] += __popc(o.n0) - __popc(s0);
                        d1[q] += __popc(o.n1) - __popc(s1);
                        d2[q] += __popc(o.n2) - __popc(s2);
                    }
                }
                if (lanes_on) {
                    lane_deltas(s_lane, w0 + i, s0, o.n0);
                    lane_deltas(s_lane + nl, w0 + i, s1, o.n1);
                    lane_deltas(s_lane + 2 * nl, w0 + i, s2, o.n2);
                }
                fl |= word_flags<MODEL>(o, s0, s1, s2);
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
            writer = has_row && team == 0;
        } else {
        writer = has_row && team % parts == 0;
        if (writer) {
            // own state again (L1/L2-resident): not kept live across the gather
            uint32_t s0[V], s1[V], s2[V];
            {
                const Vec<V> a = ld_vec<V, CG>(A.cur + off);
                const Vec<V> b = ld_vec<V, CG>(A.cur + A.plane_words + off);
                const Vec<V> e = ld_vec<V, CG>(A.cur + 2 * A.plane_words + off);
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    s0[i] = a.w[i];
                    s1[i] = b.w[i];
                    s2[i] = e.w[i];
                }
            }
            uint32_t n0[V], n1[V], n2[V];
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const WordOut o = update_word<MODEL, B>(A, node, x[i], s0[i], s1[i], s2[i], end - beg, c[i], 0u);
                n0[i] = o.n0;
                n1[i] = o.n1;
                n2[i] = o.n2;
                d0[i] += __popc(o.n0) - __popc(s0[i]);
                d1[i] += __popc(o.n1) - __popc(s1[i]);
                d2[i] += __popc(o.n2) - __popc(s2[i]);
                if (lanes_on) {
                    lane_deltas(s_lane, w0 + i, s0[i], o.n0);
                    lane_deltas(s_lane + nl, w0 + i, s1[i], o.n1);
                    lane_deltas(s_lane + 2 * nl, w0 + i, s2[i], o.n2);
                }
                fl |= word_flags<MODEL>(o, s0[i], s1[i], s2[i]);
            }
            st_vec<V>(A.nxt + off, n0);
            st_vec<V>(A.nxt + A.plane_words + off, n1);
            st_vec<V>(A.nxt + 2 * A.plane_words + off, n2);
        }
#pragma unroll
        for (int o = 1; o < TEAM; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
        }
        const bool leader = writer && tl == 0;
        const bool want = leader && fl != 0u;
        if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
        if (A.prof_bytes && leader) acc.bytes += row_bytes(SW, 3, any_need != 0u, end - beg);
        list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
        if (sparse && leader) atomicAnd(&A.bitmap[v >> 5], ~(1u << (v & 31)));
    }
#pragma unroll
    for (int i = 0; i < V; ++i) set_acc_add_warp(s_pc, ctx_slice >= 0 ? x[i].s : -1, d0[i], d1[i], d2[i]);
    flush_accum(A, acc, list_slot, WARP_ROW ? PK_MID : (BT == 4 ? PK_SMALL4 : PK_SMALL));
    set_acc_flush(A, s_pc);
    if (lanes_on) flush_lanes(A, s_lane, nl);
}

// ------------------------------------------------------------------ warp-tile kernels

// Shape of one warp's tile: SPP word slots per pass (one row slice per team, or one row
// slice per warp), NP passes.  128 slots keep the queues several batches of 32 long;
// the wide rows' 16 counter planes take 64.
template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT, int WB = kWideBits>
struct TileShape {
    static constexpr bool counts = ModelTraits<MODEL>::counts;
    static constexpr int B = counts ? (WARP_ROW ? WB : BT) : 1;
    static constexpr int SW = TEAM * V;
    static constexpr int SPP = WARP_ROW ? SW : 32 * V;
    static constexpr int RPP = WARP_ROW ? 1 : 32 / TEAM;
    static constexpr int TARGET = WARP_ROW ? 64 : 128;
    static constexpr int NP = SPP >= TARGET ? 1 : TARGET / SPP;
    static constexpr int NS = NP * SPP;
    static constexpr int NARC = counts ? 0 : 32 * V + 192;
    using T = Tile<B, ModelTraits<MODEL>::fixed_draws, NS, NP * RPP, NARC>;
    static constexpr size_t bytes = sizeof(T) * (kBlock / 32);
    // slot -> row of the tile and word within the row's slice
    static __device__ __forceinline__ int row_of_slot(int slot) {
        return WARP_ROW ? slot / SW : slot / SPP * RPP + (slot & 31) / TEAM;
    }
    static __device__ __forceinline__ int word_of_slot(int slot) {
        return WARP_ROW ? slot % SW : (slot & 31) % TEAM * V + (slot >> 5) % V;
    }
};

// Largest dynamic shared memory any row kernel is launched with: its tiles and the
// per-lane counters (run_wave bounds those by 32 KB).
constexpr size_t kLaneCounterBytes = 32 * 1024;

// Draws of the tile's count items (infection, exposure, linear thresholds): the result
// lanes replace counter plane 0.  A lane changes iff its uniform is below its threshold
// (LT) or reaches it (the survival tables).
template <int MODEL, int B, class TileT, class CtxFn>
__device__ __forceinline__ void draw_counts(const StepArgs &A, TileT &T, int n, int lane, CtxFn ctx) {
    constexpr bool LT = MODEL == FSGP_LT;
    constexpr uint32_t tag = LT ? TAG_LT_THRESH : TAG_INFECT;
    const uint32_t t = LT ? 0u : A.t;
    if (lane == 0) T.ties = 0;
    __syncwarp();
#pragma unroll 1
    for (int q0 = 0; q0 < n; q0 += 32) {
        const unsigned items = __ballot_sync(0xffffffffu, q0 + lane < n);
        if (q0 + lane >= n) continue;
        const int slot = T.qc[q0 + lane];
        uint32_t c[B];
#pragma unroll
        for (int b = 0; b < B; ++b) c[b] = T.c[b][slot];
        uint32_t node;
        int w;
        const int row = ctx(slot, node, w);
        const SetParams &sp = A.sp[w >> A.ws_shift];
        const uint32_t g = A.gbase + (uint32_t)(w & (A.Ws - 1));
        const uint32_t k0 = __ldg(&sp.key0), k1 = __ldg(&sp.key1);
        const uint32_t cand = any_count<B>(c);
        // counter planes in use among the items at hand
        int nb = 0;
#pragma unroll
        for (int b = 0; b < B; ++b) nb = __any_sync(items, c[b] != 0u) ? b + 1 : nb;
        const Planes8 P = philox4x32_10_x2(node, t, g, tag << 8, k0, k1);
        uint32_t tied = 0u, won = 0u;
        auto tie_fn = [&](uint32_t lanes, uint32_t th) {
            tied |= lanes;
            if (LT && (th & 0xffffffu) == 0u) {   // T's other bits are all ones: every tied u is <= T
                won |= lanes;
                return;
            }
            const int at = atomicAdd(&T.ties, 1);
            if (at < TileT::kTies) {
                T.tie_slot[at] = (uint16_t)slot;
                T.tie_eq[at] = lanes;
                T.tie_thr[at] = th;
            } else {
                const uint32_t less = less_from(lanes, th, 2u, node, t, g, tag, k0, k1);
                won |= LT ? less : lanes & ~less;
            }
        };
        uint32_t chg;
        if constexpr (LT) {
            const int32_t d = __ldg(A.rp + row + 1) - __ldg(A.rp + row);
            uint32_t sat = 0u;
            if ((uint64_t)d < (1ull << B)) sat = ge_const<B>(c, (uint32_t)d) & cand;
            const uint32_t rem = cand & ~sat;
            chg = sat;
            if (rem) chg |= counts_u_less_nb<B>(nb, P, c, rem, LtThr{(uint32_t)d}, tie_fn);
        } else {
            const int32_t ksat = __ldg(&sp.ksat);
            uint32_t sat = 0u;
            if ((uint64_t)ksat < (1ull << B)) sat = ge_const<B>(c, (uint32_t)ksat) & cand;
            const uint32_t rem = cand & ~sat;
            chg = __ldg(&sp.never) ? sat : cand;
            if (rem && chg == cand) chg &= ~counts_u_less_nb<B>(nb, P, c, rem, SurvThr<(B <= 8)>{sp.surv, sp.masks}, tie_fn);
        }
        T.c[0][slot] = (chg & ~tied) | won;
    }
    __syncwarp();
    const int nt = min(T.ties, TileT::kTies);
    for (int i = lane; i < nt; i += 32) {
        const int slot = T.tie_slot[i];
        const uint32_t eq = T.tie_eq[i];
        uint32_t node;
        int w;
        ctx(slot, node, w);
        const SetParams &sp = A.sp[w >> A.ws_shift];
        const uint32_t less = less_from(eq, T.tie_thr[i], 2u, node, t, A.gbase + (uint32_t)(w & (A.Ws - 1)), tag,
                                        __ldg(&sp.key0), __ldg(&sp.key1));
        const uint32_t add = LT ? less : eq & ~less;
        if (add) atomicOr(&T.c[0][slot], add);   // two groups of one word may both be tied
    }
    __syncwarp();
}

template <int MODEL, bool PAIR, class TileT, class CtxFn>
__device__ __forceinline__ void draw_arc_items(const StepArgs &A, TileT &T, int na, int lane, CtxFn ctx) {
    constexpr bool W = ModelTraits<MODEL>::weighted;
    draw_arcs<PAIR>(A, T.c[0], T.arc_eq, T.arc_pos, T.arc_slot, na, W ? TAG_ARC_INFECT : TAG_IC_EDGE, lane, ctx,
              [&A, &T](int row, uint32_t pos, const SetParams &sp) -> uint64_t {
                  if constexpr (W) return arc_thr(__ldg(&sp.beta_f), __ldg(A.arc_w + pos));
                  else if (A.ic_mode == FSGP_IC_WEIGHTED_CASCADE) return (uint64_t)T.thr[row] + 1ull;
                  else return __ldg(&sp.p_const);
              });
}

// The tile's draws after its gather (queue lengths nq, nf, na).
template <int MODEL, int B, bool PAIR, class TileT, class CtxFn>
__device__ __forceinline__ void draw_tile(const StepArgs &A, TileT &T, int nq, const int (&nf)[2], int na, int lane,
                                          CtxFn ctx) {
    __syncwarp();
    if constexpr (ModelTraits<MODEL>::counts) draw_counts<MODEL, B>(A, T, nq, lane, ctx);
    else draw_arc_items<MODEL, PAIR>(A, T, na, lane, ctx);
    if constexpr (ModelTraits<MODEL>::fixed_draws >= 1)
        draw_fixed<false>(A, T.f[0], T.eq(), T.qf[0], nf[0], lane, ctx);
    if constexpr (ModelTraits<MODEL>::fixed_draws >= 2)
        draw_fixed<true>(A, T.f[1], T.eq(), T.qf[1], nf[1], lane, ctx);
}

// Lanes of the word that may leave their state without in-arcs through fixed draw j.
template <int MODEL>
__device__ __forceinline__ uint32_t fixed_lanes(int j, uint32_t vm, uint32_t s0, uint32_t s1, uint32_t s2) {
    if (j == 0) return s0 & vm;
    return (MODEL == FSGP_SEIR ? s2 : s1) & vm;
}

// The next state of a word from its tile slot (chg: the lanes changed through in-arcs,
// f0 / f1: the results of the fixed draws).
template <int MODEL>
__device__ __forceinline__ WordOut next_word(uint32_t s0, uint32_t s1, uint32_t s2, uint32_t chg, uint32_t f0,
                                             uint32_t f1) {
    WordOut o;
    o.n1 = o.n2 = 0u;
    if constexpr (ModelTraits<MODEL>::cascade) {
        o.n0 = s0 | chg;
        o.n1 = chg;
    } else if constexpr (MODEL == FSGP_SEIR) {
        o.n0 = (s0 & ~f0) | f1;
        o.n1 = s1 | f0;
        o.n2 = (s2 & ~f1) | chg;
    } else if constexpr (MODEL == FSGP_SEIS) {
        o.n0 = (s0 & ~f0) | f1;
        o.n1 = (s1 & ~f1) | chg;
    } else {
        o.n0 = (s0 & ~f0) | chg;
        if constexpr (MODEL == FSGP_SIR || MODEL == kSirW) o.n1 = s1 | f0;
    }
    return o;
}

// Arc models: gather the in-arcs [e_begin, e_end) with stride `step` (groups of 4) and
// queue every (arc, word) pair whose source presses a lane that can change; the queue is
// worked off whenever the next arcs might not fit.  The whole warp iterates together.
template <int MODEL, int V, int NARC, bool CG, class TileT, class CtxFn>
__device__ __forceinline__ void gather_push(const StepArgs &A, TileT &T, int64_t e_begin, int64_t e_end, int64_t step,
                                            int64_t arcb, int w0, uint32_t (&need)[V], int slot0, int slot_step,
                                            int lane, int &na, CtxFn ctx) {
    const uint32_t *src = A.cur + (size_t)ModelTraits<MODEL>::src_plane * A.plane_words + w0;
    const size_t Wn = (size_t)A.Wn;
    int32_t u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = e_begin + j < e_end ? __ldg(A.col + e_begin + j) : -1;
    for (int64_t e = e_begin; __any_sync(0xffffffffu, e < e_end); e += step) {
        Vec<V> xs[4];
        uint32_t any = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (u[j] >= 0) {
                xs[j] = ld_vec<V, CG>(src + (size_t)u[j] * Wn);
            } else {
#pragma unroll
                for (int i = 0; i < V; ++i) xs[j].w[i] = 0u;
            }
        }
        const int64_t en = e + step;
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = en + j < e_end ? __ldg(A.col + en + j) : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < V; ++i) {
                xs[j].w[i] &= need[i];
                any |= xs[j].w[i];
            }
        if (!__any_sync(0xffffffffu, any != 0u)) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (na > NARC - 32 * V) {
                __syncwarp();
                draw_arc_items<MODEL, CG>(A, T, na, lane, ctx);
                na = 0;
                // lanes already reached need no more draws
                bool left = false;
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    need[i] &= ~T.c[0][slot0 + i * slot_step];
                    left |= need[i] != 0u;
#pragma unroll
                    for (int q = 0; q < 4; ++q) xs[q].w[i] &= need[i];
                }
                if (!__any_sync(0xffffffffu, left)) return;
            }
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const unsigned m = __ballot_sync(0xffffffffu, xs[j].w[i] != 0u);
                if (xs[j].w[i]) {
                    const int at = na + __popc(m & ((1u << lane) - 1u));
                    T.arc_slot[at] = (uint16_t)(slot0 + i * slot_step);
                    T.arc_pos[at] = (uint32_t)(e + j + arcb);   // the caller's arc position
                    T.arc_eq[at] = xs[j].w[i];
                }
                na += __popc(m);
            }
        }
    }
}

// Row kernel on warp tiles: one work item is one slice (TEAM*V words) of one row.
// WARP_ROW = false: one team per item; true: one warp per item.  which: as in rows_body.
// CG: state planes through L2 only (persistent step loop).  bid of nb: the CTA's place among
// those that work on these rows.
template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT, bool CG, int WB>
__device__ __forceinline__ void rows_tile(const StepArgs &A, int which, uint8_t *smem, int32_t *s_lane,
                                          unsigned long long *s_pc, int bid, int nb) {
    using S = TileShape<MODEL, V, TEAM, WARP_ROW, BT, WB>;
    constexpr int B = S::B;
    constexpr int TPW = 32 / TEAM;
    constexpr int SW = TEAM * V;
    constexpr int P = ModelTraits<MODEL>::planes;
    constexpr int NF = ModelTraits<MODEL>::fixed_draws;
    constexpr bool COUNTS = ModelTraits<MODEL>::counts;
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    const bool sparse = *(volatile const int32_t *)&C->sparse != 0;
    const int32_t *rows = nullptr;   // frontier steps: candidate rows; dense: a range
    int32_t r0 = 0;
    int64_t nrows;
    if (sparse) {
        if (which >= 2) return;
        rows = which ? A.cand_mid : A.cand_small;
        nrows = (int64_t)((volatile const uint32_t *)C->cand_n)[which];
    } else {
        r0 = which == 0 ? A.r_small : which == 1 ? A.r_mid : A.r_small4;
        nrows = which == 0 ? A.n_small : which == 1 ? A.n_mid : A.n_small4;
    }
    if (nrows == 0) return;
    const int nl = A.Wn * 32;
    const bool lanes_on = A.lane_cnt != nullptr;
    const bool build = list_wanted(A);
    if (lanes_on)
        for (int i = threadIdx.x; i < A.np * nl; i += blockDim.x) s_lane[i] = 0;
    set_acc_zero(s_pc, A.S);
    typename S::T &T = reinterpret_cast<typename S::T *>(smem)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int team = lane / TEAM;
    const int tl = lane % TEAM;
    const int64_t gwarp = ((int64_t)bid * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)nb * blockDim.x) >> 5;
    const int list_slot = A.k & 1;
    const int64_t nitems = nrows * A.nslices;
    // few rows: fewer passes per tile, so that every warp gets one
    const int np = (int)min((int64_t)S::NP, max((int64_t)1, nitems / (nwarps * S::RPP)));
    // the passes of a tile are a whole round of the grid apart: neighbouring rows (the rows
    // of a class come in descending degree buckets) go to different warps
    const int64_t round = nwarps * S::RPP;
    Accum acc;
    int ctx_slice = -1;              // slice of the valid-lane masks below
    uint32_t vm[V];
    int cur_s[V];                    // set of the plane-count changes not yet flushed
    int32_t d0[V], d1[V], d2[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
        d0[i] = d1[i] = d2[i] = 0;
        cur_s[i] = -1;
        vm[i] = 0u;
    }
    auto ctx = [&T](int slot, uint32_t &node, int &w) -> int {
        const int r = S::row_of_slot(slot);
        node = T.node[r];
        w = T.w0[r] + S::word_of_slot(slot);
        return COUNTS ? T.row[r] : r;
    };

    for (int64_t base = gwarp * S::RPP; base < nitems; base += np * round) {
        int nq = 0, na = 0;
        int nf[2] = {0, 0};
#pragma unroll 1
        for (int p = 0; p < np; ++p) {
            const int64_t item = base + p * round + (WARP_ROW ? 0 : team);
            const bool has_row = item < nitems;
            int64_t ridx = 0;
            int slice = 0;
            if (has_row) {
                ridx = div_slices(item, A.nslices, nitems);
                slice = (int)(item - ridx * A.nslices);
            }
            const int32_t v = has_row ? (rows ? __ldg(rows + ridx) : r0 + (int32_t)ridx) : 0;   // new id
            const int w0 = slice * SW + tl * V;
            if (slice != ctx_slice) {
#pragma unroll
                for (int i = 0; i < V; ++i) vm[i] = word_ctx(A, w0 + i).vm;
                ctx_slice = slice;
            }
            const size_t off = (size_t)v * A.Wn + w0;
            int32_t beg = 0, end = 0;
            uint32_t need[V], fx[2][V];
            {
                Vec<V> a{}, b{}, e{};
                if (has_row) {
                    beg = __ldg(A.rp + v);
                    end = __ldg(A.rp + v + 1);
                    a = ld_vec<V, CG>(A.cur + off);
                    if (P >= 2 && !ModelTraits<MODEL>::cascade) b = ld_vec<V, CG>(A.cur + A.plane_words + off);
                    if (P >= 3) e = ld_vec<V, CG>(A.cur + 2 * A.plane_words + off);
                }
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const uint32_t m = has_row ? vm[i] : 0u;
                    need[i] = need_of<MODEL>(m, a.w[i], b.w[i], e.w[i]);
                    fx[0][i] = NF >= 1 && (A.fixed_on & 1) ? fixed_lanes<MODEL>(0, m, a.w[i], b.w[i], e.w[i]) : 0u;
                    fx[1][i] = NF >= 2 && (A.fixed_on & 2) ? fixed_lanes<MODEL>(1, m, a.w[i], b.w[i], e.w[i]) : 0u;
                }
            }
            uint32_t any_need = 0u;
#pragma unroll
            for (int i = 0; i < V; ++i) any_need |= need[i];
#pragma unroll
            for (int o = 1; o < TEAM; o <<= 1) any_need |= __shfl_xor_sync(0xffffffffu, any_need, o);
            const int r = p * S::RPP + (WARP_ROW ? 0 : team);
            if (WARP_ROW ? lane == 0 : tl == 0) {
                T.row[r] = has_row ? v : -1;
                T.node[r] = has_row ? node_of(A, v) : 0u;
                T.w0[r] = slice * SW;
                if (A.prof_bytes && has_row) acc.bytes += row_bytes(SW, P, any_need != 0u, end - beg);
            }
            const int slot0 = WARP_ROW ? p * SW + tl * V : p * S::SPP + lane;
            constexpr int slot_step = WARP_ROW ? 1 : 32;
            if constexpr (COUNTS) {
                uint32_t c[V][B];
#pragma unroll
                for (int i = 0; i < V; ++i)
#pragma unroll
                    for (int b = 0; b < B; ++b) c[i][b] = 0u;
                constexpr int parts = WARP_ROW ? TPW : 1;
                gather_counts<MODEL, V, B, TEAM, parts, CG>(A, beg, any_need ? end - beg : 0, 8 * parts, w0, lane, c);
                constexpr bool SPLIT = WARP_ROW && TPW >= V;   // team i < V stores word i
                if constexpr (SPLIT && V == 2) {
                    // merge the teams' counters, reduce-scatter first: at the first level the
                    // partners (teams 2j, 2j+1) swap halves and keep word (team & 1) each
                    const int par = team & 1;
                    uint32_t d[B];
#pragma unroll
                    for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, par ? c[0][b] : c[1][b], TEAM);
#pragma unroll
                    for (int b = 0; b < B; ++b) c[0][b] = par ? c[1][b] : c[0][b];
                    add_sliced<B>(c[0], d);
#pragma unroll
                    for (int o = 2 * TEAM; o < 32; o <<= 1) {
#pragma unroll
                        for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, c[0][b], o);
                        add_sliced<B>(c[0], d);
                    }
#pragma unroll
                    for (int b = 0; b < B; ++b) c[1][b] = c[0][b];
                } else if constexpr (WARP_ROW) {
#pragma unroll
                    for (int o = TEAM; o < 32; o <<= 1)
#pragma unroll
                        for (int i = 0; i < V; ++i) {
                            uint32_t d[B];
#pragma unroll
                            for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, c[i][b], o);
                            add_sliced<B>(c[i], d);
                        }
                }
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    // the threads that store word i of their slice
                    const bool mine = WARP_ROW ? (SPLIT ? team == i : team == 0) : true;
                    const int slot = slot0 + i * slot_step;
                    uint32_t any = 0u;
#pragma unroll
                    for (int b = 0; b < B; ++b) {
                        c[i][b] &= need[i];
                        any |= c[i][b];
                    }
                    if (mine) {
                        T.c[0][slot] = c[i][0];
                        if (any)
#pragma unroll
                            for (int b = 1; b < B; ++b) T.c[b][slot] = c[i][b];
                    }
                    queue_push(T.qc, nq, mine && any != 0u, slot, lane);
                }
            } else {
                // (every lane of the warp joins the gather)
                const int64_t arcb = has_row ? (int64_t)__ldg(A.arc0 + v) - beg : 0;
                if (MODEL == FSGP_IC && (WARP_ROW ? lane == 0 : tl == 0))
                    T.thr[r] = 0xffffffffu / (uint32_t)max(end - beg, 1);
                if (!WARP_ROW || team == 0)
#pragma unroll
                    for (int i = 0; i < V; ++i) T.c[0][slot0 + i * slot_step] = 0u;
                __syncwarp();
                if (!any_need) end = beg;
                gather_push<MODEL, V, S::NARC, CG>(A, T, (int64_t)beg + (WARP_ROW ? 4 * team : 0), end,
                                               WARP_ROW ? 4 * TPW : 4, arcb, w0, need, slot0, slot_step, lane, na, ctx);
            }
            if constexpr (NF >= 1) {
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const bool mine = !WARP_ROW || team == 0;
                    const int slot = slot0 + i * slot_step;
#pragma unroll
                    for (int j = 0; j < NF; ++j) {
                        if (mine) T.f[j][slot] = fx[j][i];
                        queue_push(T.qf[j], nf[j], mine && fx[j][i] != 0u, slot, lane);
                    }
                }
            }
        }
        draw_tile<MODEL, B, CG>(A, T, nq, nf, na, lane, ctx);
        __syncwarp();
        // next states
        if constexpr (!WARP_ROW) {
#pragma unroll 1
            for (int p = 0; p < np; ++p) {
                const int r = p * S::RPP + team;
                const int32_t v = T.row[r];
                const int w0 = T.w0[r] + tl * V;
                uint32_t fl = 0u;
                if (v >= 0) {
                    const size_t off = (size_t)v * A.Wn + w0;
                    const Vec<V> a = ld_vec<V, CG>(A.cur + off);
                    Vec<V> b{}, e{};
                    if (P >= 2) b = ld_vec<V, CG>(A.cur + A.plane_words + off);
                    if (P >= 3) e = ld_vec<V, CG>(A.cur + 2 * A.plane_words + off);
                    uint32_t n0[V], n1[V], n2[V];
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        const int slot = p * S::SPP + i * 32 + lane;
                        const WordOut o = next_word<MODEL>(a.w[i], b.w[i], e.w[i], T.c[0][slot],
                                                           T.template fixed<0>(slot), T.template fixed<1>(slot));
                        n0[i] = o.n0;
                        n1[i] = o.n1;
                        n2[i] = o.n2;
                        const int s = (w0 + i) >> A.ws_shift;
                        if (s != cur_s[i]) {
                            if (cur_s[i] >= 0) set_acc_add(s_pc, cur_s[i], d0[i], d1[i], d2[i]);
                            d0[i] = d1[i] = d2[i] = 0;
                            cur_s[i] = s;
                        }
                        d0[i] += __popc(o.n0) - __popc(a.w[i]);
                        if (P >= 2) d1[i] += __popc(o.n1) - __popc(b.w[i]);
                        if (P >= 3) d2[i] += __popc(o.n2) - __popc(e.w[i]);
                        if (lanes_on) {
                            lane_deltas(s_lane, w0 + i, a.w[i], o.n0);
                            if (P >= 2) lane_deltas(s_lane + nl, w0 + i, b.w[i], o.n1);
                            if (P >= 3) lane_deltas(s_lane + 2 * nl, w0 + i, e.w[i], o.n2);
                        }
                        fl |= word_flags<MODEL>(o, a.w[i], b.w[i], e.w[i]);
                    }
                    st_vec<V>(A.nxt + off, n0);
                    if (P >= 2) st_vec<V>(A.nxt + A.plane_words + off, n1);
                    if (P >= 3) st_vec<V>(A.nxt + 2 * A.plane_words + off, n2);
                }
#pragma unroll
                for (int o = 1; o < TEAM; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
                const bool leader = v >= 0 && tl == 0;
                const bool want = leader && fl != 0u;
                if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
                list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
                if (sparse && leader) atomicAnd(&A.bitmap[v >> 5], ~(1u << (v & 31)));
            }
        } else {
            // one lane per word slot; a row's words are SW neighbouring lanes (a slice wider
            // than the warp: several rounds of one row)
            constexpr int GRP = SW < 32 ? SW : 32;
            uint32_t fl = 0u;
#pragma unroll 1
            for (int q0 = 0; q0 < np * SW; q0 += 32) {
                const int slot = q0 + lane;
                const int r = slot / SW;
                const int32_t v = slot < np * SW ? T.row[r] : -1;
                if (q0 % SW == 0) fl = 0u;
                if (v >= 0) {
                    const int w = T.w0[r] + slot % SW;
                    const size_t off = (size_t)v * A.Wn + w;
                    const uint32_t s0 = ld_word<CG>(A.cur + off);
                    const uint32_t s1 = P >= 2 ? ld_word<CG>(A.cur + A.plane_words + off) : 0u;
                    const uint32_t s2 = P >= 3 ? ld_word<CG>(A.cur + 2 * A.plane_words + off) : 0u;
                    const WordOut o = next_word<MODEL>(s0, s1, s2, T.c[0][slot], T.template fixed<0>(slot),
                                                       T.template fixed<1>(slot));
                    A.nxt[off] = o.n0;
                    if (P >= 2) A.nxt[A.plane_words + off] = o.n1;
                    if (P >= 3) A.nxt[2 * A.plane_words + off] = o.n2;
                    const int s = w >> A.ws_shift;
                    if (s != cur_s[0]) {
                        if (cur_s[0] >= 0) set_acc_add(s_pc, cur_s[0], d0[0], d1[0], d2[0]);
                        d0[0] = d1[0] = d2[0] = 0;
                        cur_s[0] = s;
                    }
                    d0[0] += __popc(o.n0) - __popc(s0);
                    if (P >= 2) d1[0] += __popc(o.n1) - __popc(s1);
                    if (P >= 3) d2[0] += __popc(o.n2) - __popc(s2);
                    if (lanes_on) {
                        lane_deltas(s_lane, w, s0, o.n0);
                        if (P >= 2) lane_deltas(s_lane + nl, w, s1, o.n1);
                        if (P >= 3) lane_deltas(s_lane + 2 * nl, w, s2, o.n2);
                    }
                    fl |= word_flags<MODEL>(o, s0, s1, s2);
                }
                if (SW <= 32 || (q0 + 32) % SW == 0) {
#pragma unroll
                    for (int o = 1; o < GRP; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
                    const bool leader = v >= 0 && lane % GRP == 0;
                    const bool want = leader && fl != 0u;
                    if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
                    list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
                    if (sparse && leader) atomicAnd(&A.bitmap[v >> 5], ~(1u << (v & 31)));
                    fl = 0u;
                }
            }
        }
        __syncwarp();   // the next tile overwrites the slots
    }
#pragma unroll
    for (int i = 0; i < V; ++i) set_acc_add_warp(s_pc, cur_s[i], d0[i], d1[i], d2[i]);
    flush_accum(A, acc, list_slot, WARP_ROW ? PK_MID : (BT == 4 ? PK_SMALL4 : PK_SMALL));
    set_acc_flush(A, s_pc);
    if (lanes_on) flush_lanes(A, s_lane, nl);
}

// The rows of one class: through the warp tile, or in place (SWIR).
template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT, bool CG, int WB = kWideBits, int AG = 1>
__device__ __forceinline__ void rows_class(const StepArgs &A, int which, uint8_t *smem, int32_t *s_lane,
                                           unsigned long long *s_pc, int bid, int nb) {
    if constexpr (ModelTraits<MODEL>::tiled) rows_tile<MODEL, V, TEAM, WARP_ROW, BT, CG, WB>(A, which, smem, s_lane, s_pc, bid, nb);
    else rows_body<MODEL, V, TEAM, WARP_ROW, BT, CG, WARP_ROW ? WB : BT, AG>(A, which, s_lane, s_pc, bid, nb);
}

// Dynamic shared memory of a class's tiles, and of either class's (fused kernels).
template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT>
constexpr size_t TileBytes = ModelTraits<MODEL>::tiled ? TileShape<MODEL, V, TEAM, WARP_ROW, BT>::bytes : 0;
template <int MODEL, int V, int TEAM>
constexpr size_t FusedBytes = std::max(TileBytes<MODEL, V, TEAM, true, kSmallBits>,
                                       TileBytes<MODEL, V, TEAM, false, kSmallBits>);

template <int MODEL, int V, int TEAM, bool WARP_ROW, int BT = kSmallBits>
__global__ void __launch_bounds__(kBlock, min_ctas<V>()) k_rows(StepArgs A, int which) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ unsigned long long s_pc[kPC * kMaxSets];
    constexpr size_t tile = TileBytes<MODEL, V, TEAM, WARP_ROW, BT>;
    rows_class<MODEL, V, TEAM, WARP_ROW, BT, false>(A, which, s_dyn, reinterpret_cast<int32_t *>(s_dyn + tile), s_pc,
                                                    blockIdx.x, gridDim.x);
}

// Small graphs: both row classes in one launch, the first `warp_ctas` CTAs on the rows that
// get a warp each, the others on the rows that get a team each, so that neither waits for
// the other's last row.
template <int MODEL, int V, int TEAM>
__global__ void __launch_bounds__(kBlock, V == 4 ? 2 : 3) k_rows_fused(StepArgs A, int warp_ctas) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ unsigned long long s_pc[kPC * kMaxSets];
    int32_t *s_lane = reinterpret_cast<int32_t *>(s_dyn + FusedBytes<MODEL, V, TEAM>);
    if ((int)blockIdx.x < warp_ctas)
        rows_class<MODEL, V, TEAM, true, kSmallBits, false>(A, 1, s_dyn, s_lane, s_pc, blockIdx.x, warp_ctas);
    else
        rows_class<MODEL, V, TEAM, false, kSmallBits, false>(A, 0, s_dyn, s_lane, s_pc, blockIdx.x - warp_ctas,
                                                            gridDim.x - warp_ctas);
}

// Persistent step loop of a small graph: all T dense steps in one launch, the row work of
// the fused mode (every row, one kernel) separated by grid barriers instead of kernel
// boundaries.  The step control of the launched loop is folded in: each step's plane
// popcount changes go to its own row of pc (running totals are formed after the loop),
// and the cascade models stop at the first step whose previous step activated nothing,
// a decision every CTA takes alike from the same counts.  State is read through L2
// (CG loads): a CTA reads at step k the words other CTAs wrote at step k-1.
// (bounded for 2 resident CTAs per SM: the loop is meant for graphs that fill a few CTAs
// per SM at most, and the body then keeps its state in registers)
template <int MODEL, int TEAM, int WB, int AG>
__global__ void __launch_bounds__(kBlock, kPersistCtas)
    k_rows_persist(const __grid_constant__ StepArgs A0, const __grid_constant__ PersistArgs Q) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    int32_t *s_lane = reinterpret_cast<int32_t *>(s_dyn + FusedBytes<MODEL, 1, TEAM>);
    __shared__ unsigned long long s_pc[kPC * kMaxSets];
    __shared__ StepArgs sA;
    __shared__ unsigned long long s_new[kMaxSets];   // cascade: lanes newly active at the last step
    __shared__ int s_stop;
    constexpr bool cascade = ModelTraits<MODEL>::cascade;
    Ctl *C = A0.ctl;
    {
        const int32_t *src = reinterpret_cast<const int32_t *>(&A0);
        int32_t *dst = reinterpret_cast<int32_t *>(&sA);
        for (int i = threadIdx.x; i < (int)(sizeof(StepArgs) / sizeof(int32_t)); i += blockDim.x) dst[i] = src[i];
    }
    if (cascade)
        for (int s = threadIdx.x; s < A0.S; s += blockDim.x) s_new[s] = __ldcg(Q.pc + (size_t)s * kPC + 1);
    for (int k = 1; k <= Q.T; ++k) {
        __syncthreads();
        if (threadIdx.x == 0) {
            int stop = 0;
            if (cascade) {
                stop = 1;
                for (int s = 0; s < A0.S; ++s)
                    if (s_new[s]) stop = 0;
            }
            s_stop = stop;
            sA.k = k;
            sA.t = Q.t0 + (uint32_t)k;
            sA.cur = (k & 1) ? Q.buf0 : Q.buf1;
            sA.nxt = (k & 1) ? Q.buf1 : Q.buf0;
            sA.pc = Q.pc + (size_t)k * A0.S * kPC;
        }
        __syncthreads();
        if (s_stop) {
            if (blockIdx.x == 0 && threadIdx.x == 0) C->stop = 1;
            break;
        }
        if constexpr (AG > 1) {
            rows_class<MODEL, 1, TEAM, false, kSmallBits, true, WB, AG>(sA, 0, s_dyn, s_lane, s_pc, blockIdx.x, gridDim.x);
        } else if ((int)blockIdx.x < Q.warp_ctas) {
            rows_class<MODEL, 1, TEAM, true, kSmallBits, true, WB>(sA, 1, s_dyn, s_lane, s_pc, blockIdx.x, Q.warp_ctas);
        } else {
            rows_class<MODEL, 1, TEAM, false, kSmallBits, true>(sA, 0, s_dyn, s_lane, s_pc, blockIdx.x - Q.warp_ctas,
                                                                gridDim.x - Q.warp_ctas);
        }
        if (!grid_barrier(&C->bar_count, &C->bar_gen, gridDim.x, &C->err, Q.spin_limit)) break;
        if (blockIdx.x == 0 && threadIdx.x == 0) C->steps_done = k;
        if (cascade)
            for (int s = threadIdx.x; s < A0.S; s += blockDim.x)
                s_new[s] += __ldcg(Q.pc + ((size_t)k * A0.S + s) * kPC + 1);
    }
}

// Hub rows, phase 1: one CTA per (chunk of in-arcs, word slice); per-lane partial counts
// (IC: live masks) are added into the hub's scratch slot.
//   pass 0: every chunk;
//   pass 1 (SIR/SIS): the first chunk of every hub row only; when every susceptible lane
//     of the slice already counts K_sat infected in-arcs there, the slice is flagged:
//     its lanes are infected whatever the rest of the row holds (every count from K_sat
//     on decides the same way), so its other chunks need not be read;
//   pass 2 (SIR/SIS): the other chunks of the slices not flagged.
template <int MODEL, int V, int TEAM>
__global__ void __launch_bounds__(kBlock, min_ctas<V>()) k_hub_chunks(StepArgs A, int pass) {
    __shared__ uint32_t s_cnt[kMaxR];
    constexpr int B = kWideBits;
    constexpr int TPB = kBlock / TEAM;
    constexpr int SW = TEAM * V;
    constexpr int P = ModelTraits<MODEL>::planes;
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    const bool sparse = *(volatile const int32_t *)&C->sparse != 0;
    const int nl = A.Wn * 32;
    const int tl = threadIdx.x % TEAM;
    const int team = threadIdx.x / TEAM;
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < SW * 32; i += blockDim.x) s_cnt[i] = 0u;
    __syncthreads();
    const int64_t n_items = (pass == 1 ? (int64_t)A.n_hubs : A.n_hub_chunks) * A.nslices;
    for (int64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        int64_t item = it / A.nslices;      // chunk index (pass 1: hub index)
        const int slice = (int)(it - item * A.nslices);
        int h;
        if (pass == 1) {
            h = (int)item;
            item = __ldg(A.hub_chunk_base + h);
        } else {
            int lo = 0, hi = A.n_hubs - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__ldg(A.hub_chunk_base + mid) <= item) lo = mid; else hi = mid - 1;
            }
            h = lo;
            if (pass == 2 && (item == __ldg(A.hub_chunk_base + h) ||
                              *(volatile const uint32_t *)&A.hub_sat[(int64_t)h * A.nslices + slice]))
                continue;   // the first chunk ran in pass 1, or the slice is saturated
        }
        const int32_t v = h;   // hub rows are new ids 0 .. n_hubs-1
        if (sparse && !((A.bitmap[v >> 5] >> (v & 31)) & 1u)) continue;
        const int ws0 = slice * SW;        // first word of the slice
        const int w0 = ws0 + tl * V;
        WordCtx x[V];
        uint32_t need[V];
        uint32_t any_need = 0u;
        {
            const size_t off = (size_t)v * A.Wn + w0;
            Vec<V> a = ldg_vec<V>(A.cur + off);
            Vec<V> b{}, e{};
            if (P >= 2) b = ldg_vec<V>(A.cur + A.plane_words + off);
            if (P >= 3) e = ldg_vec<V>(A.cur + 2 * A.plane_words + off);
#pragma unroll
            for (int i = 0; i < V; ++i) {
                x[i] = word_ctx(A, w0 + i);
                need[i] = need_of<MODEL>(x[i].vm, a.w[i], b.w[i], e.w[i]);
                any_need |= need[i];
            }
        }
#pragma unroll
        for (int o = 1; o < TEAM; o <<= 1) any_need |= __shfl_xor_sync(0xffffffffu, any_need, o);
        if (!any_need) continue;   // identical in every team: they share the slice
        const int32_t rb = __ldg(A.rp + v), re = __ldg(A.rp + v + 1);
        int64_t arcb = 0;
        if constexpr (!ModelTraits<MODEL>::counts) arcb = (int64_t)__ldg(A.arc0 + v) - rb;
        const int64_t cidx = item - __ldg(A.hub_chunk_base + h);
        const int64_t beg = (int64_t)rb + cidx * A.hub_chunk;
        const int64_t end = min((int64_t)re, beg + A.hub_chunk);
        uint32_t c[V][B];
        uint32_t newly[V];
        uint64_t ic_thr[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            newly[i] = 0u;
            ic_thr[i] = ModelTraits<MODEL>::counts ? 0ull : ic_threshold(A, x[i].s, re - rb);
#pragma unroll
            for (int b = 0; b < B; ++b) c[i][b] = 0u;
        }
        if constexpr (ModelTraits<MODEL>::counts)
        {
            // the warps take the chunk's groups of 8 arcs per team in turn
            constexpr int per_warp = 8 * (32 / TEAM);
            const int off = (threadIdx.x >> 5) * per_warp;
            gather_counts<MODEL, V, B, TEAM, 32 / TEAM>(A, beg + off, (int32_t)(end - beg) - off, 8 * TPB, w0, lane, c);
        }
        else
            gather_arcs<MODEL, V>(A, beg + 4 * team, end, 4 * TPB, arcb, w0, need, ic_thr, x, newly);
#pragma unroll
        for (int o = TEAM; o < 32; o <<= 1) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                if constexpr (ModelTraits<MODEL>::counts) {
                    uint32_t d[B];
#pragma unroll
                    for (int b = 0; b < B; ++b) d[b] = __shfl_xor_sync(0xffffffffu, c[i][b], o);
                    add_sliced<B>(c[i], d);
                } else {
                    newly[i] |= __shfl_xor_sync(0xffffffffu, newly[i], o);
                }
            }
        }
        if constexpr (ModelTraits<MODEL>::counts) {
            // every team holds the warp's merged counts: the lanes' counts are read out
            // by all teams, each taking every (32/TEAM)-th lane
            constexpr int TPW = 32 / TEAM;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const int wsl = w0 + i - ws0;   // word within the slice
                for (int l = team % TPW; l < 32; l += TPW) {
                    const uint32_t k = lane_count<B>(c[i], l);
                    if (k) atomicAdd(&s_cnt[wsl * 32 + l], k);
                }
            }
        } else if (lane < TEAM) {   // team 0 of the warp holds the warp's live masks
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const int wsl = w0 + i - ws0;
                if (newly[i]) atomicOr(&s_cnt[wsl], newly[i]);
            }
        }
        if (A.prof_bytes && threadIdx.x == 0)
            atomicAdd(&A.prof_bytes[PK_HUB], row_bytes(SW, P, true, end - beg));
        __syncthreads();
        if constexpr (ModelTraits<MODEL>::saturates) {
            if (pass == 1) {
                // team 0 holds the slice's susceptible lanes (need); all of them at K_sat?
                bool sat = true;
                if (team == 0) {
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        const int32_t ks = __ldg(&A.sp[x[i].s].ksat);
                        uint32_t m = need[i];
                        if (m && ks == INT32_MAX) sat = false;
                        const int wsl = w0 + i - ws0;
                        while (m && sat) {
                            const int l = __ffs(m) - 1;
                            m &= m - 1;
                            if (s_cnt[wsl * 32 + l] < (uint32_t)ks) sat = false;
                        }
                    }
                }
                if (__syncthreads_and(sat) && threadIdx.x == 0)
                    A.hub_sat[(int64_t)h * A.nslices + slice] = 1u;
            }
        }
        uint32_t *slot = A.hub_scratch + (size_t)h * nl;
        if constexpr (ModelTraits<MODEL>::counts) {
            for (int i = threadIdx.x; i < SW * 32; i += blockDim.x) {
                const uint32_t xv = s_cnt[i];
                if (xv) {
                    atomicAdd(slot + ws0 * 32 + i, xv);
                    s_cnt[i] = 0u;
                }
            }
        } else {
            for (int i = threadIdx.x; i < SW; i += blockDim.x) {
                const uint32_t xv = s_cnt[i];
                if (xv) {
                    atomicOr(slot + ws0 + i, xv);
                    s_cnt[i] = 0u;
                }
            }
        }
        __syncthreads();
    }
}

// Hub rows, phase 2: one warp per hub row; lane l decides word g0 + l.  The per-lane
// counts are re-sliced with ballots (32-bit counters), the scratch slot is cleared.
template <int MODEL>
__global__ void __launch_bounds__(kBlock) k_hub_finalize(StepArgs A) {
    extern __shared__ int32_t s_lane[];
    __shared__ unsigned long long s_pc[kPC * kMaxSets];
    constexpr int P = ModelTraits<MODEL>::planes;
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    const bool sparse = *(volatile const int32_t *)&C->sparse != 0;
    const int nl = A.Wn * 32;
    const bool lanes_on = A.lane_cnt != nullptr;
    const bool build = list_wanted(A);
    if (lanes_on)
        for (int i = threadIdx.x; i < A.np * nl; i += blockDim.x) s_lane[i] = 0;
    set_acc_zero(s_pc, A.S);
    const int lane = threadIdx.x & 31;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int list_slot = A.k & 1;
    Accum acc;
    for (int64_t h = gwarp; h < A.n_hubs; h += nwarps) {
        const int32_t v = (int32_t)h;
        const uint32_t node = node_of(A, v);
        const bool cand = !sparse || ((A.bitmap[v >> 5] >> (v & 31)) & 1u);
        uint32_t fl = 0u;
        if (cand) {
            const int32_t d = __ldg(A.rp + v + 1) - __ldg(A.rp + v);
            uint32_t *slot = A.hub_scratch + (size_t)h * nl;
            for (int g0 = 0; g0 < A.Wn; g0 += 32) {
                const int w = g0 + lane;
                const bool act = w < A.Wn;
                uint32_t c[32];
#pragma unroll
                for (int b = 0; b < 32; ++b) c[b] = 0u;
                uint32_t newly = 0u;
                if constexpr (ModelTraits<MODEL>::counts) {
                    const int nw = min(32, A.Wn - g0);
                    for (int ww = 0; ww < nw; ++ww) {
                        const uint32_t kv = slot[(g0 + ww) * 32 + lane];
                        if (kv) slot[(g0 + ww) * 32 + lane] = 0u;
#pragma unroll
                        for (int b = 0; b < 32; ++b) {
                            const uint32_t bb = __ballot_sync(0xffffffffu, (kv >> b) & 1u);
                            if (lane == ww) c[b] = bb;
                        }
                    }
                } else {
                    if (act) {
                        newly = slot[w];
                        if (newly) slot[w] = 0u;
                    }
                }
                if (act) {
                    const size_t off = (size_t)v * A.Wn + w;
                    const uint32_t s0 = __ldg(A.cur + off);
                    const uint32_t s1 = P >= 2 ? __ldg(A.cur + A.plane_words + off) : 0u;
                    const uint32_t s2 = P >= 3 ? __ldg(A.cur + 2 * A.plane_words + off) : 0u;
                    const WordCtx x = word_ctx(A, w);
                    const WordOut o = update_word<MODEL, 32>(A, node, x, s0, s1, s2, d, c, newly & x.vm & ~s0);
                    A.nxt[off] = o.n0;
                    if (P >= 2) A.nxt[A.plane_words + off] = o.n1;
                    if (P >= 3) A.nxt[2 * A.plane_words + off] = o.n2;
                    set_acc_add(s_pc, x.s, (long long)__popc(o.n0) - __popc(s0),
                                (long long)__popc(o.n1) - __popc(s1), (long long)__popc(o.n2) - __popc(s2));
                    if (lanes_on) {
                        lane_deltas(s_lane, w, s0, o.n0);
                        if (P >= 2) lane_deltas(s_lane + nl, w, s1, o.n1);
                        if (P >= 3) lane_deltas(s_lane + 2 * nl, w, s2, o.n2);
                    }
                    fl |= word_flags<MODEL>(o, s0, s1, s2);
                }
            }
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
        if (A.hub_sat)
            for (int sl = lane; sl < A.nslices; sl += 32) A.hub_sat[h * A.nslices + sl] = 0u;
        const bool want = cand && lane == 0 && fl != 0u;
        if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
        if (A.prof_bytes && cand && lane == 0)
            acc.bytes += row_bytes(A.Wn, P, false, 0) + 2ull * 4ull * 32ull * (unsigned long long)A.Wn;
        list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
        if (sparse && cand && lane == 0) atomicAnd(&A.bitmap[v >> 5], ~(1u << (v & 31)));
    }
    flush_accum(A, acc, list_slot, PK_HUBFIN);
    set_acc_flush(A, s_pc);
    if (lanes_on) flush_lanes(A, s_lane, nl);
}

// Rows with 1..3 in-arcs, and the rows without in-arcs whose state can change (listed by
// the step-0 scan: seeds, or imported rows with infected / newly active lanes; every
// other row without in-arcs keeps its state for the whole run and is never touched),
// dense steps only (on frontier steps such rows come through the candidate lists of
// k_rows).  Most rows of a power-law graph
// are of this kind and carry little gather work, so the cost is the chain of dependent
// loads per row: one THREAD per item (a slice of SWL <= 8 words of one row) keeps four
// to eight times as many rows in flight per SM as a team per row.
// lane_body (SWIR): the thread loads its own words and the (at most three) sources' words at
// once, stages them in shared memory, and then decides its words one at a time through a
// single, non-unrolled copy of the per-word update (counts of at most 3 need 2-bit counters).
// lane_tile (the other models): the same rows through the warp tile.
constexpr int kLaneMaxDeg = 3;
template <int SWL, int NP>
struct LaneStage {
    uint32_t v[NP + 3][SWL][kBlock];   // own planes, then the sources' words (x0, x1, x2)
};

template <int MODEL, int SWL>
__device__ __forceinline__ void lane_body(const StepArgs &A, uint8_t *smem, int32_t *s_lane, unsigned long long *s_pc) {
    static_assert(!ModelTraits<MODEL>::tiled && ModelTraits<MODEL>::planes == 3, "the other models go through the warp tile");
    constexpr int P = 3;
    LaneStage<SWL, P> &st = *reinterpret_cast<LaneStage<SWL, P> *>(smem);
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    if (*(volatile const int32_t *)&C->sparse) return;
    const int nsl = A.Wn / SWL;
    const int64_t n_rows = (int64_t)A.n_lane + *(volatile const uint32_t *)&C->d0_n;
    const int64_t nitems = n_rows * nsl;
    if (nitems == 0) return;
    const int nl = A.Wn * 32;
    const bool lanes_on = A.lane_cnt != nullptr;
    const bool build = list_wanted(A);
    if (lanes_on)
        for (int i = threadIdx.x; i < A.np * nl; i += blockDim.x) s_lane[i] = 0;
    set_acc_zero(s_pc, A.S);
    const int list_slot = A.k & 1;
    const int tid = threadIdx.x;
    const uint32_t *src_plane = A.cur + (size_t)ModelTraits<MODEL>::src_plane * A.plane_words;
    Accum acc;
    int cur_s = -1;           // set of the plane-count deltas not yet flushed
    int32_t dd0 = 0, dd1 = 0, dd2 = 0;
    for (int64_t item = (int64_t)blockIdx.x * blockDim.x + tid; item - tid < nitems;
         item += (int64_t)gridDim.x * blockDim.x) {
        const bool has = item < nitems;
        int32_t v = 0, d = 0;            // v: new id
        uint32_t node = 0u;              // Philox subject
        int w0 = 0;
        uint32_t busy = 0u;
        if (has) {
            const int64_t r = div_slices(item, nsl, nitems);
            w0 = (int)(item - r * nsl) * SWL;
            int4 e;
            if (r < A.n_lane) {
                e = __ldg(A.lane_tab + r);   // the node and its sources in one entry
                v = A.r_lane + (int32_t)r;
            } else {
                v = A.d0_list[r - A.n_lane];
                e = make_int4((int32_t)node_of(A, v), -1, -1, -1);
            }
            node = (uint32_t)e.x;
            const int32_t u[kLaneMaxDeg] = {e.y, e.z, e.w};
            d = (e.y >= 0) + (e.z >= 0) + (e.w >= 0);
            const size_t off = (size_t)v * A.Wn + w0;
            // own words and sources' words, 4 (or fewer) words per load; `busy` records
            // whether any lane can change at this step (an infected lane to recover, or a
            // lane that can change with a set source lane in its in-arcs)
#pragma unroll
            for (int q = 0; q < SWL; q += (SWL < 4 ? SWL : 4)) {
                constexpr int VL = SWL < 4 ? SWL : 4;
                const Vec<VL> a = ldg_vec<VL>(A.cur + off + q);
                const Vec<VL> bb = ldg_vec<VL>(A.cur + A.plane_words + off + q);
                const Vec<VL> ee = ldg_vec<VL>(A.cur + 2 * A.plane_words + off + q);
                uint32_t xs[VL];
#pragma unroll
                for (int i = 0; i < VL; ++i) {
                    st.v[0][q + i][tid] = a.w[i];
                    st.v[1][q + i][tid] = bb.w[i];
                    st.v[2][q + i][tid] = ee.w[i];
                    xs[i] = 0u;
                }
#pragma unroll
                for (int j = 0; j < kLaneMaxDeg; ++j) {
                    Vec<VL> x{};
                    if (u[j] >= 0) x = ldg_vec<VL>(src_plane + (size_t)u[j] * A.Wn + w0 + q);
#pragma unroll
                    for (int i = 0; i < VL; ++i) {
                        st.v[P + j][q + i][tid] = x.w[i];
                        xs[i] |= x.w[i];
                    }
                }
#pragma unroll
                for (int i = 0; i < VL; ++i) {
                    // an infectious lane may recover, and a set source lane can change another
                    busy |= a.w[i] | (need_of<MODEL>(~0u, a.w[i], bb.w[i], ee.w[i]) & xs[i]);
                }
            }
        }
        uint32_t fl = 0u;
        if (has && !busy) {
            // no lane can change: the next state is this one
            const size_t off = (size_t)v * A.Wn + w0;
#pragma unroll
            for (int q = 0; q < SWL; q += (SWL < 4 ? SWL : 4)) {
                constexpr int VL = SWL < 4 ? SWL : 4;
#pragma unroll
                for (int pl = 0; pl < P; ++pl) {
                    uint32_t nw[VL];
#pragma unroll
                    for (int i = 0; i < VL; ++i) nw[i] = st.v[pl][q + i][tid];
                    st_vec<VL>(A.nxt + pl * A.plane_words + off + q, nw);
                }
            }
        } else if (has) {
#pragma unroll 1
            for (int i = 0; i < SWL; ++i) {
                const WordCtx x = word_ctx(A, w0 + i);
                const uint32_t s0 = st.v[0][i][tid];
                const uint32_t s1 = st.v[1][i][tid];
                const uint32_t s2 = st.v[2][i][tid];
                const uint32_t x0 = st.v[P][i][tid], x1 = st.v[P + 1][i][tid], x2 = st.v[P + 2][i][tid];
                const uint32_t need = need_of<MODEL>(x.vm, s0, s1, s2);
                // counts of set source lanes (at most 3): two bit-planes
                const uint32_t c[2] = {(x0 ^ x1 ^ x2) & need, ((x0 & x1) | (x2 & (x0 ^ x1))) & need};
                const WordOut o = update_word<MODEL, 2>(A, node, x, s0, s1, s2, d, c, 0u);
                st.v[0][i][tid] = o.n0;
                st.v[1][i][tid] = o.n1;
                st.v[2][i][tid] = o.n2;
                if (x.s != cur_s) {
                    if (cur_s >= 0) set_acc_add(s_pc, cur_s, dd0, dd1, dd2);
                    cur_s = x.s;
                    dd0 = dd1 = dd2 = 0;
                }
                dd0 += __popc(o.n0) - __popc(s0);
                dd1 += __popc(o.n1) - __popc(s1);
                dd2 += __popc(o.n2) - __popc(s2);
                if (lanes_on) {
                    lane_deltas(s_lane, w0 + i, s0, o.n0);
                    lane_deltas(s_lane + nl, w0 + i, s1, o.n1);
                    lane_deltas(s_lane + 2 * nl, w0 + i, s2, o.n2);
                }
                fl |= word_flags<MODEL>(o, s0, s1, s2);
            }
            const size_t off = (size_t)v * A.Wn + w0;
#pragma unroll
            for (int q = 0; q < SWL; q += (SWL < 4 ? SWL : 4)) {
                constexpr int VL = SWL < 4 ? SWL : 4;
#pragma unroll
                for (int pl = 0; pl < P; ++pl) {
                    uint32_t nw[VL];
#pragma unroll
                    for (int i = 0; i < VL; ++i) nw[i] = st.v[pl][q + i][tid];
                    st_vec<VL>(A.nxt + pl * A.plane_words + off + q, nw);
                }
            }
        }
        const bool want = has && fl != 0u;
        if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
        if (A.prof_bytes && has) acc.bytes += row_bytes(SWL, P, d > 0, d);
        list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
    }
    set_acc_add_warp(s_pc, cur_s, dd0, dd1, dd2);
    flush_accum(A, acc, list_slot, PK_LANE);
    set_acc_flush(A, s_pc);
    if (lanes_on) flush_lanes(A, s_lane, nl);
}

// The same rows through the warp tile: 32 row slices of SWL words per warp.
template <int MODEL, int SWL>
struct LaneShape {
    static constexpr bool counts = ModelTraits<MODEL>::counts;
    static constexpr int B = counts ? 2 : 1;
    static constexpr int NARC = counts ? 0 : 256;
    using T = Tile<B, ModelTraits<MODEL>::fixed_draws, 32 * SWL, 32, NARC>;
    static constexpr size_t bytes = sizeof(T) * (kBlock / 32);
};

template <int MODEL, int SWL>
__device__ __forceinline__ void lane_tile(const StepArgs &A, uint8_t *smem, int32_t *s_lane, unsigned long long *s_pc) {
    using S = LaneShape<MODEL, SWL>;
    constexpr int P = ModelTraits<MODEL>::planes;
    constexpr int NF = ModelTraits<MODEL>::fixed_draws;
    constexpr int VL = SWL < 4 ? SWL : 4;
    constexpr bool COUNTS = ModelTraits<MODEL>::counts;
    const Ctl *C = A.ctl;
    if (*(volatile const int32_t *)&C->stop) return;
    if (*(volatile const int32_t *)&C->sparse) return;
    const int nsl = A.Wn / SWL;
    const int64_t n_rows = (int64_t)A.n_lane + *(volatile const uint32_t *)&C->d0_n;
    const int64_t nitems = n_rows * nsl;
    if (nitems == 0) return;
    const int nl = A.Wn * 32;
    const bool lanes_on = A.lane_cnt != nullptr;
    const bool build = list_wanted(A);
    if (lanes_on)
        for (int i = threadIdx.x; i < A.np * nl; i += blockDim.x) s_lane[i] = 0;
    set_acc_zero(s_pc, A.S);
    typename S::T &T = reinterpret_cast<typename S::T *>(smem)[threadIdx.x >> 5];
    const int list_slot = A.k & 1;
    const int lane = threadIdx.x & 31;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t *src_plane = A.cur + (size_t)ModelTraits<MODEL>::src_plane * A.plane_words;
    Accum acc;
    int cur_s = -1;           // set of the plane-count deltas not yet flushed
    int32_t dd0 = 0, dd1 = 0, dd2 = 0;
    auto ctx = [&T](int slot, uint32_t &node, int &w) -> int {
        node = T.node[slot & 31];
        w = T.w0[slot & 31] + (slot >> 5);
        return COUNTS ? T.row[slot & 31] : (slot & 31);
    };
    for (int64_t base = gwarp * 32; base < nitems; base += nwarps * 32) {
        const int64_t item = base + lane;
        const bool has = item < nitems;
        int nq = 0, na = 0;
        int nf[2] = {0, 0};
        int32_t v = 0, beg = 0, d = 0;   // v: new id
        int w0 = 0;
        int4 e4 = make_int4(0, -1, -1, -1);
        if (has) {
            const int64_t r = div_slices(item, nsl, nitems);
            w0 = (int)(item - r * nsl) * SWL;
            if (r < A.n_lane) {
                e4 = __ldg(A.lane_tab + r);   // the node and its sources in one entry
                v = A.r_lane + (int32_t)r;
            } else {
                v = A.d0_list[r - A.n_lane];
                e4.x = (int32_t)node_of(A, v);
            }
            d = (e4.y >= 0) + (e4.z >= 0) + (e4.w >= 0);
            if (!COUNTS && d > 0) beg = __ldg(A.arc0 + v);   // arc positions key the draws
        }
        T.row[lane] = has ? v : -1;
        T.node[lane] = (uint32_t)e4.x;
        T.w0[lane] = w0;
        if (MODEL == FSGP_IC) T.thr[lane] = 0xffffffffu / (uint32_t)max(d, 1);
        __syncwarp();
        const size_t off = (size_t)v * A.Wn + w0;
        const int32_t u[kLaneMaxDeg] = {e4.y, e4.z, e4.w};
#pragma unroll
        for (int q = 0; q < SWL; q += VL) {
            Vec<VL> a{}, b{}, ee{}, x[kLaneMaxDeg];
            if (has) {
                a = ldg_vec<VL>(A.cur + off + q);
                if (P >= 2 && !ModelTraits<MODEL>::cascade) b = ldg_vec<VL>(A.cur + A.plane_words + off + q);
                if (P >= 3) ee = ldg_vec<VL>(A.cur + 2 * A.plane_words + off + q);
            }
#pragma unroll
            for (int j = 0; j < kLaneMaxDeg; ++j) {
                x[j] = Vec<VL>{};
                if (u[j] >= 0) x[j] = ldg_vec<VL>(src_plane + (size_t)u[j] * A.Wn + w0 + q);
            }
#pragma unroll
            for (int i = 0; i < VL; ++i) {
                const int slot = (q + i) * 32 + lane;
                const uint32_t vm = has ? word_ctx(A, w0 + q + i).vm : 0u;
                const uint32_t need = need_of<MODEL>(vm, a.w[i], b.w[i], ee.w[i]);
                const uint32_t x0 = x[0].w[i], x1 = x[1].w[i], x2 = x[2].w[i];
                if constexpr (COUNTS) {
                    const uint32_t c0 = (x0 ^ x1 ^ x2) & need;
                    const uint32_t c1 = ((x0 & x1) | (x2 & (x0 ^ x1))) & need;
                    T.c[0][slot] = c0;
                    T.c[1][slot] = c1;
                    queue_push(T.qc, nq, (c0 | c1) != 0u, slot, lane);
                } else {
                    T.c[0][slot] = 0u;
                    const uint32_t xs[kLaneMaxDeg] = {x0 & need, x1 & need, x2 & need};
#pragma unroll
                    for (int j = 0; j < kLaneMaxDeg; ++j) {
                        const unsigned m = __ballot_sync(0xffffffffu, xs[j] != 0u);
                        if (m == 0u) continue;
                        if (na > S::NARC - 32) {
                            __syncwarp();
                            draw_arc_items<MODEL, false>(A, T, na, lane, ctx);
                            na = 0;
                        }
                        if (xs[j]) {
                            const int at = na + __popc(m & ((1u << lane) - 1u));
                            T.arc_slot[at] = (uint16_t)slot;
                            T.arc_pos[at] = (uint32_t)(beg + j);
                            T.arc_eq[at] = xs[j];
                        }
                        na += __popc(m);
                    }
                }
                if constexpr (NF >= 1) {
                    const uint32_t f0 = (A.fixed_on & 1) ? fixed_lanes<MODEL>(0, vm, a.w[i], b.w[i], ee.w[i]) : 0u;
                    T.f[0][slot] = f0;
                    queue_push(T.qf[0], nf[0], f0 != 0u, slot, lane);
                }
                if constexpr (NF >= 2) {
                    const uint32_t f1 = (A.fixed_on & 2) ? fixed_lanes<MODEL>(1, vm, a.w[i], b.w[i], ee.w[i]) : 0u;
                    T.f[1][slot] = f1;
                    queue_push(T.qf[1], nf[1], f1 != 0u, slot, lane);
                }
            }
        }
        draw_tile<MODEL, S::B, false>(A, T, nq, nf, na, lane, ctx);
        __syncwarp();
        uint32_t fl = 0u;
        if (has) {
#pragma unroll
            for (int q = 0; q < SWL; q += VL) {
                const Vec<VL> a = ldg_vec<VL>(A.cur + off + q);
                Vec<VL> b{}, ee{};
                if (P >= 2) b = ldg_vec<VL>(A.cur + A.plane_words + off + q);
                if (P >= 3) ee = ldg_vec<VL>(A.cur + 2 * A.plane_words + off + q);
                uint32_t n0[VL], n1[VL], n2[VL];
#pragma unroll
                for (int i = 0; i < VL; ++i) {
                    const int slot = (q + i) * 32 + lane;
                    const WordOut o = next_word<MODEL>(a.w[i], b.w[i], ee.w[i], T.c[0][slot], T.template fixed<0>(slot),
                                                       T.template fixed<1>(slot));
                    n0[i] = o.n0;
                    n1[i] = o.n1;
                    n2[i] = o.n2;
                    const int s = (w0 + q + i) >> A.ws_shift;
                    if (s != cur_s) {
                        if (cur_s >= 0) set_acc_add(s_pc, cur_s, dd0, dd1, dd2);
                        cur_s = s;
                        dd0 = dd1 = dd2 = 0;
                    }
                    dd0 += __popc(o.n0) - __popc(a.w[i]);
                    if (P >= 2) dd1 += __popc(o.n1) - __popc(b.w[i]);
                    if (P >= 3) dd2 += __popc(o.n2) - __popc(ee.w[i]);
                    if (lanes_on) {
                        lane_deltas(s_lane, w0 + q + i, a.w[i], o.n0);
                        if (P >= 2) lane_deltas(s_lane + nl, w0 + q + i, b.w[i], o.n1);
                        if (P >= 3) lane_deltas(s_lane + 2 * nl, w0 + q + i, ee.w[i], o.n2);
                    }
                    fl |= word_flags<MODEL>(o, a.w[i], b.w[i], ee.w[i]);
                }
                st_vec<VL>(A.nxt + off + q, n0);
                if (P >= 2) st_vec<VL>(A.nxt + A.plane_words + off + q, n1);
                if (P >= 3) st_vec<VL>(A.nxt + 2 * A.plane_words + off + q, n2);
            }
        }
        const bool want = has && fl != 0u;
        if (want && (fl & 1u)) acc.push_deg += out_degree(A, v);
        if (A.prof_bytes && has) acc.bytes += row_bytes(SWL, P, d > 0, d);
        list_append(A, build, want, (int32_t)((uint32_t)v | ((fl & 1u) ? kPushBit : 0u)), list_slot);
        __syncwarp();   // the next tile overwrites the slots
    }
    set_acc_add_warp(s_pc, cur_s, dd0, dd1, dd2);
    flush_accum(A, acc, list_slot, PK_LANE);
    set_acc_flush(A, s_pc);
    if (lanes_on) flush_lanes(A, s_lane, nl);
}

// Bytes of the staging area or of the warps' tiles.
template <int MODEL, int SWL>
constexpr size_t kLaneSmem = ModelTraits<MODEL>::tiled ? LaneShape<MODEL, SWL>::bytes
                                                       : sizeof(LaneStage<SWL, ModelTraits<MODEL>::planes>);

template <int MODEL, int SWL>
__global__ void __launch_bounds__(kBlock, ModelTraits<MODEL>::tiled ? 3 : 1) k_rows_lane(StepArgs A) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ unsigned long long s_pc[kPC * kMaxSets];
    int32_t *s_lane = reinterpret_cast<int32_t *>(s_dyn + kLaneSmem<MODEL, SWL>);
    if constexpr (ModelTraits<MODEL>::tiled) lane_tile<MODEL, SWL>(A, s_dyn, s_lane, s_pc);
    else lane_body<MODEL, SWL>(A, s_dyn, s_lane, s_pc);
}

// Resident CTAs per SM of a kernel with `tile` bytes of dynamic shared memory (`smem` with
// the per-lane counters of this run).  The kernel also asks for no more of the SM's 256 KB
// than those CTAs' shared memory: the default takes the largest carve-out as soon as one
// more CTA would fit by shared memory alone, and what is left as L1 (28 KB) then has too
// few lines for the gathered rows in flight (random 32-byte rows out of L2: 287e9 rows/s
// with 60 KB of L1 or more, 153e9 with 28 KB).  The kernel's own preference is that of runs
// without per-lane counters, the same every time, since host threads of a batch may set it
// concurrently; a run with counters asks for its share at each launch (RowFit::carve; with
// the kernel's preference one CTA of two stayed out: SIR with per-realization counts, R = 1000,
// T = 40, BA n = 250k: 36.1 and 24.1 ms; n = 20k: 4.9 and 3.2; SIS, R-MAT n = 1M, T = 20: 26.5 and
// 19.5).
inline RowFit resident_ctas(const void *kern, size_t smem, size_t tile) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(tile + kLaneCounterBytes));
    int z = 1, z0 = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&z, kern, kBlock, smem + tile);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&z0, kern, kBlock, tile);
    RowFit f{std::max(z, 1), 0};
    cudaFuncAttributes at{};
    int per_sm = 0, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaFuncGetAttributes(&at, kern) == cudaSuccess &&
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess && per_sm > 0) {
        auto percent = [&](int ctas, size_t dynamic) {   // 1 KB of each CTA is the system's
            const size_t need = (size_t)ctas * (dynamic + at.sharedSizeBytes + 1024);
            return (int)std::min<size_t>(100, (need * 100 + per_sm - 1) / (size_t)per_sm);
        };
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, percent(std::max(z0, 1), tile));
        if (smem) f.carve = percent(f.ctas, smem + tile);
    }
    return f;
}

// The same, asked once per kernel, device and size in a row (a small graph's run is shorter
// than a handful of driver queries are cheap).
template <auto Kern>
RowFit occupancy_one(size_t smem, size_t tile) {
    static std::atomic<uint64_t> last{0};   // 1 << 63 | device << 48 | smem << 16 | carve << 8 | CTAs
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 1 << 15) return resident_ctas((const void *)Kern, smem, tile);
    const uint64_t key = 1ull << 63 | (uint64_t)dev << 48 | (uint64_t)smem << 16;
    const uint64_t seen = last.load(std::memory_order_acquire);
    if ((seen & ~0xffffull) == key) return RowFit{(int)(seen & 0xff), (int)(seen >> 8 & 0xff)};
    const RowFit f = resident_ctas((const void *)Kern, smem, tile);
    last.store(key | (uint64_t)f.carve << 8 | (uint64_t)f.ctas, std::memory_order_release);
    return f;
}

// Launch of a row kernel; carve: the share of the SM's memory asked for as shared memory, in
// percent (0: the kernel's own preference).
template <class... P, class... Q>
void launch_row_kernel(void (*kern)(P...), int grid, size_t smem, int carve, cudaStream_t s, Q... args) {
    if (carve == 0) {
        kern<<<grid, kBlock, smem, s>>>(args...);
        return;
    }
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at.val.sharedMemCarveout = (unsigned)carve;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3(kBlock);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kern, args...);
}

// Widest slice of the one-thread-per-row kernel: the staging area of the three-plane
// models (planes + 3 sources, SWL words, 256 threads) grows past 48 KB with 8 words.
template <int MODEL>
constexpr int lane_swl_max() { return ModelTraits<MODEL>::planes >= 3 ? 4 : 8; }

template <int MODEL>
int launch_rows_lane(const StepArgs &A, int swl, int grid, size_t smem, int carve, cudaStream_t s) {
    switch (swl) {
        case 1: launch_row_kernel(k_rows_lane<MODEL, 1>, grid, smem + kLaneSmem<MODEL, 1>, carve, s, A); break;
        case 2: launch_row_kernel(k_rows_lane<MODEL, 2>, grid, smem + kLaneSmem<MODEL, 2>, carve, s, A); break;
        case 4: launch_row_kernel(k_rows_lane<MODEL, 4>, grid, smem + kLaneSmem<MODEL, 4>, carve, s, A); break;
        case 8:
            if constexpr (lane_swl_max<MODEL>() >= 8) {
                launch_row_kernel(k_rows_lane<MODEL, 8>, grid, smem + kLaneSmem<MODEL, 8>, carve, s, A);
                break;
            }
            return fail(FSGP_EINVAL, "lane kernel slice width");
        default: return fail(FSGP_EINVAL, "lane kernel slice width");
    }
    return FSGP_OK;
}

template <int MODEL, int SWL>
RowFit occupancy_lane_w(size_t smem) {
    return occupancy_one<k_rows_lane<MODEL, SWL>>(smem, kLaneSmem<MODEL, SWL>);
}

template <int MODEL>
RowFit occupancy_lane(int swl, size_t smem) {
    switch (swl) {
        case 1: return occupancy_lane_w<MODEL, 1>(smem);
        case 2: return occupancy_lane_w<MODEL, 2>(smem);
        case 4: return occupancy_lane_w<MODEL, 4>(smem);
        default:
            if constexpr (lane_swl_max<MODEL>() >= 8) return occupancy_lane_w<MODEL, 8>(smem);
            else return occupancy_lane_w<MODEL, 4>(smem);
    }
}

// ------------------------------------------------------------------------- launch

template <int MODEL, int V, int TEAM>
int launch_rows_vt(const StepArgs &A, const StepLaunch &L, cudaStream_t s) {
    Prof *pr = L.prof;
    if (L.fused) {
        if (pr) pr->start(PK_SMALL, s);
        launch_row_kernel(k_rows_fused<MODEL, V, TEAM>, L.grid_mid + L.grid_small,
                          L.smem_lanes + FusedBytes<MODEL, V, TEAM>, L.carve_fused, s, A, L.grid_mid);
        if (pr) pr->stop(s);
        return FSGP_OK;
    }
    if (L.have_hub) {
        if (pr) pr->start(PK_HUB, s);
        if (A.hub_sat) {
            k_hub_chunks<MODEL, V, TEAM><<<L.grid_hub, kBlock, 0, s>>>(A, 1);
            k_hub_chunks<MODEL, V, TEAM><<<L.grid_hub, kBlock, 0, s>>>(A, 2);
        } else {
            k_hub_chunks<MODEL, V, TEAM><<<L.grid_hub, kBlock, 0, s>>>(A, 0);
        }
        if (pr) { pr->stop(s); pr->start(PK_HUBFIN, s); }
        k_hub_finalize<MODEL><<<L.grid_fin, kBlock, L.smem_lanes, s>>>(A);
        if (pr) pr->stop(s);
    }
    if (L.have_mid) {
        if (pr) pr->start(PK_MID, s);
        launch_row_kernel(k_rows<MODEL, V, TEAM, true>, L.grid_mid,
                          L.smem_lanes + TileBytes<MODEL, V, TEAM, true, kSmallBits>, L.carve_mid, s, A, 1);
        if (pr) pr->stop(s);
    }
    if (L.have_small) {
        if (pr) pr->start(PK_SMALL, s);
        launch_row_kernel(k_rows<MODEL, V, TEAM, false>, L.grid_small,
                          L.smem_lanes + TileBytes<MODEL, V, TEAM, false, kSmallBits>, L.carve_small, s, A, 0);
        if (pr) pr->stop(s);
    }
    if (L.have_small4) {
        if (pr) pr->start(PK_SMALL4, s);
        launch_row_kernel(k_rows<MODEL, V, TEAM, false, 4>, L.grid_small4,
                          L.smem_lanes + TileBytes<MODEL, V, TEAM, false, 4>, L.carve_small4, s, A, 3);
        if (pr) pr->stop(s);
    }
    if (L.have_lane) {
        if (pr) pr->start(PK_LANE, s);
        const int rc = launch_rows_lane<MODEL>(A, L.swl, L.grid_lane, L.smem_lanes, L.carve_lane, s);
        if (pr) pr->stop(s);
        if (rc) return rc;
    }
    return FSGP_OK;
}

template <int MODEL, int V, int TEAM>
void occupancy_vt(size_t smem, RowOccupancy *o) {
    if (o->fused_only) {
        o->fused = occupancy_one<k_rows_fused<MODEL, V, TEAM>>(smem, FusedBytes<MODEL, V, TEAM>);
        return;
    }
    o->hub = occupancy_one<k_hub_chunks<MODEL, V, TEAM>>(0, 0);
    o->small4 = occupancy_one<k_rows<MODEL, V, TEAM, false, 4>>(smem, TileBytes<MODEL, V, TEAM, false, 4>);
    o->small = occupancy_one<k_rows<MODEL, V, TEAM, false>>(smem, TileBytes<MODEL, V, TEAM, false, kSmallBits>);
    o->mid = occupancy_one<k_rows<MODEL, V, TEAM, true>>(smem, TileBytes<MODEL, V, TEAM, true, kSmallBits>);
}

#define FSGP_VT_SWITCH(MACRO)                          \
    switch (V * 100 + TEAM) {                          \
        case 101: MACRO(1, 1); break;                  \
        case 102: MACRO(1, 2); break;                  \
        case 104: MACRO(1, 4); break;                  \
        case 108: MACRO(1, 8); break;                  \
        case 116: MACRO(1, 16); break;                 \
        case 132: MACRO(1, 32); break;                 \
        case 201: MACRO(2, 1); break;                  \
        case 401: MACRO(4, 1); break;                  \
        case 402: MACRO(4, 2); break;                  \
        case 404: MACRO(4, 4); break;                  \
        case 408: MACRO(4, 8); break;                  \
        case 416: MACRO(4, 16); break;                 \
        case 432: MACRO(4, 32); break;                 \
        case 202: MACRO(2, 2); break;                  \
        case 204: MACRO(2, 4); break;                  \
        case 208: MACRO(2, 8); break;                  \
        case 216: MACRO(2, 16); break;                 \
        case 232: MACRO(2, 32); break;                 \
        default: return fail(FSGP_EINVAL, "unsupported words-per-thread / team combination"); \
    }

template <int MODEL>
int launch_rows(const StepArgs &A, const StepLaunch &L, cudaStream_t s) {
    const int V = L.V, TEAM = L.TEAM;
#define FSGP_L(v_, t_) launch_rows_vt<MODEL, v_, t_>(A, L, s)
    FSGP_VT_SWITCH(FSGP_L)
#undef FSGP_L
    return FSGP_OK;
}

// Only the CTA-split pair (chunks, then finalize), for callers that treat every row as
// a split row.
template <int MODEL, int V, int TEAM>
int launch_split_vt(const StepArgs &A, int grid_chunks, int grid_fin, cudaStream_t s) {
    k_hub_chunks<MODEL, V, TEAM><<<grid_chunks, kBlock, 0, s>>>(A, 0);
    k_hub_finalize<MODEL><<<grid_fin, kBlock, 0, s>>>(A);
    return FSGP_OK;
}

template <int MODEL>
int launch_split_rows(const StepArgs &A, int V, int TEAM, int grid_chunks, int grid_fin,
                      cudaStream_t s) {
#define FSGP_S(v_, t_) launch_split_vt<MODEL, v_, t_>(A, grid_chunks, grid_fin, s)
    FSGP_VT_SWITCH(FSGP_S)
#undef FSGP_S
    return FSGP_OK;
}

template <int MODEL>
int occupancy_rows(int V, int TEAM, size_t smem, RowOccupancy *o) {
#define FSGP_O(v_, t_) occupancy_vt<MODEL, v_, t_>(smem, o)
    FSGP_VT_SWITCH(FSGP_O)
#undef FSGP_O
    if (!o->fused_only) o->lane = occupancy_lane<MODEL>(o->swl, smem);
    return FSGP_OK;
}

// Cooperative launch of the persistent step loop (one word per thread).  The grid is what
// can be resident at once, at most the launched step's (grid_mid + grid_small CTAs), shared
// out between the two row classes in the same proportion; *grid_out gets the grid used.
// FSGP_EUNSUPPORTED: it does not fit (the caller runs the launched loop instead).
template <int MODEL, int TEAM, int WB = kWideBits, int AG = 1>
int launch_persist_t(const StepArgs &A, const PersistArgs &Q, int grid_mid, int grid_small, size_t smem, int sm_count,
                     cudaStream_t s, int *grid_out) {
    // SWIR, decided in place, pays for 16-bit counters in its chain, and at one or two words a row
    // gets two teams where all rows are short and fit at once, on as few CTAs as that takes
    // (T = 40; most rows a warp with 16-bit counters, and now: ER n = 1200, R = 32: 423 and
    // 376 us; n = 2000, R = 64: 454 and 405; n = 10k, R = 650: 979 and 824.  Two teams on every
    // row of BA n = 2000, R = 32: 568, two classes 418; of ER n = 500k, R = 64: 2376 and 1780).
    // The tiles gain from 8-bit counters where rows are short (ER n = 1289, R = 458, SEIR 721 and
    // 697 us; n = 2000, R = 64, LT 522 and 490) and few (n = 10k, R = 64, SIR 554 and 557), and lose
    // where they are not short (BA n = 1752, R = 582, SIS 1543 and 1666).
    constexpr int per_cta = kBlock / (TEAM * (AG > 1 ? AG : 2));   // rows of a CTA
    const int64_t team_ctas = ((int64_t)A.n * A.nslices + per_cta - 1) / per_cta;
    if constexpr (ModelTraits<MODEL>::counts && WB != kSmallBits) {
        if (ModelTraits<MODEL>::tiled ? Q.max_deg < 64 && grid_mid > 0 && (int64_t)A.n * A.nslices <= 48 * sm_count
                                      : Q.max_deg < 1 << kSmallBits) {
            if constexpr (!ModelTraits<MODEL>::tiled && TEAM <= 2)
                if (Q.max_deg < 64 && team_ctas <= 2 * sm_count)
                    return launch_persist_t<MODEL, TEAM, kSmallBits, 2>(A, Q, 0, (int)team_ctas, smem, sm_count, s, grid_out);
            return launch_persist_t<MODEL, TEAM, kSmallBits>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        }
    }
    StepArgs a = A;
    PersistArgs q = Q;
    if constexpr (AG > 1) {   // every row a team row
        a.r_small = 0;
        a.n_small = A.n;
        a.n_mid = 0;
    }
    auto kern = k_rows_persist<MODEL, TEAM, WB, AG>;
    const int per_sm = occupancy_one<k_rows_persist<MODEL, TEAM, WB, AG>>(smem, FusedBytes<MODEL, 1, TEAM>).ctas;
    const int cap = per_sm * sm_count;
    if (cap < 2) return FSGP_EUNSUPPORTED;
    if (grid_mid + grid_small > cap) {
        const int m = grid_mid ? std::max(1, (int)((int64_t)grid_mid * cap / (grid_mid + grid_small))) : 0;
        grid_mid = grid_small ? std::min(m, cap - 1) : cap;
        grid_small = cap - grid_mid;
    }
    q.warp_ctas = grid_mid;
    void *args[] = {&a, &q};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void *)kern, dim3(grid_mid + grid_small), dim3(kBlock), args,
                                                      smem + FusedBytes<MODEL, 1, TEAM>, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchCooperativeKernel (persistent step loop)");
    *grid_out = grid_mid + grid_small;
    return FSGP_OK;
}

template <int MODEL>
int launch_persist(const StepArgs &A, const PersistArgs &Q, int TEAM, int grid_mid, int grid_small, size_t smem, int sm_count,
                   cudaStream_t s, int *grid_out) {
    switch (TEAM) {
        case 1: return launch_persist_t<MODEL, 1>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        case 2: return launch_persist_t<MODEL, 2>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        case 4: return launch_persist_t<MODEL, 4>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        case 8: return launch_persist_t<MODEL, 8>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        case 16: return launch_persist_t<MODEL, 16>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        case 32: return launch_persist_t<MODEL, 32>(A, Q, grid_mid, grid_small, smem, sm_count, s, grid_out);
        default: return FSGP_EUNSUPPORTED;
    }
}

}  // namespace fsgp
