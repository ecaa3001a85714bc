// tile.cuh -- the row kernels' warp tile: gather first, draw afterwards.
//
// A warp takes a tile of row words, gathers and counts their in-arcs, and leaves what has
// to be drawn as items in shared memory; it then works the items off 32 at a time and
// finally forms the next states.  What bounds these kernels on GB300 is instruction
// issue: a word's draws are one or two Philox blocks of dependent integer operations
// (about 60 instructions each), and how many a word needs differs from word to word.
// Deciding each word in the thread that gathered it made every warp pay the deepest word's
// blocks at every word (17 to 23 of 32 threads active per instruction, measured on R-MAT,
// SIS, R = 256); the queues keep the threads full, because a thread works on an item that
// has something to draw, and items that need more blocks are packed again before the next
// one.  Deciding in place before, and now, with the counters and gathers of rows.cuh: SIR on
// R-MAT n = 16.8M, R = 256, T = 100: 283 to 201 ms; SIS on n = 8M: 257 to 167 ms; weighted
// SIR on n = 4.2M: 154 to 113 ms; batch of 32 mixed requests: 281 to 96 ms.
#pragma once

#include "step.cuh"

namespace fsgp {

// Lanes of p's 32 uniforms whose next bit is compared with bit t (a mask, 0 or ~0): the
// three-input majority is one step of the least-significant-first comparison "u < t".
__device__ __forceinline__ uint32_t maj_less(uint32_t p, uint32_t t, uint32_t lt) {
    return (~p & t) | (~p & lt) | (t & lt);
}

// Bit b (0 = least significant) of x as a mask.
__device__ __forceinline__ uint32_t bit_mask(uint32_t x, int b) { return (uint32_t)((int32_t)(x << (31 - b)) >> 31); }

// Eight threshold bits as masks, most significant first.
struct Masks8 {
    uint32_t m[8];
};
__device__ __forceinline__ Masks8 masks_of(uint32_t t8) {
    Masks8 r;
#pragma unroll
    for (int j = 0; j < 8; ++j) r.m[j] = bit_mask(t8, 7 - j);
    return r;
}
// ... from a table: two 16-byte loads, mostly of addresses the warp shares, in place of
// sixteen operations of the pipe that the compares and half of Philox already fill.
__device__ __forceinline__ Masks8 masks_at(const uint4 *t) {
    const uint4 a = __ldg(t), b = __ldg(t + 1);
    return Masks8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// u < t (lt) and u <= t (le) of the top eight bits, lanes in parallel; p[0] is the most
// significant plane.
__device__ __forceinline__ void less8(const Planes8 &P, const Masks8 &t, uint32_t &lt, uint32_t &le) {
    lt = 0u;
    le = 0xffffffffu;
#pragma unroll
    for (int j = 7; j >= 0; --j) {
        lt = maj_less(P.p[j], t.m[j], lt);
        le = maj_less(P.p[j], t.m[j], le);
    }
}

// Lanes of eq whose uniform is below th, the first 4 * m0 bits being known to be equal.
__device__ __forceinline__ uint32_t less_from(uint32_t eq, uint32_t th, uint32_t m0, uint32_t a, uint32_t t,
                                              uint32_t g, uint32_t tag, uint32_t k0, uint32_t k1) {
    uint32_t lt = 0u;
#pragma unroll 1
    for (uint32_t m = m0; m < 8u && eq; ++m) {
        const uint4 P = philox4x32_10(make_uint4(a, t, g, (tag << 8) | m), k0, k1);
        const uint32_t p[4] = {P.x, P.y, P.z, P.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t tb = bit_mask(th, 31 - ((int)m * 4 + i));
            lt |= eq & ~p[i] & tb;
            eq &= ~(p[i] ^ tb);
        }
    }
    return lt;
}

// The threshold of a lane with count k < 2^24, below which its uniform must lie, and eight
// bits as masks that decide every uniform whose own top eight bits differ from them: the
// survival table (a lane at or above it is infected), or the linear threshold's
// floor(k * 2^32 / d) + 1, which is below 2^32 for k < d.
template <bool TABLE>   // masks from the table (counts up to 255)
struct SurvThr {
    const uint64_t *surv;
    const uint4 *table;
    static constexpr bool falls = true;   // with k
    __device__ __forceinline__ uint32_t operator()(uint32_t k) const { return (uint32_t)__ldg(surv + k); }
    __device__ __forceinline__ Masks8 masks(uint32_t k) const {
        if constexpr (TABLE) return masks_at(table + 2 * k);
        else return masks_of((*this)(k) >> 24);
    }
};
// (u < floor(k * 2^32 / d) + 1 is u <= T, T = floor(k * 2^32 / d), whose top eight bits are
// floor(256 k / d): the 64-bit division is left to the ties.)
struct LtThr {
    uint32_t d;
    static constexpr bool falls = false;
    __device__ __forceinline__ uint32_t operator()(uint32_t k) const { return (uint32_t)(((uint64_t)k << 32) / d) + 1u; }
    __device__ __forceinline__ Masks8 masks(uint32_t k) const { return masks_of((k << 8) / d); }
};

// P: the top eight planes of the lanes' uniforms.
// Lanes of M (M != 0; counts at least 1, thresholds thr(k) monotone in k and in
// [1, 2^32)) whose uniform is below their threshold.  All lanes are
// first compared with the thresholds of the smallest and the largest count on the top
// eight bits; a lane outside that range is decided, and the few inside it (on average one
// in five words has one, R-MAT, SIS, beta = 0.01) are compared by groups of equal count.
// Lanes tied with their threshold in those bits (1 in 256) need further blocks: tie(lanes,
// threshold) takes them out of the result.
template <int B, class Thr, class TieFn>
__device__ __forceinline__ uint32_t counts_u_less(const Planes8 &P, const uint32_t (&c)[B], uint32_t M, Thr thr_of,
                                                  TieFn tie_fn) {
    const uint32_t ka = min_count<B>(c, M), kb = max_count<B>(c, M);
    uint32_t lt_lo = 0u, le_hi = 0xffffffffu;
    {
        const Masks8 lo = thr_of.masks(Thr::falls ? kb : ka), hi = thr_of.masks(Thr::falls ? ka : kb);
#pragma unroll
        for (int j = 7; j >= 0; --j) {
            lt_lo = maj_less(P.p[j], lo.m[j], lt_lo);
            le_hi = maj_less(P.p[j], hi.m[j], le_hi);
        }
    }
    uint32_t res = M & lt_lo;
    uint32_t U = M & ~lt_lo & le_hi;
#pragma unroll 1
    while (U) {
        const int sh = __clz(U & (0u - U));   // 31 - the lowest lane of U
        uint32_t k = 0u, Mk = U;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const uint32_t bit = (uint32_t)((int32_t)(c[b] << sh) >> 31);
            k |= bit & (1u << b);
            Mk &= ~(c[b] ^ bit);
        }
        U &= ~Mk;
        uint32_t lt, le;
        less8(P, thr_of.masks(k), lt, le);
        res |= Mk & lt;
        const uint32_t tie = Mk & le & ~lt;
        if (tie) tie_fn(tie, thr_of(k));
    }
    return res;
}

// The same on the first nb planes only (the others are zero): half or a quarter of the
// planes when the counts are small, as most are.
template <int B, class Thr, class TieFn>
__device__ __forceinline__ uint32_t counts_u_less_nb(int nb, const Planes8 &P, const uint32_t (&c)[B], uint32_t M,
                                                     Thr thr_of, TieFn tie_fn) {
    if constexpr (B > 4) {
        if (nb <= B / 2) {
            uint32_t h[B / 2];
#pragma unroll
            for (int b = 0; b < B / 2; ++b) h[b] = c[b];
            if constexpr (B == 16 && Thr::falls)
                return counts_u_less_nb<8>(nb, P, h, M, SurvThr<true>{thr_of.surv, thr_of.table}, tie_fn);
            else
                return counts_u_less_nb<B / 2>(nb, P, h, M, thr_of, tie_fn);
        }
    }
    return counts_u_less<B>(P, c, M, thr_of, tie_fn);
}

// Groups of tied lanes a tile queues: 1 lane in 256 is tied (measured mid-run on R-MAT,
// SIS: 23 per tile of the 256-word lane tiles, 2 per tile of the others).
constexpr int tie_cap(int B) { return B <= 1 ? 1 : (B == 2 ? 48 : 16); }

// Shared memory of one warp's tile of NS word slots: what the gather leaves for the draws.
// Count models: c[b] are the counter planes of the lanes that can change (c[0] receives
// the lanes that change through their in-arcs).  Arc models: c[0] collects the lanes some
// live arc reached.  f[0]: infectious lanes (then those that recover); f[1]: exposed lanes
// (then those that turn infectious).
template <int B, int NF, int NS, int NROW, int NARC>
struct Tile {
    uint32_t c[B][NS];
    uint32_t f[NF > 0 ? NF : 1][NF > 0 ? NS : 1];
    uint32_t eq_[NF > 0 && B == 1 ? NS : 1];
    int32_t row[NROW];                   // row (new id), or -1
    uint32_t node[NROW];                 // Philox subject
    int32_t w0[NROW];                    // first word of the row's slice
    uint32_t thr[NARC > 0 ? NROW : 1];   // IC: largest uniform that makes an arc live
    uint32_t arc_eq[NARC > 0 ? NARC : 1], arc_pos[NARC > 0 ? NARC : 1];
    // (slot numbers are 16-bit: stores through a byte pointer may alias anything, and the
    // reloads they forced cost the IC warp rows 36 against 23 ms per run, BA n = 1M)
    uint16_t arc_slot[NARC > 0 ? NARC : 1];
    uint16_t qc[B > 1 ? NS : 1];          // slots with lanes to decide by count
    static constexpr int kTies = tie_cap(B);
    uint32_t tie_eq[kTies], tie_thr[kTies];   // lanes tied after eight bits
    uint16_t tie_slot[kTies];
    int32_t ties;                        // entries wanted (those past kTies are drawn in place)
    uint16_t qf[NF > 0 ? NF : 1][NF > 0 ? NS : 1];

    // lanes of the fixed draws still tied, by queue position (the counter planes above 0 are
    // free by then)
    __device__ __forceinline__ uint32_t *eq() {
        if constexpr (B > 1) return c[1];
        else return eq_;
    }

    // result of fixed draw j (0 when the model has none)
    template <int J>
    __device__ __forceinline__ uint32_t fixed(int slot) const {
        if constexpr (J < NF) return f[J][slot];
        else return 0u;
    }
};

// Append `slot` of the threads with `want` to queue q (count n, uniform over the warp).
__device__ __forceinline__ void queue_push(uint16_t *q, int &n, bool want, int slot, int lane) {
    const unsigned m = __ballot_sync(0xffffffffu, want);
    if (want) q[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)slot;
    n += __popc(m);
}

// Fixed-threshold items (recovery, latent exit): f holds the lanes to draw and receives
// those whose uniform lies below the set's threshold.  Two Philox blocks (eight bits) per item and
// round: with 5 to 15 lanes per word every second item needs the second block, and one
// round of two interleaved blocks costs less than packing the items between single ones.
// The items with lanes still tied are packed for the next round (in place: a round writes
// only positions it has read).  ctx(slot, node, w): the slot's subject and word.
// LATENT: the exposed lanes' exit, else recovery.
template <bool LATENT, class CtxFn>
__device__ __forceinline__ void draw_fixed(const StepArgs &A, uint32_t *f, uint32_t *eqs, uint16_t *q, int n, int lane,
                                           CtxFn ctx) {
    constexpr uint32_t tag = LATENT ? TAG_LATENT : TAG_RECOVER;
#pragma unroll 1
    for (uint32_t m = 0; m < 8u && n > 0; m += 2) {
        int n2 = 0;
#pragma unroll 1
        for (int q0 = 0; q0 < n; q0 += 32) {
            uint32_t eq = 0u;
            int slot = 0;
            if (q0 + lane < n) {
                slot = q[q0 + lane];
                uint32_t node;
                int w;
                ctx(slot, node, w);
                const SetParams &sp = A.sp[w >> A.ws_shift];
                const uint64_t thr = __ldg(LATENT ? &sp.a_lat : &sp.g_rec);
                const uint32_t now = f[slot];
                uint32_t less = m ? now : 0u;
                eq = m ? eqs[q0 + lane] : now;
                if (thr >= TWO32) {
                    less = eq;
                    eq = 0u;
                } else if (thr == 0ull) {
                    eq = 0u;
                } else {
                    const Planes8 P = philox4x32_10_x2(node, A.t, A.gbase + (uint32_t)(w & (A.Ws - 1)), (tag << 8) | m,
                                                       __ldg(&sp.key0), __ldg(&sp.key1));
                    uint32_t lt, le;
                    less8(P, m ? masks_of(((uint32_t)thr << (4u * m)) >> 24) : masks_at(LATENT ? sp.lat_masks : sp.rec_masks),
                          lt, le);
                    less |= eq & lt;
                    eq &= le & ~lt;
                }
                f[slot] = less;
            }
            __syncwarp();
            const unsigned more = __ballot_sync(0xffffffffu, eq != 0u);
            if (eq) {
                const int at = n2 + __popc(more & ((1u << lane) - 1u));
                q[at] = (uint16_t)slot;
                eqs[at] = eq;
            }
            n2 += __popc(more);
            __syncwarp();
        }
        n = n2;
    }
}

// Arc items (IC, weighted graphs): lanes of slot arc_slot that an active source presses
// through the arc at caller position arc_pos.  Lanes whose uniform makes the arc live are
// added to c0[slot].  thr_of(row of the tile, pos, set): the arc is live iff its uniform
// lies below (0 = never, >= 2^32 = certain).
// PAIR: two interleaved Philox blocks (eight bits) per round instead of one, for small graphs,
// whose step is one row's chain of rounds (IC, ER n = 1289, R = 458: 319 and 305 us; n = 6929,
// R = 519: 895 and 860; weighted SIS, ER n = 2000, R = 64: 1049 and 964).
template <bool PAIR, class CtxFn, class ThrFn>
__device__ __forceinline__ void draw_arcs(const StepArgs &A, uint32_t *c0, uint32_t *arc_eq, uint32_t *arc_pos,
                                          uint16_t *arc_slot, int n, uint32_t tag, int lane, CtxFn ctx, ThrFn thr_of) {
#pragma unroll 1
    for (uint32_t m = 0; m < 8u && n > 0; m += PAIR ? 2 : 1) {
        int n2 = 0;
#pragma unroll 1
        for (int q0 = 0; q0 < n; q0 += 32) {
            uint32_t eq = 0u, pos = 0u;
            int slot = 0;
            if (q0 + lane < n) {
                slot = arc_slot[q0 + lane];
                pos = arc_pos[q0 + lane];
                eq = arc_eq[q0 + lane];
                uint32_t node;
                int w;
                const int row = ctx(slot, node, w);
                const SetParams &sp = A.sp[w >> A.ws_shift];
                const uint64_t thr = thr_of(row, pos, sp);
                uint32_t lt = 0u;
                if (thr >= TWO32) {
                    lt = eq;
                    eq = 0u;
                } else if (thr == 0ull) {
                    eq = 0u;
                } else {
                    const uint32_t th = (uint32_t)thr;
                    const uint32_t g = A.gbase + (uint32_t)(w & (A.Ws - 1));
                    auto compare = [&](const uint32_t *p, int n, uint32_t bits) {   // n bits, most significant first
#pragma unroll
                        for (int i = 0; i < n; ++i) {
                            const uint32_t tb = bit_mask(bits, n - 1 - i);
                            lt |= eq & ~p[i] & tb;
                            eq &= ~(p[i] ^ tb);
                        }
                    };
                    if constexpr (PAIR) {
                        const Planes8 P = philox4x32_10_x2(pos, A.t, g, (tag << 8) | m, __ldg(&sp.key0), __ldg(&sp.key1));
                        compare(P.p, 8, (th << (4u * m)) >> 24);
                    } else {
                        const uint4 P = philox4x32_10(make_uint4(pos, A.t, g, (tag << 8) | m), __ldg(&sp.key0), __ldg(&sp.key1));
                        const uint32_t p[4] = {P.x, P.y, P.z, P.w};
                        compare(p, 4, (th << (4u * m)) >> 28);
                    }
                }
                if (lt) atomicOr(&c0[slot], lt);   // several arcs may reach one slot
            }
            __syncwarp();
            const unsigned more = __ballot_sync(0xffffffffu, eq != 0u);
            if (eq) {
                const int at = n2 + __popc(more & ((1u << lane) - 1u));
                arc_slot[at] = (uint16_t)slot;
                arc_pos[at] = pos;
                arc_eq[at] = eq;
            }
            n2 += __popc(more);
            __syncwarp();
        }
        n = n2;
    }
}

}  // namespace fsgp
