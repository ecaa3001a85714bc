// surrogate.cu -- learned seed-set surrogate: a 3-layer message-passing network that
// predicts each node's infection probability from the seed set and the model
// parameters, trained on the simulator's own per-node final frequencies, used to
// screen many candidate seed sets before Monte Carlo re-scores the best of them.
// The paper has no learned component; this is the project's screening surrogate.
//
//   x_v  = [seed_v, beta, gamma, log(1+d_in), log(1+d_out), log(1+k_v), 0, 0]
//          (k_v = in-arcs of v whose source is a seed, with multiplicity)
//   m_v  = mean over in-arcs u -> v of h_u          (message passing, Sec. 3.1 Eq. agg)
//   h'_v = ReLU(h_v Ws_l + m_v Wn_l + b_l), l = 1..3, width 64
//   p_v  = sigmoid(h3_v . w_o + b_o),  loss = mean_v (p_v - y_v)^2
//
// The forward dense layers run on the fifth-generation tensor cores (tcgen05.mma into
// tensor memory, bfloat16 operands, float32 accumulation; the last layer applies the
// output head in its epilogue); the backward products use mma.sync m16n8k16 on the same
// operand types.  Activations are stored as bfloat16, gradients and the Adam state in
// float32.  Every kernel is this project's own.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "fsgp_internal.cuh"

namespace fsgp {
namespace sg {

constexpr int H = 64;          // hidden width
constexpr int F0 = 8;          // input features (5 used, zero padded)
// flat parameter layout (float32): Ws1 Wn1 b1 Ws2 Wn2 b2 Ws3 Wn3 b3 wo bo
constexpr int kW1 = F0 * H, kW = H * H;
constexpr int OFF_WS1 = 0, OFF_WN1 = OFF_WS1 + kW1, OFF_B1 = OFF_WN1 + kW1;
constexpr int OFF_WS2 = OFF_B1 + H, OFF_WN2 = OFF_WS2 + kW, OFF_B2 = OFF_WN2 + kW;
constexpr int OFF_WS3 = OFF_B2 + H, OFF_WN3 = OFF_WS3 + kW, OFF_B3 = OFF_WN3 + kW;
constexpr int OFF_WO = OFF_B3 + H, OFF_BO = OFF_WO + H;
constexpr int N_PARAMS = OFF_BO + 1;

__host__ __device__ constexpr int off_ws(int l) { return l == 1 ? OFF_WS1 : (l == 2 ? OFF_WS2 : OFF_WS3); }
__host__ __device__ constexpr int off_wn(int l) { return l == 1 ? OFF_WN1 : (l == 2 ? OFF_WN2 : OFF_WN3); }
__host__ __device__ constexpr int off_b(int l) { return l == 1 ? OFF_B1 : (l == 2 ? OFF_B2 : OFF_B3); }

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

// ------------------------------------------------------------------ forward kernels

// Input features; seed bits come from the (device) seed list of candidate *cur.
__global__ void k_features(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ out_ptr,
                           int32_t n, float beta, float gamma, bf16 *x) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const float din = (float)(row_ptr[v + 1] - row_ptr[v]);
        const float dout = (float)(out_ptr[v + 1] - out_ptr[v]);
        bf16 *r = x + (size_t)v * F0;
        r[0] = __float2bfloat16(0.f);
        r[1] = __float2bfloat16(beta);
        r[2] = __float2bfloat16(gamma);
        r[3] = __float2bfloat16(log1pf(din));
        r[4] = __float2bfloat16(log1pf(dout));
        r[5] = r[6] = r[7] = __float2bfloat16(0.f);
    }
}

// Seed in-arc counts: for every out-arc s -> v of the seeds of candidate *cur add `delta`
// to cnt[v] (one CTA per seed, so hub seeds spread over the CTA's threads).
__global__ void k_seed_count(const int32_t *__restrict__ cand, int32_t k, const int32_t *cur,
                             const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_dst,
                             int32_t delta, int32_t *cnt) {
    const int c = *cur;
    for (int i = blockIdx.x; i < k; i += gridDim.x) {
        const int32_t sd = cand[(size_t)c * k + i];
        for (int64_t a = (int64_t)out_ptr[sd] + threadIdx.x; a < out_ptr[sd + 1]; a += blockDim.x)
            atomicAdd(&cnt[out_dst[a]], delta);
    }
}

// Feature 5 = log(1 + cnt[v]) for the out-neighbours of the seeds of candidate *cur.
__global__ void k_seed_feat(const int32_t *__restrict__ cand, int32_t k, const int32_t *cur,
                            const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_dst,
                            const int32_t *__restrict__ cnt, bf16 *x) {
    const int c = *cur;
    for (int i = blockIdx.x; i < k; i += gridDim.x) {
        const int32_t sd = cand[(size_t)c * k + i];
        for (int64_t a = (int64_t)out_ptr[sd] + threadIdx.x; a < out_ptr[sd + 1]; a += blockDim.x) {
            const int32_t v = out_dst[a];
            x[(size_t)v * F0 + 5] = __float2bfloat16(log1pf((float)cnt[v]));
        }
    }
}

// Set (value 1) or clear (value 0) the seed bit of the seeds of candidate *cur; the
// clearing pass also advances *cur.
__global__ void k_seed_bits(const int32_t *__restrict__ cand, int32_t k, int32_t *cur, float value,
                            int advance, bf16 *x) {
    const int c = *cur;
    for (int i = threadIdx.x; i < k; i += blockDim.x) x[(size_t)cand[(size_t)c * k + i] * F0] = __float2bfloat16(value);
    __syncthreads();
    if (advance && threadIdx.x == 0) *cur = c + 1;
}

// Screening: take back candidate *cur's seed features and set candidate *cur + 1's (at most
// kClusterSeeds seeds), then advance *cur; past the last candidate only the taking back is
// done.  One cluster of CTAs with cluster barriers between its phases (clear, count, write
// the counts' logarithms) in place of seven launches of a microsecond or two each.  The
// seeds' out-arcs are taken as one list, the cluster's threads side by side: with a CTA per
// seed the largest hub held up the candidate, and eight CTAs are fewer than the seeds
// (screening 16 candidates of the 64 largest hubs: R-MAT n = 600k 10.9 ms with a CTA per seed,
// 9.1 so; n = 4M 116 and 104; 8 mixed candidates, R-MAT n = 2M, 16 arcs per node: 21.0 and 20.2).
constexpr int kSeedCtas = 8, kSeedThreads = 256, kClusterSeeds = 64;
__device__ __forceinline__ void cluster_barrier() {
    __threadfence();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __cluster_dims__(kSeedCtas, 1, 1) __launch_bounds__(kSeedThreads)
    k_seed_next(const int32_t *__restrict__ cand, int32_t k, int32_t n_cand, int32_t *cur,
                const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_dst, int32_t *cnt, bf16 *x) {
    // [0] candidate c - 1, [1] candidate c: each seed's first out-arc, and the out-arcs before it
    __shared__ int32_t s_beg[2][kClusterSeeds];
    __shared__ int64_t s_off[2][kClusterSeeds + 1];
    const int c = *(volatile int32_t *)cur + 1;
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (q < 2) {   // two seeds per lane
        const int cc = c - 1 + q;
        int32_t b[2] = {0, 0}, d[2] = {0, 0};
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = 2 * lane + j;
            if (cc >= 0 && cc < n_cand && i < k) {
                const int32_t sd = __ldg(cand + (size_t)cc * k + i);
                b[j] = __ldg(out_ptr + sd);
                d[j] = __ldg(out_ptr + sd + 1) - b[j];
                if (blockIdx.x == 0 && q == 0) x[(size_t)sd * F0] = __float2bfloat16(0.f);
            }
        }
        int64_t sum = (int64_t)d[0] + d[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t up = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += up;
        }
        s_beg[q][2 * lane] = b[0];
        s_beg[q][2 * lane + 1] = b[1];
        s_off[q][2 * lane + 1] = sum - d[1];
        s_off[q][2 * lane + 2] = sum;
        if (lane == 0) s_off[q][0] = 0;
    }
    __syncthreads();
    // f(target) for the out-arcs of candidate c - 1 + w, four of a thread's targets in flight
    auto each_out = [&](int w, auto f) {
        const int64_t total = s_off[w][kClusterSeeds], step = (int64_t)kSeedCtas * kSeedThreads;
        int i = 0;   // seed of the arc at hand
        for (int64_t t = (int64_t)blockIdx.x * kSeedThreads + threadIdx.x; t < total; t += 4 * step) {
            int32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t a = t + u * step;
                v[u] = -1;
                if (a < total) {
                    while (s_off[w][i + 1] <= a) ++i;
                    v[u] = __ldg(out_dst + (s_beg[w][i] + (a - s_off[w][i])));
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (v[u] >= 0) f(v[u]);
        }
    };
    each_out(0, [&](int32_t v) {
        cnt[v] = 0;
        x[(size_t)v * F0 + 5] = __float2bfloat16(0.f);
    });
    cluster_barrier();
    if (c < n_cand && blockIdx.x == 0)
        for (int i = threadIdx.x; i < k; i += blockDim.x)
            x[(size_t)cand[(size_t)c * k + i] * F0] = __float2bfloat16(1.f);
    each_out(1, [&](int32_t v) { atomicAdd(&cnt[v], 1); });
    cluster_barrier();
    each_out(1, [&](int32_t v) { x[(size_t)v * F0 + 5] = __float2bfloat16(log1pf((float)__ldcg(cnt + v))); });
    if (blockIdx.x == 0 && threadIdx.x == 0) *cur = c;
}

// Sixteen bytes of a gathered row, zeros without a row.  In assembly so that a round's eight
// loads are issued one behind the other: left to itself the compiler kept registers, not
// loads (32 registers and two or so loads in flight).
__device__ __forceinline__ uint4 ld_row16(const void *p, bool has) {
    uint4 r;
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n mov.b32 %0, 0;\n mov.b32 %1, 0;\n mov.b32 %2, 0;\n"
                 " mov.b32 %3, 0;\n @p ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n}"
                 : "=&r"(r.x), "=&r"(r.y), "=&r"(r.z), "=&r"(r.w) : "l"(p), "r"((uint32_t)has));
    return r;
}

__device__ __forceinline__ void add_bf16x8(float (&sum)[8], const uint4 &x) {
    const bf162 *xp = reinterpret_cast<const bf162 *>(&x);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        sum[2 * i] += __bfloat162float(xp[i].x);
        sum[2 * i + 1] += __bfloat162float(xp[i].y);
    }
}

// Sums of h_u over the chunks of long in-rows (items {row, begin, end, slot}), added to
// acc[slot] in float32.  Eight lanes take one chunk of kSgChunk arcs, eight at a time: F = 64
// 16 bytes of every source row each, F = 8 one source row each (their sums meet by
// shuffle).  (Chunks of 256 arcs, two at a time, took 76 us beside a layer's 182, BA
// n = 300k: few of them, each one long chain.)
template <int F>
__global__ void __launch_bounds__(256) k_agg_long(const int32_t *__restrict__ col, const bf16 *__restrict__ h,
                                                  const int4 *__restrict__ items, int32_t n_items, float *acc) {
    const int lane = threadIdx.x & 31, j = lane & 7, g0 = lane & 24;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) >> 3;
    for (int64_t v = t >> 3; __any_sync(0xffffffffu, v < n_items); v += groups) {
        int4 it = make_int4(0, 0, 0, -1);
        if (v < n_items) it = __ldg(items + v);
        float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        uint32_t b = it.y;
        int32_t mine = arc_in(b, j, it.z) ? __ldg(col + b + j) : -1;
        while (__any_sync(0xffffffffu, b < (uint32_t)it.z)) {
            if constexpr (F == H) {
                uint4 x[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int32_t u = __shfl_sync(0xffffffffu, mine, g0 + q);
                    x[q] = ld_row16(h + (size_t)max(u, 0) * F + 8 * j, u >= 0);
                }
                b += 8;
                mine = arc_in(b, j, it.z) ? __ldg(col + b + j) : -1;
#pragma unroll
                for (int q = 0; q < 8; ++q) add_bf16x8(sum, x[q]);
            } else {
                const int32_t u = mine;
                b += 8;
                mine = arc_in(b, j, it.z) ? __ldg(col + b + j) : -1;
                if (u >= 0) add_bf16x8(sum, __ldg(reinterpret_cast<const uint4 *>(h + (size_t)u * F)));
            }
        }
        if constexpr (F != H) {
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int i = 0; i < 8; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
        }
        if (it.w < 0 || (F != H && j != 0)) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i) atomicAdd(acc + (size_t)it.w * F + (F == H ? 8 * j : 0) + i, sum[i]);
    }
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ------------------------------------- one layer: aggregation and tcgen05 / TMEM product
//
// m_v = mean over in-arcs u -> v of h_u (float32 sums), y = ReLU([h | m] W + b), for tiles of
// 128 rows, K = 2F (16 or 128), N = 64.  What bounds a layer is the gather of the source
// rows out of L2 (d_in x 128 bytes per node); the product is a few percent of the tensor
// pipe.  So the CTA that gathers a tile's means also multiplies it: the means go to shared
// memory as the right half of the A operand, are never written to memory (unless the
// backward pass wants them) and never read back, and three CTAs per SM cover one another's
// products with their gathers.  Rows are taken in degree-bucket order, so that the rows a
// warp gathers together are of similar length; the long rows (the first n_long of that
// order) come summed from k_agg_long.
//   Gather: F/8 lanes per row, 16 bytes each, eight arcs in flight per lane (F = 8: four
//   lanes per row, one arc each).
//   Product: both operands in the canonical K-major layout without swizzle (8-row x 16-byte
//   core matrices; the two K-neighbour core matrices of one instruction lie 128 B apart,
//   8-row groups K*16 B apart); one elected thread issues K/16 tcgen05.mma (kind::f16:
//   bfloat16 in, float32 accumulate) into a 128-lane x 64-column tensor-memory accumulator
//   and commits them to an mbarrier; the eight warps read 32 lanes x 32 columns each back
//   (tcgen05.ld) for bias, ReLU and the bfloat16 rows, which leave through shared memory so
//   that every store covers whole 128-byte rows.  W^T is staged once per CTA.
// Measured on BA n = 500k, m = 4: 105 us a layer (F = 64) plus 25 for the long rows, against
// 119 for the aggregation and 77 for the product as separate kernels; a screened candidate
// 0.475 to 0.325 ms.

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, leading (K) and stride (8-row group)
// byte offsets, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Byte offset of the 16-byte chunk kc of row r in a K-major core-matrix tile of KC chunks.
__device__ __forceinline__ uint32_t core_off(int r, int kc, int KC) {
    return (uint32_t)(((r >> 3) * KC + kc) * 128 + (r & 7) * 16);
}

constexpr int kTcRows = 128;            // rows per tile (MMA M)
constexpr int kTcThreads = 256;
constexpr int kTcCtas = 3;              // per SM
constexpr int kTcWaitLimit = 1 << 24;   // mbarrier polls before giving up

// The A tile, reused for the tile's output rows (128 x 64 bfloat16), and W^T.
template <int F>
__host__ __device__ constexpr int tc_a_bytes() { return kTcRows * 2 * F * 2 > kTcRows * H * 2 ? kTcRows * 2 * F * 2 : kTcRows * H * 2; }
template <int F>
constexpr size_t tc_smem_bytes() { return (size_t)tc_a_bytes<F>() + (size_t)H * (2 * F) * 2; }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    // a source size of 0 fills the 16 bytes with zeros (rows past the end)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0));
}

__device__ __forceinline__ uint4 scaled_bf16x8(const float (&sum)[8], float inv) {
    uint4 o;
    bf162 *op = reinterpret_cast<bf162 *>(&o);
#pragma unroll
    for (int i = 0; i < 4; ++i) op[i] = __floats2bfloat162_rn(sum[2 * i] * inv, sum[2 * i + 1] * inv);
    return o;
}

// HEAD: the epilogue also applies the output head, p = sigmoid(h . w_o + b_o) of the
// bfloat16 layer output, and writes p (when p_out is set) and / or adds the sum of p
// into psum[*cur] (screening).  m_out and y may be null (not wanted).
template <int F, bool HEAD>
__global__ void __launch_bounds__(kTcThreads, kTcCtas)
    k_layer_tc(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col, const int32_t *__restrict__ order,
               int32_t n, const bf16 *__restrict__ h, const bf16 *__restrict__ Ws, const bf16 *__restrict__ Wn,
               const float *__restrict__ bias, int32_t n_long, float *acc, bf16 *m_out, bf16 *y,
               const bf16 *__restrict__ wo, const float *__restrict__ bo, float *p_out, float *psum,
               const int32_t *cur, int32_t *err) {
    constexpr int K = 2 * F;
    constexpr int KC = K / 8;            // 16-byte chunks per row
    constexpr int FC = F / 8;            // of them own features
    extern __shared__ __align__(1024) uint8_t tc_smem[];
    uint8_t *sA = tc_smem;                          // 128 x K, then 128 x 64 output rows
    uint8_t *sB = tc_smem + tc_a_bytes<F>();        // 64 x K (W transposed)
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int32_t s_node[2][kTcRows];
    __shared__ float s_bias[H], s_wo[HEAD ? H : 1], s_dot[HEAD ? 2 : 1][HEAD ? kTcRows : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t tiles = ((int64_t)n + kTcRows - 1) / kTcRows;
    if ((int64_t)blockIdx.x >= tiles) return;
    // B: output column c holds its K inputs, Ws rows then Wn rows (16-byte row reads,
    // element-wise transposed stores)
#pragma unroll
    for (int i = tid; i < K * H / 8; i += kTcThreads) {
        const int k = i / (H / 8), c8 = i % (H / 8) * 8;
        const uint4 x = *reinterpret_cast<const uint4 *>((k < F ? Ws + k * H : Wn + (k - F) * H) + c8);
        const bf16 *w = reinterpret_cast<const bf16 *>(&x);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            *reinterpret_cast<bf16 *>(sB + core_off(c8 + q, k >> 3, KC) + (k & 7) * 2) = w[q];
    }
    if (tid < H) {
        s_bias[tid] = bias[tid];
        if constexpr (HEAD) s_wo[tid] = __bfloat162float(wo[tid]);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(smem_addr(&tmem_base)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // kind::f16: D f32 (bit 4), A and B bf16 (bits 7, 10), K-major, N = 64, M = 128
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(H >> 3) << 17) |
                               ((uint32_t)(kTcRows >> 4) << 24);
    const float bo_f = HEAD ? bo[0] : 0.f;
    float psum_local = 0.f;
    uint32_t phase = 0;
    bool ok = true;
    int nb = 0;
    // This thread's rows: LPR lanes per row, ITS rows one after another.  The next tile's
    // nodes, arc ranges and first column indices are loaded while this tile is gathered,
    // multiplied and stored.
    constexpr int LPR = F == H ? 8 : 4, RPW = 32 / LPR, ITS = 16 / RPW;
    const int j = lane % LPR, g0 = lane - j, r0 = warp * 16 + lane / LPR;
    int32_t node[ITS], beg[ITS], end[ITS], c0[ITS], c1[F == H ? 1 : ITS];
    auto nodes_of = [&](int64_t tile) {
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
            const int64_t i = tile * kTcRows + r0 + it * RPW;
            node[it] = i < n ? __ldg(order + i) : -1;
        }
    };
    auto ranges_of = [&](int64_t tile) {
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
            beg[it] = end[it] = 0;
            if (node[it] >= 0) {
                beg[it] = __ldg(row_ptr + node[it]);
                end[it] = __ldg(row_ptr + node[it] + 1);
            }
        }
    };
    auto cols_of = [&](int64_t tile) {
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
            const bool mine = tile * kTcRows + r0 + it * RPW >= n_long;
            c0[it] = mine && arc_in(beg[it], j, end[it]) ? __ldg(col + beg[it] + j) : -1;
            if constexpr (F != H) c1[it] = mine && arc_in(beg[it], j + 4, end[it]) ? __ldg(col + beg[it] + j + 4) : -1;
        }
    };
    nodes_of(blockIdx.x);
    ranges_of(blockIdx.x);
    cols_of(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, nb ^= 1) {
        const int64_t i0 = tile * kTcRows;   // position in `order` of the tile's first row
        const int64_t next = tile + gridDim.x;
        if (j == 0)
#pragma unroll
            for (int it = 0; it < ITS; ++it) s_node[nb][r0 + it * RPW] = node[it];
        __syncthreads();                     // the previous tile's rows have left sA
#pragma unroll
        for (int it = 0; it < ITS; ++it)     // own features, chunk j
            if (j < FC)
                cp_async16(smem_addr(sA) + core_off(r0 + it * RPW, j, KC),
                           h + (size_t)max(node[it], 0) * F + j * 8, node[it] >= 0);
        asm volatile("cp.async.commit_group;");
#pragma unroll
        for (int it = 0; it < ITS; ++it) {
            const int r = r0 + it * RPW;
            const int32_t v = node[it];
            const uint32_t e = end[it];
            uint32_t b = beg[it];
            const float inv = e > b ? 1.f / (float)(e - b) : 0.f;
            float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (i0 + r < n_long && v >= 0) {   // summed already; the accumulator goes back to zero
                if (F == H || j == 0) {
                    float4 *a = reinterpret_cast<float4 *>(acc + (size_t)(i0 + r) * F + (F == H ? 8 * j : 0));
                    const float4 s0 = a[0], s1 = a[1];
                    a[0] = a[1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    sum[0] = s0.x, sum[1] = s0.y, sum[2] = s0.z, sum[3] = s0.w;
                    sum[4] = s1.x, sum[5] = s1.y, sum[6] = s1.z, sum[7] = s1.w;
                }
                b = e;
            }
            int32_t mine = c0[it];
            if constexpr (F == H) {
                // the row's eight lanes hold eight arcs' sources and take 16 bytes of each
                while (__any_sync(0xffffffffu, b < e)) {
                    uint4 x[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int32_t u = __shfl_sync(0xffffffffu, mine, g0 + q);
                        x[q] = ld_row16(h + (size_t)max(u, 0) * F + 8 * j, u >= 0);
                    }
                    b += 8;
                    mine = arc_in(b, j, e) ? __ldg(col + b + j) : -1;
#pragma unroll
                    for (int q = 0; q < 8; ++q) add_bf16x8(sum, x[q]);
                }
                const uint4 o = scaled_bf16x8(sum, inv);
                *reinterpret_cast<uint4 *>(sA + core_off(r, FC + j, KC)) = o;
                if (m_out && v >= 0) reinterpret_cast<uint4 *>(m_out + (size_t)v * F)[j] = o;
            } else {
                // a source row is 16 bytes: the four lanes take every fourth arc each, two at
                // a time
                int32_t mine2 = c1[it];
                for (uint32_t a = b + j; a < e; a += 8) {
                    const uint4 x = ld_row16(h + (size_t)mine * F, true);
                    const uint4 x2 = ld_row16(h + (size_t)max(mine2, 0) * F, mine2 >= 0);
                    mine = a + 8 < e ? __ldg(col + a + 8) : -1;
                    mine2 = a + 12 < e ? __ldg(col + a + 12) : -1;
                    add_bf16x8(sum, x);
                    add_bf16x8(sum, x2);
                }
                __syncwarp();
#pragma unroll
                for (int o = 1; o < 4; o <<= 1)
#pragma unroll
                    for (int i = 0; i < 8; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
                if (j == 0) {
                    const uint4 o = scaled_bf16x8(sum, inv);
                    *reinterpret_cast<uint4 *>(sA + core_off(r, FC, KC)) = o;
                    if (m_out && v >= 0) *reinterpret_cast<uint4 *>(m_out + (size_t)v * F) = o;
                }
            }
        }
        nodes_of(next);   // (past the last tile: no rows)
        asm volatile("cp.async.wait_group 0;");
        asm volatile("fence.proxy.async.shared::cta;");   // smem writes -> tensor-core reads
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t tbase = tmem_base;
        if (tid == 0) {
            const uint32_t a0 = smem_addr(sA), b0 = smem_addr(sB);
#pragma unroll
            for (int k = 0; k < K / 16; ++k) {
                const uint64_t ad = umma_desc(a0 + k * 256, 128, KC * 128);
                const uint64_t bd = umma_desc(b0 + k * 256, 128, KC * 128);
                const uint32_t accum = k > 0 ? 1u : 0u;
                asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                             " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                             ::"r"(tbase), "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         ::"r"(smem_addr(&mbar)));
        }
        ranges_of(next);
        uint32_t done = 0;
        for (int it = 0; it < kTcWaitLimit && !done; ++it)
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                         " selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(smem_addr(&mbar)), "r"(phase));
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!done) {
            ok = false;
            atomicExch(err, 1);
            // give the issued MMAs a second bounded wait before the TMEM is freed
            for (int it = 0; it < kTcWaitLimit && !done; ++it)
                asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                             " selp.u32 %0, 1, 0, p;\n}"
                             : "=r"(done) : "r"(smem_addr(&mbar)), "r"(phase ^ 1u));
        } else {
            cols_of(next);
            // this thread: row 32 * (warp % 4) + lane, columns 32 * (warp / 4) .. + 31
            const int r = 32 * (warp & 3) + lane, half = warp >> 2;
            float dot = 0.f;
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                const int c0 = half * 32 + cc * 16;   // first of 16 columns
                uint32_t d[16];
                const uint32_t taddr = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                             : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]),
                               "=r"(d[7]), "=r"(d[8]), "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]),
                               "=r"(d[13]), "=r"(d[14]), "=r"(d[15])
                             : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                bf162 o[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    o[j] = __floats2bfloat162_rn(fmaxf(__uint_as_float(d[2 * j]) + s_bias[c0 + 2 * j], 0.f),
                                                 fmaxf(__uint_as_float(d[2 * j + 1]) + s_bias[c0 + 2 * j + 1], 0.f));
                if constexpr (HEAD) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        dot += __bfloat162float(o[j].x) * s_wo[c0 + 2 * j] + __bfloat162float(o[j].y) * s_wo[c0 + 2 * j + 1];
                }
                if (y) {   // 16-byte chunk c of row r lies at chunk c ^ (r & 7): no bank conflicts
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        *reinterpret_cast<uint4 *>(sA + r * 128 + (((c0 >> 3) + q) ^ (r & 7)) * 16) =
                            *reinterpret_cast<const uint4 *>(&o[4 * q]);
                }
            }
            if constexpr (HEAD) s_dot[half][r] = dot;
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        ok = __syncthreads_and(ok) != 0;   // also orders this tile's TMEM reads before the next tile
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!ok) break;
        if (y) {
#pragma unroll
            for (int c = tid; c < kTcRows * 8; c += kTcThreads) {
                const int r = c >> 3, q = c & 7;
                const int32_t v = s_node[nb][r];
                if (v >= 0)
                    reinterpret_cast<uint4 *>(y + (size_t)v * H)[q] =
                        *reinterpret_cast<const uint4 *>(sA + r * 128 + (q ^ (r & 7)) * 16);
            }
        }
        if constexpr (HEAD) {
            if (tid < kTcRows) {
                const int32_t v = s_node[nb][tid];
                if (v >= 0) {
                    const float pv = 1.f / (1.f + expf(-(s_dot[0][tid] + s_dot[1][tid] + bo_f)));
                    if (p_out) p_out[v] = pv;
                    psum_local += pv;
                }
            }
        }
    }
    if constexpr (HEAD) {
        if (psum) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) psum_local += __shfl_xor_sync(0xffffffffu, psum_local, o);
            if (lane == 0 && psum_local != 0.f) atomicAdd(psum + *cur, psum_local);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem_base));
}

// ----------------------------------------------------------------- backward kernels

// dlogit = 2 (p - y) / n * p (1 - p); dh3 = dlogit * wo; grad wo += sum h3 dlogit,
// grad bo += sum dlogit; loss += sum (p - y)^2 / n (double).
__global__ void k_head_bwd(const bf16 *__restrict__ h3, const bf16 *__restrict__ wo, const float *__restrict__ p,
                           const float *__restrict__ y, int32_t n, float *dh, float *grad, double *loss) {
    __shared__ float s_gwo[8][H];
    __shared__ float s_gbo[8];
    __shared__ double s_loss[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const bf162 w = reinterpret_cast<const bf162 *>(wo)[lane];
    float g0 = 0.f, g1 = 0.f, gb = 0.f;
    double ls = 0.0;
    for (int64_t v = warp; v < n; v += nw) {
        const float pv = p[v], diff = pv - y[v];
        const float dl = 2.f * diff / (float)n * pv * (1.f - pv);
        const bf162 x = reinterpret_cast<const bf162 *>(h3 + (size_t)v * H)[lane];
        g0 += __bfloat162float(x.x) * dl;
        g1 += __bfloat162float(x.y) * dl;
        reinterpret_cast<float2 *>(dh + (size_t)v * H)[lane] =
            make_float2(dl * __bfloat162float(w.x), dl * __bfloat162float(w.y));
        if (lane == 0) {
            gb += dl;
            ls += (double)diff * diff;
        }
    }
    s_gwo[wid][2 * lane] = g0;
    s_gwo[wid][2 * lane + 1] = g1;
    if (lane == 0) {
        s_gbo[wid] = gb;
        s_loss[wid] = ls;
    }
    __syncthreads();
    if (threadIdx.x < H) {
        float s = 0.f;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += s_gwo[i][threadIdx.x];
        atomicAdd(grad + OFF_WO + threadIdx.x, s);
    }
    if (threadIdx.x == 0) {
        float s = 0.f;
        double l = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            s += s_gbo[i];
            l += s_loss[i];
        }
        atomicAdd(grad + OFF_BO, s);
        atomicAdd(loss, l / (double)n);
    }
}

// One layer backward on the tensor cores.  dz = dy * (y > 0) is rounded to bfloat16 and
// both products take bfloat16 operands with float32 accumulation:
//   input gradients   [dah | dam] = dz W^T      (rows x 2F, float32 out; skipped for layer 1);
//                     dam is written as dam / d_in, the term its adjoint aggregation sums
//   weight gradients  [gWs ; gWn] += [h | m]^T dz   (2F x 64, accumulated in registers)
//   bias gradient     gb += sum_rows dz          (float32, from the unrounded dz)
// A CTA of 8 warps walks 32-row tiles staged in shared memory: dz (row-major), the input
// tile A = [h | m] (row-major) and W = [Ws ; Wn] (2F x 64, row-major, staged once).  The
// fragments come from ldmatrix, transposed where the reduction runs over the tile's rows
// (packing them from half-words took 20 instructions per product); a warp's eight
// weight-gradient tiles share their column block, and with it the dz fragments.  The next
// tile's rows are loaded into registers while this one is multiplied.  (BA n = 300k, F = 64:
// 287 to 108 us.)
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t &a, uint32_t &b, const bf16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(a), "=r"(b) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}

template <int F>
__global__ void __launch_bounds__(256, 3) k_dense_bwd(const bf16 *__restrict__ h, const bf16 *__restrict__ m,
                                                      const bf16 *__restrict__ y, const float *__restrict__ dy,
                                                      const bf16 *__restrict__ Ws, const bf16 *__restrict__ Wn,
                                                      const float *__restrict__ inv_din, int32_t n, float *dah,
                                                      float *dam, float *grad, int l, int input_grad) {
    constexpr int K = 2 * F;
    constexpr int RT = 32;            // rows per tile
    constexpr int WP = H + 8;         // padded row of W and dz (bank spread)
    constexpr int AP = K + 8;         // padded row of the input tile
    constexpr int MT = K / 16;        // weight-gradient row blocks (each warp: its 8 columns of all)
    constexpr int AC = RT * (K / 8);  // 16-byte chunks of the input tile
    constexpr int APT = (AC + 255) / 256;
    __shared__ __align__(16) bf16 Wsm[K * WP];
    __shared__ __align__(16) bf16 Zs[RT * WP];
    __shared__ __align__(16) bf16 As[RT * AP];
    __shared__ float s_b[8][H];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, tg = lane & 3;
    for (int i = tid; i < K * H; i += blockDim.x) {
        const int k = i / H, c = i % H;
        Wsm[k * WP + c] = k < F ? Ws[k * H + c] : Wn[(k - F) * H + c];
    }
    float wacc[MT][4];
#pragma unroll
    for (int q = 0; q < MT; ++q) wacc[q][0] = wacc[q][1] = wacc[q][2] = wacc[q][3] = 0.f;
    float gb0 = 0.f, gb1 = 0.f;       // bias columns 2 lane, 2 lane + 1
    // the tile's rows in registers: dy and y (rows warp, warp + 8, ..: column pair `lane`)
    // and 16-byte chunks of [h | m]
    float2 rdy[RT / 8];
    bf162 ry[RT / 8];
    uint4 ra[APT];
    auto load = [&](int64_t r0) {
#pragma unroll
        for (int q = 0; q < RT / 8; ++q) {
            const int64_t r = r0 + warp + 8 * q;
            rdy[q] = make_float2(0.f, 0.f);
            ry[q] = __floats2bfloat162_rn(0.f, 0.f);
            if (r < n) {
                rdy[q] = __ldg(reinterpret_cast<const float2 *>(dy + (size_t)r * H) + lane);
                ry[q] = reinterpret_cast<const bf162 *>(y + (size_t)r * H)[lane];
            }
        }
#pragma unroll
        for (int q = 0; q < APT; ++q) {
            const int i = tid + 256 * q, rr = i / (K / 8), c = i % (K / 8);
            const int64_t r = r0 + rr;
            ra[q] = make_uint4(0u, 0u, 0u, 0u);
            if (i < AC && r < n)
                ra[q] = __ldg(c < F / 8 ? reinterpret_cast<const uint4 *>(h + (size_t)r * F) + c
                                        : reinterpret_cast<const uint4 *>(m + (size_t)r * F) + (c - F / 8));
        }
    };
    const int64_t step = (int64_t)gridDim.x * RT;
    int64_t r0 = (int64_t)blockIdx.x * RT;
    load(r0);
    for (; r0 < n; r0 += step) {
        __syncthreads();              // previous tile's readers are done (and W is staged)
#pragma unroll
        for (int q = 0; q < RT / 8; ++q) {
            const float2 d = make_float2(__bfloat162float(ry[q].x) > 0.f ? rdy[q].x : 0.f,
                                         __bfloat162float(ry[q].y) > 0.f ? rdy[q].y : 0.f);
            gb0 += d.x;
            gb1 += d.y;
            *reinterpret_cast<bf162 *>(Zs + (warp + 8 * q) * WP + 2 * lane) = __floats2bfloat162_rn(d.x, d.y);
        }
#pragma unroll
        for (int q = 0; q < APT; ++q) {
            const int i = tid + 256 * q, rr = i / (K / 8), c = i % (K / 8);
            if (i < AC) *reinterpret_cast<uint4 *>(As + rr * AP + 8 * c) = ra[q];
        }
        __syncthreads();
        load(r0 + step);              // (rows past the end read as zeros)
        // input gradients: 2 row blocks x K/8 column blocks over the warps
        if (input_grad) {
            const int mt = warp & 1;
            uint32_t a[H / 16][4];
#pragma unroll
            for (int ks = 0; ks < H / 16; ++ks)
                ldsm_x4(a[ks], Zs + (mt * 16 + (lane & 15)) * WP + ks * 16 + (lane >> 4) * 8);
#pragma unroll 2
            for (int nt = warp >> 1; nt < K / 8; nt += 4) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
                uint32_t w[2][4];     // K-steps 0, 1 and 2, 3 of the 8 columns
                ldsm_x4(w[0], Wsm + (nt * 8 + (lane & 7)) * WP + (lane >> 3) * 8);
                ldsm_x4(w[1], Wsm + (nt * 8 + (lane & 7)) * WP + 32 + (lane >> 3) * 8);
#pragma unroll
                for (int ks = 0; ks < H / 16; ++ks) mma_bf16(acc, a[ks], w[ks >> 1][(ks & 1) * 2], w[ks >> 1][(ks & 1) * 2 + 1]);
                const int k = nt * 8 + 2 * tg;
                const int64_t ra_ = r0 + mt * 16 + g, rb_ = ra_ + 8;
                if (k < F) {
                    if (ra_ < n) *reinterpret_cast<float2 *>(dah + (size_t)ra_ * F + k) = make_float2(acc[0], acc[1]);
                    if (rb_ < n) *reinterpret_cast<float2 *>(dah + (size_t)rb_ * F + k) = make_float2(acc[2], acc[3]);
                } else {
                    if (ra_ < n) {
                        const float iv = __ldg(inv_din + ra_);
                        *reinterpret_cast<float2 *>(dam + (size_t)ra_ * F + k - F) = make_float2(acc[0] * iv, acc[1] * iv);
                    }
                    if (rb_ < n) {
                        const float iv = __ldg(inv_din + rb_);
                        *reinterpret_cast<float2 *>(dam + (size_t)rb_ * F + k - F) = make_float2(acc[2] * iv, acc[3] * iv);
                    }
                }
            }
        }
        // weight gradients: A^T (K x RT) times dz (RT x 64), reduction over the tile's rows;
        // this warp's columns 8 warp .. + 7
#pragma unroll
        for (int ks = 0; ks < RT / 16; ++ks) {
            uint32_t b0, b1;
            ldsm_x2_t(b0, b1, Zs + (ks * 16 + (lane & 15)) * WP + warp * 8);
#pragma unroll
            for (int q = 0; q < MT; ++q) {
                uint32_t a[4];
                ldsm_x4_t(a, As + (ks * 16 + (lane & 7) + ((lane >> 4) & 1) * 8) * AP + q * 16 + ((lane >> 3) & 1) * 8);
                mma_bf16(wacc[q], a, b0, b1);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < MT; ++q) {
        const int c = warp * 8 + 2 * tg;
        const int ka = q * 16 + g, kb = ka + 8;
        float *ga = grad + (ka < F ? off_ws(l) + ka * H : off_wn(l) + (ka - F) * H) + c;
        float *gbp = grad + (kb < F ? off_ws(l) + kb * H : off_wn(l) + (kb - F) * H) + c;
        atomicAdd(ga, wacc[q][0]);
        atomicAdd(ga + 1, wacc[q][1]);
        atomicAdd(gbp, wacc[q][2]);
        atomicAdd(gbp + 1, wacc[q][3]);
    }
    s_b[warp][2 * lane] = gb0;
    s_b[warp][2 * lane + 1] = gb1;
    __syncthreads();
    if (tid < H) {
        float sb = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) sb += s_b[w][tid];
        atomicAdd(grad + off_b(l) + tid, sb);
    }
}

// dh_u = dah_u + sum over out-arcs u -> v of dam_v   (adjoint of the mean; k_dense_bwd wrote
// dam already divided by d_in).  Sixteen lanes per item take 16 bytes of every row, eight
// arcs in flight; items are the rows in degree-bucket order (out-degrees follow the
// in-degrees on most graphs), behind the chunks of the long out-rows, whose partial sums go
// to acc[slot] for k_agg_bwd_fin.  (A thread per feature, one arc at a time: 183 us, BA
// n = 300k; 106 so.)
__global__ void __launch_bounds__(256) k_agg_bwd(const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_dst,
                                                 const int32_t *__restrict__ order, int32_t n,
                                                 const float *__restrict__ dah, const float *__restrict__ dam, float *dh,
                                                 int32_t long_min, const int4 *__restrict__ items, int32_t n_items,
                                                 float *acc) {
    constexpr int F = H;
    const int lane = threadIdx.x & 31, j = lane & 15, g0 = lane & 16;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) >> 4;
    const int64_t total = (int64_t)n + n_items;
    for (int64_t v = t >> 4; __any_sync(0xffffffffu, v < total); v += groups) {
        int32_t u = -1, slot = -1;
        uint32_t b = 0, e = 0;
        if (v < n_items) {   // the long rows' chunks first
            const int4 it = __ldg(items + v);
            u = it.x, b = it.y, e = it.z, slot = it.w;
        } else if (v < total) {
            u = __ldg(order + (v - n_items));
            b = __ldg(out_ptr + u);
            e = __ldg(out_ptr + u + 1);
            if (e - b >= (uint32_t)long_min) u = -1, e = b;
        }
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        int32_t mine = j < 8 && arc_in(b, j, e) ? __ldg(out_dst + b + j) : -1;
        while (__any_sync(0xffffffffu, b < e)) {
            uint4 x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int32_t w = __shfl_sync(0xffffffffu, mine, g0 + q);
                x[q] = ld_row16(dam + (size_t)max(w, 0) * F + 4 * j, w >= 0);
            }
            b += 8;
            mine = j < 8 && arc_in(b, j, e) ? __ldg(out_dst + b + j) : -1;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                s.x += __uint_as_float(x[q].x);
                s.y += __uint_as_float(x[q].y);
                s.z += __uint_as_float(x[q].z);
                s.w += __uint_as_float(x[q].w);
            }
        }
        if (u < 0) continue;
        if (slot < 0) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(dah + (size_t)u * F) + j);
            reinterpret_cast<float4 *>(dh + (size_t)u * F)[j] = make_float4(a.x + s.x, a.y + s.y, a.z + s.z, a.w + s.w);
        } else {
            float *p = acc + (size_t)slot * F + 4 * j;
            atomicAdd(p, s.x);
            atomicAdd(p + 1, s.y);
            atomicAdd(p + 2, s.z);
            atomicAdd(p + 3, s.w);
        }
    }
}

template <int F>
__global__ void k_agg_bwd_fin(const int32_t *__restrict__ long_rows, int32_t n_long, const float *__restrict__ dah,
                              float *acc, float *dh) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)n_long * F;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slot = i / F;
        const int j = (int)(i % F);
        const size_t o = (size_t)long_rows[slot] * F + j;
        dh[o] = dah[o] + acc[i];
        acc[i] = 0.f;
    }
}

// Per-graph tables, built on the device: what each row has of long-row chunks.  Position i
// of the degree order (in-rows, its first n_in_long) and node v (out-rows); the entries past
// the last are zero, so that the scans end in the totals.
__device__ __forceinline__ int32_t chunks_of(int32_t d, int32_t long_min) {
    return d >= long_min ? (int32_t)arc_chunks(d, kSgChunk) : 0;
}
__global__ void k_table_counts(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ out_ptr,
                               const int32_t *__restrict__ order, int32_t n, int32_t n_in_long, int32_t long_min,
                               int32_t *in_chunks, int32_t *out_long, int32_t *out_chunks) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = v < n ? out_ptr[v + 1] - out_ptr[v] : 0;
        out_long[v] = d >= long_min;
        out_chunks[v] = chunks_of(d, long_min);
        if (v <= n_in_long) {
            const int32_t u = v < n_in_long ? order[v] : 0;
            in_chunks[v] = v < n_in_long ? chunks_of(row_ptr[u + 1] - row_ptr[u], long_min) : 0;
        }
    }
}
__global__ void k_table_totals(const int32_t *in_total, const int32_t *long_total, const int32_t *out_total, int32_t *totals) {
    totals[0] = *in_total;
    totals[1] = *long_total;
    totals[2] = *out_total;
}

// 1 / d_in, and the long out-rows by slot.
__global__ void k_table_rows(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ out_ptr, int32_t n,
                             int32_t long_min, const int32_t *__restrict__ out_slot, float *inv, int32_t *out_rows) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = row_ptr[v + 1] - row_ptr[v];
        inv[v] = d > 0 ? 1.f / (float)d : 0.f;
        if (out_ptr[v + 1] - out_ptr[v] >= long_min) out_rows[out_slot[v]] = (int32_t)v;
    }
}

// Chunk t of the m rows whose first chunks are first[0 .. m] (row j: ids[j], or j; its slot:
// slots[j], or j): one thread per chunk, so that a hub's thousands spread out.
__global__ void k_table_items(const int32_t *__restrict__ ptr, const int32_t *__restrict__ ids,
                              const int32_t *__restrict__ slots, const int32_t *__restrict__ first, int32_t m,
                              int32_t total, int4 *items) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int32_t lo = 0, hi = m - 1;   // the last row whose first chunk is t or before
        while (lo < hi) {
            const int32_t mid = lo + (hi - lo + 1) / 2;
            if (first[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int32_t row = ids ? ids[lo] : lo;
        const int64_t b = ptr[row] + (t - first[lo]) * kSgChunk;
        items[t] = make_int4(row, (int32_t)b, (int32_t)min(b + kSgChunk, (int64_t)ptr[row + 1]), slots ? slots[lo] : lo);
    }
}

// Adam (Kingma and Ba, 2015) with bias correction, then the bfloat16 copies.
__global__ void k_adam(float *theta, float *m, float *v, const float *g, int np, float lr, float b1,
                       float b2, float eps, float c1, float c2, bf16 *wb) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += blockDim.x * gridDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float th = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        theta[i] = th;
        wb[i] = __float2bfloat16(th);
    }
}

__global__ void k_to_bf16(const float *theta, int np, bf16 *wb) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += blockDim.x * gridDim.x)
        wb[i] = __float2bfloat16(theta[i]);
}

}  // namespace sg
}  // namespace fsgp

using namespace fsgp;
using namespace fsgp::sg;

struct fsgp_surrogate {
    int device = 0;
    int sm_count = 0;
    float *theta = nullptr, *adam_m = nullptr, *adam_v = nullptr, *grad = nullptr;
    bf16 *wb = nullptr;        // bfloat16 copy of theta (same layout)
    int64_t step = 0;
    // activations / gradients for graphs up to cap nodes
    int64_t cap = 0;
    bf16 *x = nullptr, *m1 = nullptr, *h1 = nullptr, *m2 = nullptr, *h2 = nullptr, *m3 = nullptr, *h3 = nullptr;
    float *p = nullptr, *y = nullptr, *dh = nullptr, *dah = nullptr, *dam = nullptr, *dh2 = nullptr;
    double *loss = nullptr;
    int32_t *cur = nullptr;
    int32_t *cnt = nullptr;     // seed in-arc counts per node (kept at zero between calls)
    int32_t *tc_err = nullptr;  // set by a dense-layer CTA whose tensor-core wait ran out
};

namespace {

void sg_free_acts(fsgp_surrogate *s) {
    void *ptrs[] = {s->x, s->m1, s->h1, s->m2, s->h2, s->m3, s->h3, s->p, s->y, s->dh, s->dah, s->dam, s->dh2, s->cnt};
    for (void *p : ptrs) cudaFree(p);
    s->cnt = nullptr;
    s->x = s->m1 = s->h1 = s->m2 = s->h2 = s->m3 = s->h3 = nullptr;
    s->p = s->y = s->dh = s->dah = s->dam = s->dh2 = nullptr;
    s->cap = 0;
}

int sg_ensure(fsgp_surrogate *s, int64_t n) {
    if (n <= s->cap) return FSGP_OK;
    sg_free_acts(s);
    const size_t nb = (size_t)n;
    cudaError_t e;
    if ((e = cudaMalloc(&s->x, nb * F0 * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->m1, nb * F0 * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->h1, nb * H * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->m2, nb * H * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->h2, nb * H * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->m3, nb * H * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->h3, nb * H * sizeof(bf16))) != cudaSuccess ||
        (e = cudaMalloc(&s->p, nb * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->y, nb * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->dh, nb * H * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->dah, nb * H * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->dam, nb * H * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->dh2, nb * H * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&s->cnt, nb * sizeof(int32_t))) != cudaSuccess ||
        (e = cudaMemset(s->cnt, 0, nb * sizeof(int32_t))) != cudaSuccess) {
        sg_free_acts(s);
        return cuda_fail(e, "cudaMalloc (surrogate activations)");
    }
    s->cap = n;
    return FSGP_OK;
}

// Persistent CTAs of a layer: kTcCtas per SM at most.
int tc_grid(const fsgp_surrogate *s, int64_t n) {
    const int64_t tiles = (n + kTcRows - 1) / kTcRows;
    return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)s->sm_count * kTcCtas));
}

// The layer kernel's shared-memory limit, and a carve-out that leaves the rest of the SM's
// memory as L1 for the gathers (its three CTAs' share of 228 KB).
template <int F, bool HEAD>
cudaError_t tc_attributes() {
    cudaError_t e = cudaFuncSetAttribute(k_layer_tc<F, HEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tc_smem_bytes<F>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_layer_tc<F, HEAD>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)std::min<size_t>(100, (kTcCtas * (tc_smem_bytes<F>() + 4096) * 100) / (228 * 1024) + 1));
    return e;
}

// A tensor-core wait of an earlier launch ran out (the flag is sticky): FSGP_ETIMEOUT.
int sg_check_tc(fsgp_surrogate *s, cudaStream_t st) {
    int32_t h = 0;
    FSGP_CUDA(cudaMemcpyAsync(&h, s->tc_err, sizeof h, cudaMemcpyDeviceToHost, st));
    FSGP_CUDA(cudaStreamSynchronize(st));
    if (h) return fail(FSGP_ETIMEOUT, "a tensor-core completion wait of the surrogate's dense layer ran out");
    return FSGP_OK;
}

int grid_of(const fsgp_surrogate *s, int64_t work, int threads, int per_sm = 8) {
    int64_t g = (work + threads - 1) / threads;
    g = std::min<int64_t>(g, (int64_t)s->sm_count * per_sm);
    return (int)std::max<int64_t>(g, 1);
}

// Build the graph's aggregation tables on first use (synchronises st; call outside
// captures).  Scratch: activation and gradient buffers of s, which hold nothing yet and
// have room for n + 1 counts each.
// (Copying the long rows to the host, sorting and expanding them there took as much as the
// call: the first gradient on BA n = 300k 1.82 ms, 1.10 so, later ones 0.88; on R-MAT n = 4M
// 33.7, 14.0 and 13.7; screening 8 candidates on R-MAT n = 4M 62.0, 41.6 and 41.1.)
int sg_cache(fsgp_surrogate *s, const fsgp_graph *gc, cudaStream_t st) {
    fsgp_graph *g = const_cast<fsgp_graph *>(gc);   // lazily built cache of the handle
    if (g->sgc.mem) return FSGP_OK;
    SgCache C;
    const int32_t n = g->n;
    int bucket = 0;   // long_min is 2^bucket
    while (C.long_min < kSgLongMax && ((int64_t)C.long_min * n < 4 * g->nnz || (C.long_min << 14) < n)) C.long_min *= 2;
    while ((1 << bucket) < C.long_min) ++bucket;
    C.n_in_long = g->cls.bucket_start[bucket];
    int32_t *in_chunks = (int32_t *)s->h1, *in_first = (int32_t *)s->h2;
    int32_t *is_long = (int32_t *)s->dh, *out_slot = (int32_t *)s->dah;
    int32_t *out_chunks = (int32_t *)s->dam, *out_first = (int32_t *)s->dh2;
    int64_t *tiles = (int64_t *)s->m2;
    int32_t *d_totals = (int32_t *)s->m3;
    int32_t totals[3] = {0, 0, 0};
    if (g->max_deg >= C.long_min || g->max_out_deg >= C.long_min) {
        k_table_counts<<<grid_of(s, (int64_t)n + 1, 256), 256, 0, st>>>(g->row_ptr, g->out_ptr, g->rows_sorted, n, C.n_in_long,
                                                                        C.long_min, in_chunks, is_long, out_chunks);
        int rc = exclusive_scan_i32(in_chunks, (int64_t)C.n_in_long + 1, in_first, tiles, st);
        if (rc == FSGP_OK) rc = exclusive_scan_i32(is_long, (int64_t)n + 1, out_slot, tiles, st);
        if (rc == FSGP_OK) rc = exclusive_scan_i32(out_chunks, (int64_t)n + 1, out_first, tiles, st);
        if (rc) return rc;
        k_table_totals<<<1, 1, 0, st>>>(in_first + C.n_in_long, out_slot + n, out_first + n, d_totals);
        FSGP_CUDA(cudaMemcpyAsync(totals, d_totals, sizeof totals, cudaMemcpyDeviceToHost, st));
        FSGP_CUDA(cudaStreamSynchronize(st));
    }
    C.n_in_items = totals[0];
    C.n_out_long = totals[1];
    C.n_out_items = totals[2];
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_in = al(sizeof(int4) * (size_t)C.n_in_items), b_out = al(sizeof(int4) * (size_t)C.n_out_items);
    const size_t b_inv = al(sizeof(float) * (size_t)n), b_long = al(sizeof(int32_t) * (size_t)C.n_out_long);
    const size_t b_acc = al(sizeof(float) * H * (size_t)std::max(C.n_in_long, C.n_out_long));
    FSGP_CUDA(cudaMalloc(&C.mem, b_in + b_out + b_inv + b_long + b_acc));
    uint8_t *p = (uint8_t *)C.mem;
    C.in_items = (int4 *)p;
    C.out_items = (int4 *)(p += b_in);
    C.inv_din = (float *)(p += b_out);
    C.out_long = (int32_t *)(p += b_inv);
    C.acc = (float *)(p += b_long);
    k_table_rows<<<grid_of(s, n, 256), 256, 0, st>>>(g->row_ptr, g->out_ptr, n, C.long_min, out_slot, C.inv_din, C.out_long);
    if (C.n_in_items)
        k_table_items<<<grid_of(s, C.n_in_items, 256), 256, 0, st>>>(g->row_ptr, g->rows_sorted, nullptr, in_first,
                                                                     C.n_in_long, C.n_in_items, C.in_items);
    if (C.n_out_items)
        k_table_items<<<grid_of(s, C.n_out_items, 256), 256, 0, st>>>(g->out_ptr, nullptr, out_slot, out_first, n,
                                                                      C.n_out_items, C.out_items);
    cudaError_t e = b_acc ? cudaMemsetAsync(C.acc, 0, b_acc, st) : cudaSuccess;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaFree(C.mem);
        return cuda_fail(e, "surrogate tables");
    }
    g->sgc = C;
    return FSGP_OK;
}

// One layer (the head with it when p or psum is set): y from h, the means kept in m if set.
template <int F, bool HEAD>
void sg_layer(fsgp_surrogate *s, const fsgp_graph *g, int l, const bf16 *h, bf16 *m, bf16 *y, float *p, float *psum,
              cudaStream_t st) {
    const SgCache &C = g->sgc;
    if (C.n_in_items)
        k_agg_long<F><<<grid_of(s, (int64_t)C.n_in_items * 8, 256), 256, 0, st>>>(
            g->col, h, C.in_items, C.n_in_items, C.acc);
    k_layer_tc<F, HEAD><<<tc_grid(s, g->n), kTcThreads, tc_smem_bytes<F>(), st>>>(
        g->row_ptr, g->col, g->rows_sorted, g->n, h, s->wb + off_ws(l), s->wb + off_wn(l), s->theta + off_b(l),
        C.n_in_long, C.acc, m, y, s->wb + OFF_WO, s->theta + OFF_BO, p, psum, s->cur, s->tc_err);
}

// Forward of the three layers and the head from features s->x (already seeded).  keep: the
// backward pass follows (it reads the means and the last layer's output).
void sg_forward(fsgp_surrogate *s, const fsgp_graph *g, float *p, float *psum, bool keep, cudaStream_t st) {
    sg_layer<F0, false>(s, g, 1, s->x, keep ? s->m1 : nullptr, s->h1, nullptr, nullptr, st);
    sg_layer<H, false>(s, g, 2, s->h1, keep ? s->m2 : nullptr, s->h2, nullptr, nullptr, st);
    sg_layer<H, true>(s, g, 3, s->h2, keep ? s->m3 : nullptr, keep ? s->h3 : nullptr, p, psum, st);
}

int sg_prepare_inputs(fsgp_surrogate *s, const fsgp_graph *g, const int32_t *seeds_host, int64_t ns,
                      double beta, double gamma, cudaStream_t st) {
    for (int64_t i = 0; i < ns; ++i)
        if (seeds_host[i] < 0 || seeds_host[i] >= g->n) return fail(FSGP_EINVAL, "seed node out of range");
    int rc = sg_ensure(s, g->n);
    if (rc) return rc;
    rc = sg_cache(s, g, st);
    if (rc) return rc;
    k_features<<<grid_of(s, g->n, 256), 256, 0, st>>>(g->row_ptr, g->out_ptr, g->n, (float)beta, (float)gamma, s->x);
    if (ns > 0) {
        // seed bits: small host list staged through the activation buffer y (floats)
        int32_t *d_seeds = reinterpret_cast<int32_t *>(s->y);
        if (ns > s->cap) return fail(FSGP_EINVAL, "more seeds than nodes");
        FSGP_CUDA(cudaMemcpyAsync(d_seeds, seeds_host, sizeof(int32_t) * (size_t)ns, cudaMemcpyHostToDevice, st));
        FSGP_CUDA(cudaMemsetAsync(s->cur, 0, sizeof(int32_t), st));
        k_seed_bits<<<1, 256, 0, st>>>(d_seeds, (int32_t)ns, s->cur, 1.f, 0, s->x);
        const int gk = (int)std::min<int64_t>(ns, 1024);
        k_seed_count<<<gk, 256, 0, st>>>(d_seeds, (int32_t)ns, s->cur, g->out_ptr, g->out_dst, 1, s->cnt);
        k_seed_feat<<<gk, 256, 0, st>>>(d_seeds, (int32_t)ns, s->cur, g->out_ptr, g->out_dst, s->cnt, s->x);
        k_seed_count<<<gk, 256, 0, st>>>(d_seeds, (int32_t)ns, s->cur, g->out_ptr, g->out_dst, -1, s->cnt);
    }
    FSGP_CUDA(cudaGetLastError());
    return FSGP_OK;
}

int sg_backward(fsgp_surrogate *s, const fsgp_graph *g, cudaStream_t st) {
    const int32_t n = g->n;
    const bf16 *W = s->wb;
    FSGP_CUDA(cudaMemsetAsync(s->grad, 0, sizeof(float) * N_PARAMS, st));
    FSGP_CUDA(cudaMemsetAsync(s->loss, 0, sizeof(double), st));
    k_head_bwd<<<grid_of(s, (int64_t)n * 32, 256), 256, 0, st>>>(s->h3, W + OFF_WO, s->p, s->y, n, s->dh, s->grad, s->loss);
    const SgCache &C = g->sgc;
    const int gb = grid_of(s, ((int64_t)n + 31) / 32, 1, 3);
    // layer 3: dy = dh (float), outputs dh2 = d h2
    k_dense_bwd<H><<<gb, 256, 0, st>>>(s->h2, s->m3, s->h3, s->dh, W + OFF_WS3, W + OFF_WN3, C.inv_din, n, s->dah, s->dam, s->grad, 3, 1);
    const int64_t items = (int64_t)n + C.n_out_items;
    k_agg_bwd<<<grid_of(s, items * 16, 256), 256, 0, st>>>(g->out_ptr, g->out_dst, g->rows_sorted, n, s->dah, s->dam, s->dh2,
                                                            C.long_min, C.out_items, C.n_out_items, C.acc);
    if (C.n_out_long)
        k_agg_bwd_fin<H><<<grid_of(s, (int64_t)C.n_out_long * H, 256), 256, 0, st>>>(C.out_long, C.n_out_long,
                                                                                  s->dah, C.acc, s->dh2);
    // layer 2
    k_dense_bwd<H><<<gb, 256, 0, st>>>(s->h1, s->m2, s->h2, s->dh2, W + OFF_WS2, W + OFF_WN2, C.inv_din, n, s->dah, s->dam, s->grad, 2, 1);
    k_agg_bwd<<<grid_of(s, items * 16, 256), 256, 0, st>>>(g->out_ptr, g->out_dst, g->rows_sorted, n, s->dah, s->dam, s->dh,
                                                            C.long_min, C.out_items, C.n_out_items, C.acc);
    if (C.n_out_long)
        k_agg_bwd_fin<H><<<grid_of(s, (int64_t)C.n_out_long * H, 256), 256, 0, st>>>(C.out_long, C.n_out_long,
                                                                                  s->dah, C.acc, s->dh);
    // layer 1 (input gradients not needed beyond the weights)
    k_dense_bwd<F0><<<gb, 256, 0, st>>>(s->x, s->m1, s->h1, s->dh, W + OFF_WS1, W + OFF_WN1, C.inv_din, n, s->dah, s->dam, s->grad, 1, 0);
    FSGP_CUDA(cudaGetLastError());
    return FSGP_OK;
}

// init: He normal weights from a SplitMix64 stream (Box-Muller), zero biases
uint64_t sm64(uint64_t &x) {
    uint64_t z = (x += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" int fsgp_surrogate_num_params(void) { return N_PARAMS; }

extern "C" int fsgp_surrogate_create(uint64_t init_seed, fsgp_surrogate **out) {
    set_error("");
    if (!out) return fail(FSGP_EINVAL, "out is NULL");
    *out = nullptr;
    fsgp_surrogate *s = new (std::nothrow) fsgp_surrogate();
    if (!s) return fail(FSGP_ENOMEM, "host allocation failed");
    cudaError_t e;
    if ((e = cudaGetDevice(&s->device)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, s->device)) != cudaSuccess ||
        (e = cudaMalloc(&s->theta, sizeof(float) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMalloc(&s->adam_m, sizeof(float) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMalloc(&s->adam_v, sizeof(float) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMalloc(&s->grad, sizeof(float) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMalloc(&s->wb, sizeof(bf16) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMalloc(&s->loss, sizeof(double))) != cudaSuccess ||
        (e = cudaMalloc(&s->cur, sizeof(int32_t))) != cudaSuccess ||
        (e = cudaMalloc(&s->tc_err, sizeof(int32_t))) != cudaSuccess ||
        (e = cudaMemset(s->tc_err, 0, sizeof(int32_t))) != cudaSuccess ||
        (e = tc_attributes<F0, false>()) != cudaSuccess || (e = tc_attributes<H, false>()) != cudaSuccess ||
        (e = tc_attributes<H, true>()) != cudaSuccess) {
        fsgp_surrogate_destroy(s);
        return cuda_fail(e, "cudaMalloc (surrogate)");
    }
    std::vector<float> th(N_PARAMS, 0.f);
    uint64_t st = init_seed;
    auto normal = [&]() {
        const double u1 = ((sm64(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        const double u2 = ((sm64(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        return sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
    };
    auto fill = [&](int off, int count, double sd) {
        for (int i = 0; i < count; ++i) th[off + i] = (float)(sd * normal());
    };
    fill(OFF_WS1, kW1, sqrt(2.0 / (2 * F0)));
    fill(OFF_WN1, kW1, sqrt(2.0 / (2 * F0)));
    for (int l = 2; l <= 3; ++l) {
        fill(off_ws(l), kW, sqrt(2.0 / (2 * H)));
        fill(off_wn(l), kW, sqrt(2.0 / (2 * H)));
    }
    fill(OFF_WO, H, sqrt(1.0 / H));
    if ((e = cudaMemcpy(s->theta, th.data(), sizeof(float) * N_PARAMS, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemset(s->adam_m, 0, sizeof(float) * N_PARAMS)) != cudaSuccess ||
        (e = cudaMemset(s->adam_v, 0, sizeof(float) * N_PARAMS)) != cudaSuccess) {
        fsgp_surrogate_destroy(s);
        return cuda_fail(e, "surrogate init");
    }
    k_to_bf16<<<32, 256>>>(s->theta, N_PARAMS, s->wb);
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) {
        fsgp_surrogate_destroy(s);
        return cuda_fail(e, "surrogate init");
    }
    *out = s;
    return FSGP_OK;
}

extern "C" int fsgp_surrogate_destroy(fsgp_surrogate *s) {
    set_error("");
    if (!s) return FSGP_OK;
    cudaDeviceSynchronize();
    sg_free_acts(s);
    cudaFree(s->theta);
    cudaFree(s->adam_m);
    cudaFree(s->adam_v);
    cudaFree(s->grad);
    cudaFree(s->wb);
    cudaFree(s->loss);
    cudaFree(s->cur);
    cudaFree(s->tc_err);
    delete s;
    return FSGP_OK;
}

extern "C" int fsgp_surrogate_params(fsgp_surrogate *s, float *get_host, const float *set_host) {
    set_error("");
    if (!s) return fail(FSGP_EINVAL, "surrogate is NULL");
    if (set_host) {
        FSGP_CUDA(cudaMemcpy(s->theta, set_host, sizeof(float) * N_PARAMS, cudaMemcpyHostToDevice));
        FSGP_CUDA(cudaMemset(s->adam_m, 0, sizeof(float) * N_PARAMS));
        FSGP_CUDA(cudaMemset(s->adam_v, 0, sizeof(float) * N_PARAMS));
        s->step = 0;
        k_to_bf16<<<32, 256>>>(s->theta, N_PARAMS, s->wb);
        FSGP_CUDA(cudaDeviceSynchronize());
    }
    if (get_host) FSGP_CUDA(cudaMemcpy(get_host, s->theta, sizeof(float) * N_PARAMS, cudaMemcpyDeviceToHost));
    return FSGP_OK;
}

extern "C" int fsgp_surrogate_forward(fsgp_surrogate *s, const fsgp_graph *g, const int32_t *seeds_host,
                                      int64_t n_seeds, double beta, double gamma, float *p_out, void *stream) {
    set_error("");
    if (!s || !g || !p_out || (n_seeds > 0 && !seeds_host)) return fail(FSGP_EINVAL, "NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    int rc = sg_prepare_inputs(s, g, seeds_host, n_seeds, beta, gamma, st);
    if (rc) return rc;
    sg_forward(s, g, p_out, nullptr, false, st);
    FSGP_CUDA(cudaGetLastError());
    return FSGP_OK;
}

extern "C" int fsgp_surrogate_grad(fsgp_surrogate *s, const fsgp_graph *g, const int32_t *seeds_host,
                                   int64_t n_seeds, double beta, double gamma, const float *y,
                                   double *loss_out, float *grad_out, void *stream) {
    set_error("");
    if (!s || !g || !y || (n_seeds > 0 && !seeds_host)) return fail(FSGP_EINVAL, "NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    int rc = sg_prepare_inputs(s, g, seeds_host, n_seeds, beta, gamma, st);
    if (rc) return rc;
    FSGP_CUDA(cudaMemcpyAsync(s->y, y, sizeof(float) * (size_t)g->n, cudaMemcpyDeviceToDevice, st));
    sg_forward(s, g, s->p, nullptr, true, st);
    rc = sg_backward(s, g, st);
    if (rc) return rc;
    if (loss_out) FSGP_CUDA(cudaMemcpyAsync(loss_out, s->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    if (grad_out) FSGP_CUDA(cudaMemcpyAsync(grad_out, s->grad, sizeof(float) * N_PARAMS, cudaMemcpyDeviceToHost, st));
    return sg_check_tc(s, st);
}

extern "C" int fsgp_surrogate_train_step(fsgp_surrogate *s, const fsgp_graph *g, const int32_t *seeds_host,
                                         int64_t n_seeds, double beta, double gamma, const float *y,
                                         float lr, double *loss_out, void *stream) {
    set_error("");
    if (!s || !g || !y || (n_seeds > 0 && !seeds_host)) return fail(FSGP_EINVAL, "NULL argument");
    if (!(lr > 0.f)) return fail(FSGP_EINVAL, "learning rate must be positive");
    cudaStream_t st = (cudaStream_t)stream;
    int rc = sg_prepare_inputs(s, g, seeds_host, n_seeds, beta, gamma, st);
    if (rc) return rc;
    FSGP_CUDA(cudaMemcpyAsync(s->y, y, sizeof(float) * (size_t)g->n, cudaMemcpyDeviceToDevice, st));
    sg_forward(s, g, s->p, nullptr, true, st);
    rc = sg_backward(s, g, st);
    if (rc) return rc;
    s->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)s->step), c2 = 1.f - powf(b2, (float)s->step);
    k_adam<<<grid_of(s, N_PARAMS, 256), 256, 0, st>>>(s->theta, s->adam_m, s->adam_v, s->grad, N_PARAMS, lr,
                                                      b1, b2, 1e-8f, c1, c2, s->wb);
    FSGP_CUDA(cudaGetLastError());
    if (loss_out) {
        FSGP_CUDA(cudaMemcpyAsync(loss_out, s->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        FSGP_CUDA(cudaStreamSynchronize(st));
    }
    return FSGP_OK;
}

extern "C" int fsgp_surrogate_screen(fsgp_surrogate *s, const fsgp_graph *g, const int32_t *cand_host,
                                     int32_t k, int32_t n_cand, double beta, double gamma, float *scores_out,
                                     void *stream) {
    set_error("");
    if (!s || !g || !cand_host || !scores_out || k < 1 || n_cand < 1) return fail(FSGP_EINVAL, "bad argument");
    for (int64_t i = 0; i < (int64_t)k * n_cand; ++i)
        if (cand_host[i] < 0 || cand_host[i] >= g->n) return fail(FSGP_EINVAL, "candidate node out of range");
    cudaStream_t caller = (cudaStream_t)stream;
    int rc = sg_ensure(s, g->n);
    if (rc) return rc;
    rc = sg_cache(s, g, caller);
    if (rc) return rc;
    // captures are not allowed on the legacy default stream: work on a private stream
    // ordered after the caller's work
    cudaStream_t st = nullptr;
    cudaEvent_t ev = nullptr;
    int32_t *d_cand = nullptr;
    float *d_scores = nullptr;
    cudaError_t e;
    rc = FSGP_OK;
    do {
        if ((e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) != cudaSuccess ||
            (e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess ||
            (e = cudaEventRecord(ev, caller)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(st, ev, 0)) != cudaSuccess ||
            (e = cudaMalloc(&d_cand, sizeof(int32_t) * (size_t)k * n_cand)) != cudaSuccess ||
            (e = cudaMalloc(&d_scores, sizeof(float) * (size_t)n_cand)) != cudaSuccess) {
            rc = cuda_fail(e, "screen setup");
            break;
        }
        if ((e = cudaMemcpyAsync(d_cand, cand_host, sizeof(int32_t) * (size_t)k * n_cand, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
            (e = cudaMemsetAsync(d_scores, 0, sizeof(float) * (size_t)n_cand, st)) != cudaSuccess ||
            (e = cudaMemsetAsync(s->cur, k <= kClusterSeeds ? 0xff : 0, sizeof(int32_t), st)) != cudaSuccess) {
            rc = cuda_fail(e, "screen setup");
            break;
        }
        k_features<<<grid_of(s, g->n, 256), 256, 0, st>>>(g->row_ptr, g->out_ptr, g->n, (float)beta, (float)gamma, s->x);
        // one candidate = set its seed bits, forward, add sum(p) into its score, clear the
        // bits and advance the device-side candidate index; captured once, replayed n_cand times
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        if ((e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) {
            rc = cuda_fail(e, "capture");
            break;
        }
        const int gk = std::min<int32_t>(k, 1024);
        const bool clustered = k <= kClusterSeeds;
        if (clustered) {
            k_seed_next<<<kSeedCtas, kSeedThreads, 0, st>>>(d_cand, k, n_cand, s->cur, g->out_ptr, g->out_dst, s->cnt, s->x);
        } else {
            k_seed_bits<<<1, 256, 0, st>>>(d_cand, k, s->cur, 1.f, 0, s->x);
            k_seed_count<<<gk, 256, 0, st>>>(d_cand, k, s->cur, g->out_ptr, g->out_dst, 1, s->cnt);
            k_seed_feat<<<gk, 256, 0, st>>>(d_cand, k, s->cur, g->out_ptr, g->out_dst, s->cnt, s->x);
        }
        sg_forward(s, g, nullptr, d_scores, false, st);
        if (!clustered) {
            k_seed_count<<<gk, 256, 0, st>>>(d_cand, k, s->cur, g->out_ptr, g->out_dst, -1, s->cnt);
            k_seed_feat<<<gk, 256, 0, st>>>(d_cand, k, s->cur, g->out_ptr, g->out_dst, s->cnt, s->x);
            k_seed_bits<<<1, 256, 0, st>>>(d_cand, k, s->cur, 0.f, 1, s->x);
        }
        e = cudaStreamEndCapture(st, &graph);
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "screen graph");
            break;
        }
        for (int32_t c = 0; c < n_cand && e == cudaSuccess; ++c) e = cudaGraphLaunch(exec, st);
        if (clustered)   // take the last candidate's seed features back
            k_seed_next<<<kSeedCtas, kSeedThreads, 0, st>>>(d_cand, k, n_cand, s->cur, g->out_ptr, g->out_dst, s->cnt, s->x);
        if (e == cudaSuccess) e = cudaMemcpyAsync(scores_out, d_scores, sizeof(float) * (size_t)n_cand, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaGraphExecDestroy(exec);
        if (e != cudaSuccess) rc = cuda_fail(e, "screen");
        else rc = sg_check_tc(s, st);
    } while (0);
    cudaFree(d_cand);
    cudaFree(d_scores);
    if (ev) cudaEventDestroy(ev);
    if (st) cudaStreamDestroy(st);
    return rc;
}
