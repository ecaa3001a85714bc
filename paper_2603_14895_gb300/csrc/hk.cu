// hk.cu -- Hegselmann-Krause opinion dynamics (Appendix A.2): continuous opinions, R
// independent opinion vectors (realizations) updated synchronously.  At step k node i
// takes the mean of the opinions h_j of its in-neighbours j (arcs with multiplicity)
// with |h_i - h_j| < eps; with none it keeps its opinion (the NaN case of the appendix).
//
// GB300 layout: opinions are [n][Rp] float32 (Rp = R rounded up to 32), so that a gathered
// in-neighbour is one contiguous row segment of 128 to 512 bytes.  The step is bound by the
// latency and the bandwidth of those random row reads; a team of 8, 16 or 32 lanes takes 16
// bytes each of one node's segment, two to four nodes to a warp, with eight rows in flight
// per node and the next node's indices already loaded.  The arcs of a row are visited in
// col_idx order and summed in single precision with one division, the order the
// definition's sum is taken in, so that the result is exactly the sequential one.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fsgp_internal.cuh"

namespace fsgp {
namespace {

// [R][n] (caller) -> [n][Rp] (padding realizations get 0), by 32 x 32 tiles through shared
// memory so that both sides are read and written along their rows; *bad is set when an
// opinion is not finite.  (One thread per element read or wrote with a stride of n floats;
// with the step kernel's change, BA n = 1M, R = 64, T = 30: 62.6 to 32.9 ms.)
__global__ void __launch_bounds__(256) k_hk_in(const float *__restrict__ src, int32_t n, int32_t R, int32_t Rp,
                                               float *dst, int32_t *bad) {
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t nv = ((int64_t)n + 31) / 32, tiles = nv * (Rp / 32);
    bool finite = true;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t v0 = t % nv * 32;
        const int32_t r0 = (int32_t)(t / nv) * 32;
#pragma unroll
        for (int j = ty; j < 32; j += 8) {
            const bool has = r0 + j < R && v0 + tx < n;
            const float x = has ? src[(size_t)(r0 + j) * n + v0 + tx] : 0.0f;
            finite &= isfinite(x);
            tile[j][tx] = x;
        }
        __syncthreads();
#pragma unroll
        for (int j = ty; j < 32; j += 8)
            if (v0 + j < n) dst[(size_t)(v0 + j) * Rp + r0 + tx] = tile[tx][j];
        __syncthreads();
    }
    if (!finite) atomicExch(bad, 1);
}

// [n][Rp] -> [R][n]
__global__ void __launch_bounds__(256) k_hk_out(const float *__restrict__ src, int32_t n, int32_t R, int32_t Rp,
                                                float *dst) {
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t nv = ((int64_t)n + 31) / 32, tiles = nv * (Rp / 32);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t v0 = t % nv * 32;
        const int32_t r0 = (int32_t)(t / nv) * 32;
#pragma unroll
        for (int j = ty; j < 32; j += 8)
            if (v0 + j < n) tile[j][tx] = src[(size_t)(v0 + j) * Rp + r0 + tx];
        __syncthreads();
#pragma unroll
        for (int j = ty; j < 32; j += 8)
            if (r0 + j < R && v0 + tx < n) dst[(size_t)(r0 + j) * n + v0 + tx] = tile[tx][j];
        __syncthreads();
    }
}

constexpr int kHkUnroll = 8;     // gathered rows in flight per node
constexpr int kHkStages = 4;     // blocks of rows in flight for a long row

// Sixteen bytes of an in-neighbour's opinions; infinities (never within eps) without one.
// In assembly so that a round's loads are issued one behind the other.
__device__ __forceinline__ float4 hk_row16(const float *p, bool has) {
    float4 r;
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n mov.b32 %0, 0x7f800000;\n mov.b32 %1, 0x7f800000;\n"
                 " mov.b32 %2, 0x7f800000;\n mov.b32 %3, 0x7f800000;\n @p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n}"
                 : "=&f"(r.x), "=&f"(r.y), "=&f"(r.z), "=&f"(r.w) : "l"(p), "r"((uint32_t)has));
    return r;
}

// The four realizations of one lane: own opinions, running sum and count of neighbours
// within eps, in the order the arcs are added.
struct HkAcc {
    float h[4], sum[4];
    int32_t cnt[4];
    __device__ __forceinline__ HkAcc(const float4 &own) : h{own.x, own.y, own.z, own.w}, sum{}, cnt{} {}
    __device__ __forceinline__ void add(const float4 &o, float eps) {
        const float x[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (fabsf(__fsub_rn(h[v], x[v])) < eps) {
                sum[v] = __fadd_rn(sum[v], x[v]);
                ++cnt[v];
            }
    }
    // writes the new opinions, returns how many of the realizations r0 .. R-1 changed
    __device__ __forceinline__ uint32_t store(float *p, int32_t r0, int32_t R) const {
        float out[4];
        uint32_t ch = 0u;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            out[v] = cnt[v] > 0 ? __fdiv_rn(sum[v], (float)cnt[v]) : h[v];
            if (r0 + v < R && out[v] != h[v]) ++ch;
        }
        *reinterpret_cast<float4 *>(p) = make_float4(out[0], out[1], out[2], out[3]);
        return ch;
    }
};

// One synchronous step.  changes: (node, realization) pairs whose opinion changed.
// TL lanes take the segment of 4 * TL realizations of one node; the nodes come in
// degree-bucket order, so that the teams of a warp have rows of similar length.
// order may be null (node order) when there are no long rows.
// The first n_long * segments CTAs take one long row each: its sum has to run through all
// arcs in order, so one team adds while the whole CTA (256 threads) copies the next kHkStages blocks of
// rows to shared memory (a team on its own waits a memory latency for every eight arcs, and
// the hub of a BA graph then outlasts the step: BA n = 1M, R = 64, a step 1.55 ms so, 0.66 with
// the copies ahead and the padding arcs' infinities in place of their tests).
template <int TL>
__global__ void __launch_bounds__(256) k_hk_step(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                                 const int32_t *__restrict__ order, int32_t n, int32_t n_long, int32_t R,
                                                 int32_t Rp, float eps, const float *__restrict__ cur,
                                                 float *__restrict__ nxt, unsigned long long *changes) {
    constexpr int TPW = 32 / TL;
    constexpr int RPS = 256 / TL;       // rows of a block
    __shared__ float4 s_row[kHkStages][256];
    const int tid = threadIdx.x, lane = tid & 31, tl = lane % TL, g0 = lane - tl;
    const int segs = Rp / (4 * TL);     // segments of a node's row
    const int64_t long_items = (int64_t)n_long * segs;
    unsigned long long ch = 0ull;
    if ((int64_t)blockIdx.x < long_items) {
        const int32_t q = (int32_t)(blockIdx.x / segs), seg = (int32_t)blockIdx.x - q * segs;
        const int32_t node = __ldg(order + q), b = __ldg(row_ptr + node), e = __ldg(row_ptr + node + 1);
        const int t = tid % TL;         // this thread's 16 bytes of row tid / TL of a block
        const float *base = cur + (seg * TL + t) * 4;
        const int32_t r0 = (seg * TL + t) * 4;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_row[0][tid]);
        const uint32_t len = (uint32_t)(e - b), blocks = (len + RPS - 1) / RPS;
        auto col_of = [&](uint32_t k) {
            const uint32_t at = k * RPS + tid / TL;   // (past the row's end by up to kHkStages blocks)
            return at < len ? __ldg(col + b + at) : -1;
        };
        int32_t c = col_of(0);
        auto copy = [&](uint32_t k) {    // block k, whose column index is in c; c of the next
            if (c >= 0)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + k % kHkStages * 4096u),
                             "l"(base + (size_t)c * Rp));
            asm volatile("cp.async.commit_group;");
            c = col_of(k + 1);
        };
        for (uint32_t k = 0; k < kHkStages - 1; ++k) copy(k);
        HkAcc acc(__ldg(reinterpret_cast<const float4 *>(base + (size_t)node * Rp)));
        for (uint32_t k = 0; k < blocks; ++k) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kHkStages - 2));
            __syncthreads();            // block k has landed; block k - 1 has been added
            copy(k + kHkStages - 1);
            if (tid < TL) {
                const float4 *x = s_row[k % kHkStages] + t;
                const int m = (int)min((uint32_t)RPS, len - k * RPS);
                if (m == RPS) {
#pragma unroll
                    for (int u = 0; u < RPS; ++u) acc.add(x[u * TL], eps);
                } else {
                    for (int u = 0; u < m; ++u) acc.add(x[u * TL], eps);
                }
            }
        }
        asm volatile("cp.async.wait_group 0;");
        if (tid < TL) ch = acc.store(nxt + (size_t)node * Rp + r0, r0, R);
    } else {
        const int64_t items = (int64_t)n * segs;
        const int64_t team = ((((int64_t)blockIdx.x - long_items) * blockDim.x + tid) >> 5) * TPW + lane / TL + long_items;
        const int64_t nteams = ((((int64_t)gridDim.x - long_items) * blockDim.x) >> 5) * TPW;
        // node, segment and arcs of the team's next item
        int32_t i = -1, seg = 0, beg = 0, end = 0;
        auto fetch = [&](int64_t it) {
            i = -1;
            beg = end = 0;
            if (it < items) {
                const int64_t q = segs == 1 ? it : it / segs;
                seg = (int32_t)(it - q * segs);
                i = order ? __ldg(order + q) : (int32_t)q;
                beg = __ldg(row_ptr + i);
                end = __ldg(row_ptr + i + 1);
            }
        };
        fetch(team);
        // the whole warp iterates together (the column indices are handed out by shuffles)
        for (int64_t it = team; __any_sync(0xffffffffu, i >= 0); it += nteams) {
            const int32_t node = i, r0 = (seg * TL + tl) * 4;
            const uint32_t e = end;
            uint32_t b = beg;
            const float *base = cur + r0;
            const size_t own = (size_t)max(node, 0) * Rp;
            int32_t mine = tl < kHkUnroll && arc_in(b, tl, e) ? __ldg(col + b + tl) : -1;
            HkAcc acc(hk_row16(base + own, node >= 0));
            fetch(it + nteams);
            while (__any_sync(0xffffffffu, b < e)) {
                float4 x[kHkUnroll];
#pragma unroll
                for (int u = 0; u < kHkUnroll; ++u) {
                    const int32_t j = __shfl_sync(0xffffffffu, mine, g0 + u);
                    x[u] = hk_row16(base + (size_t)max(j, 0) * Rp, j >= 0);
                }
                b += kHkUnroll;
                mine = tl < kHkUnroll && arc_in(b, tl, e) ? __ldg(col + b + tl) : -1;
#pragma unroll
                for (int u = 0; u < kHkUnroll; ++u) acc.add(x[u], eps);
            }
            if (node >= 0) ch += acc.store(nxt + own + r0, r0, R);
        }
    }
    __shared__ unsigned long long s_ch;
    if (tid == 0) s_ch = 0ull;
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ch += __shfl_xor_sync(0xffffffffu, ch, o);
    if (lane == 0 && ch) atomicAdd(&s_ch, ch);
    __syncthreads();
    if (tid == 0 && s_ch) atomicAdd(changes, s_ch);
}

}  // namespace
}  // namespace fsgp

using namespace fsgp;

extern "C" int fsgp_hk(const fsgp_graph *gc, const float *h0, int32_t R, int32_t T, double eps, float *h_out,
                       uint64_t *changes, uint32_t flags, void *stream) {
    set_error("");
    fsgp_graph *g = const_cast<fsgp_graph *>(gc);
    if (!g || !h0 || !h_out) return fail(FSGP_EINVAL, "NULL argument");
    if (R < 1 || R > kMaxR) return fail(FSGP_EINVAL, "R must be in [1, 4096]");
    if (T < 0) return fail(FSGP_EINVAL, "T must be >= 0");
    if (!(eps >= 0.0) || std::isinf(eps)) return fail(FSGP_EINVAL, "eps must be finite and >= 0");
    if (flags != FSGP_PTR_HOST && flags != FSGP_PTR_DEVICE) return fail(FSGP_EINVAL, "bad flags");
    int dev = 0;
    FSGP_CUDA(cudaGetDevice(&dev));
    if (dev != g->device) return fail(FSGP_EINVAL, "current device differs from the graph's device");
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t n = g->n;
    const int32_t Rp = (R + 31) & ~31;
    const int64_t m = (int64_t)R * n;
    if (flags == FSGP_PTR_HOST)
        for (int64_t i = 0; i < m; ++i)
            if (std::isnan(h0[i]) || std::isinf(h0[i])) return fail(FSGP_EINVAL, "opinions must be finite");
    // workspace: two [n][Rp] buffers, the per-step change counts, a flag, and (host
    // buffers) a [R][n] staging area
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_state = al(sizeof(float) * (size_t)n * Rp);
    const size_t b_ch = al(sizeof(unsigned long long) * ((size_t)T + 1));
    const size_t b_flag = al(sizeof(int32_t));
    const size_t b_stage = flags == FSGP_PTR_HOST ? al(sizeof(float) * (size_t)std::max<int64_t>(m, 1)) : 0;
    int rc = ensure_workspace(g, 2 * b_state + b_ch + b_flag + b_stage);
    if (rc) return rc;
    uint8_t *ws = (uint8_t *)g->ws.ptr;
    float *buf0 = (float *)ws;
    float *buf1 = (float *)(ws + b_state);
    unsigned long long *d_ch = (unsigned long long *)(ws + 2 * b_state);
    int32_t *d_flag = (int32_t *)(ws + 2 * b_state + b_ch);
    float *stage = b_stage ? (float *)(ws + 2 * b_state + b_ch + b_flag) : nullptr;
    // 32 x 32 tiles of the transposes
    const int grid_el = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)n + 31) / 32 * (Rp / 32),
                                                                     (int64_t)g->sm_count * 16));
    const float *src = h0;
    FSGP_CUDA(cudaMemsetAsync(d_flag, 0, sizeof(int32_t), s));
    if (flags == FSGP_PTR_HOST) {
        if (m > 0) FSGP_CUDA(cudaMemcpyAsync(stage, h0, sizeof(float) * (size_t)m, cudaMemcpyHostToDevice, s));
        src = stage;
    }
    if (n > 0) k_hk_in<<<grid_el, 256, 0, s>>>(src, n, R, Rp, buf0, d_flag);
    if (flags == FSGP_PTR_DEVICE && m > 0) {
        int32_t bad = 0;
        FSGP_CUDA(cudaMemcpyAsync(&bad, d_flag, sizeof bad, cudaMemcpyDeviceToHost, s));
        FSGP_CUDA(cudaStreamSynchronize(s));
        if (bad) return fail(FSGP_EINVAL, "opinions must be finite");
    }
    FSGP_CUDA(cudaMemsetAsync(d_ch, 0, sizeof(unsigned long long) * ((size_t)T + 1), s));
    const float eps_f = (float)eps;
    // lanes per node: as wide a segment as divides the row (the column indices are loaded
    // once per segment)
    int TL = Rp % 128 == 0 ? 32 : (Rp % 64 == 0 ? 16 : 8);
    // long rows: at least 256 in-arcs and sixteen times the mean, a power of two, so that they
    // are the first of the degree-bucket order; from 32 arcs and four times the mean where four
    // CTAs per SM hold them all, since a small graph's step lasts as long as its longest row
    int lb = 8;
    while (lb < 31 && ((int64_t)n << lb) < 16 * g->nnz) ++lb;
    for (int b = 5; b < lb; ++b)
        if (((int64_t)n << b) >= 4 * g->nnz && (int64_t)g->cls.bucket_start[b] * (Rp / (4 * TL)) <= (int64_t)g->sm_count * 4)
            lb = b;
    const int32_t n_long = g->cls.bucket_start[lb];
    // Where no row is long and every node has its teams at once, a step is the chain of one
    // row: the narrowest teams (four nodes' chains to a warp) on CTAs of 128 threads, which
    // spread over more SMs, and in node order, since the degree order would gain nothing and is
    // one more load in the chain.  (ER, mean degree 4 to 6, R = 33..64, 20 steps: n = 1000 225 us
    // with teams of 16 on CTAs of 256 threads, 184 so; n = 3000 224 and 184; n = 1500, mean degree
    // 16, R = 50 267 and 186; a warp per node with 4 bytes per lane 186, 186 and 228.)
    const bool one_round = n_long == 0 && (int64_t)n * (Rp / 32) * 8 <= (int64_t)g->sm_count * 8 * 256;
    if (one_round) TL = 8;
    const int threads = one_round ? 128 : 256;   // (long rows want 256)
    const int segs = Rp / (4 * TL);
    const int64_t teams = (int64_t)(n - n_long) * segs;
    const int grid = (int)(std::min<int64_t>((teams * TL + threads - 1) / threads, (int64_t)g->sm_count * (2048 / threads)) +
                           (int64_t)n_long * segs);
    const int32_t *order = n_long == 0 && teams * TL <= (int64_t)g->sm_count * 8 * 256 ? nullptr : g->rows_sorted;
    float *cur = buf0, *nxt = buf1;
    for (int32_t k = 1; k <= T && n > 0; ++k) {
        if (TL == 32)
            k_hk_step<32><<<grid, threads, 0, s>>>(g->row_ptr, g->col, order, n, n_long, R, Rp, eps_f, cur, nxt, d_ch + k);
        else if (TL == 16)
            k_hk_step<16><<<grid, threads, 0, s>>>(g->row_ptr, g->col, order, n, n_long, R, Rp, eps_f, cur, nxt, d_ch + k);
        else
            k_hk_step<8><<<grid, threads, 0, s>>>(g->row_ptr, g->col, order, n, n_long, R, Rp, eps_f, cur, nxt, d_ch + k);
        std::swap(cur, nxt);
    }
    FSGP_CUDA(cudaGetLastError());
    float *dst = flags == FSGP_PTR_HOST ? stage : h_out;
    if (n > 0) k_hk_out<<<grid_el, 256, 0, s>>>(cur, n, R, Rp, dst);
    FSGP_CUDA(cudaGetLastError());
    if (flags == FSGP_PTR_HOST) {
        if (m > 0) FSGP_CUDA(cudaMemcpyAsync(h_out, stage, sizeof(float) * (size_t)m, cudaMemcpyDeviceToHost, s));
        if (changes)
            FSGP_CUDA(cudaMemcpyAsync(changes, d_ch, sizeof(uint64_t) * ((size_t)T + 1), cudaMemcpyDeviceToHost, s));
        FSGP_CUDA(cudaStreamSynchronize(s));
    } else if (changes) {
        FSGP_CUDA(cudaMemcpyAsync(changes, d_ch, sizeof(uint64_t) * ((size_t)T + 1), cudaMemcpyDeviceToDevice, s));
    }
    return FSGP_OK;
}
