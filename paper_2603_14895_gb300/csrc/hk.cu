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

constexpr int kHkUnroll = 8;   // gathered rows in flight per node

// One synchronous step.  TL lanes take the segment of 4 * TL realizations of one node; the
// nodes come in degree-bucket order, so that the teams of a warp have rows of similar
// length.  changes: (node, realization) pairs whose opinion changed.
template <int TL>
__global__ void __launch_bounds__(256) k_hk_step(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                                 const int32_t *__restrict__ order, int32_t n, int32_t R, int32_t Rp,
                                                 float eps, const float *__restrict__ cur, float *__restrict__ nxt,
                                                 unsigned long long *changes) {
    constexpr int TPW = 32 / TL;
    const int lane = threadIdx.x & 31, tl = lane % TL, g0 = lane - tl;
    const int segs = Rp / (4 * TL);     // segments of a node's row
    const int64_t items = (int64_t)n * segs;
    const int64_t team = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * TPW + lane / TL;
    const int64_t nteams = (((int64_t)gridDim.x * blockDim.x) >> 5) * TPW;
    unsigned long long ch = 0ull;
    // node, segment and arcs of the team's next item
    int32_t i = -1, seg = 0, beg = 0, end = 0;
    auto fetch = [&](int64_t it) {
        i = -1;
        beg = end = 0;
        if (it < items) {
            const int64_t q = segs == 1 ? it : it / segs;
            seg = (int32_t)(it - q * segs);
            i = __ldg(order + q);
            beg = __ldg(row_ptr + i);
            end = __ldg(row_ptr + i + 1);
        }
    };
    fetch(team);
    // the whole warp iterates together (the column indices are handed out by shuffles)
    for (int64_t it = team; __any_sync(0xffffffffu, i >= 0); it += nteams) {
        const int32_t node = i, b = beg, e = end;
        const float *base = cur + (seg * TL + tl) * 4;
        const size_t own = (size_t)(node < 0 ? 0 : node) * Rp;
        const int32_t r0 = (seg * TL + tl) * 4;
        int32_t mine = tl < kHkUnroll && b + tl < e ? __ldg(col + b + tl) : -1;
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
        if (node >= 0) h = __ldg(reinterpret_cast<const float4 *>(base + own));
        fetch(it + nteams);
        const float hi[4] = {h.x, h.y, h.z, h.w};
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
        int32_t cnt[4] = {0, 0, 0, 0};
        for (int32_t a = b; __any_sync(0xffffffffu, a < e); a += kHkUnroll) {
            float4 hj[kHkUnroll];
            unsigned has = 0u;
#pragma unroll
            for (int u = 0; u < kHkUnroll; ++u) {
                const int32_t j = __shfl_sync(0xffffffffu, mine, g0 + u);
                if (j >= 0) {
                    hj[u] = __ldg(reinterpret_cast<const float4 *>(base + (size_t)j * Rp));
                    has |= 1u << u;
                }
            }
            const int32_t an = a + kHkUnroll + tl;
            mine = tl < kHkUnroll && an < e ? __ldg(col + an) : -1;
#pragma unroll
            for (int u = 0; u < kHkUnroll; ++u) {
                const float x[4] = {hj[u].x, hj[u].y, hj[u].z, hj[u].w};
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if ((has >> u & 1u) && fabsf(__fsub_rn(hi[v], x[v])) < eps) {
                        sum[v] = __fadd_rn(sum[v], x[v]);
                        ++cnt[v];
                    }
                }
            }
        }
        if (node >= 0) {
            float out[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                out[v] = cnt[v] > 0 ? __fdiv_rn(sum[v], (float)cnt[v]) : hi[v];
                if (r0 + v < R && out[v] != hi[v]) ++ch;
            }
            *reinterpret_cast<float4 *>(nxt + own + r0) = make_float4(out[0], out[1], out[2], out[3]);
        }
    }
    __shared__ unsigned long long s_ch;
    if (threadIdx.x == 0) s_ch = 0ull;
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ch += __shfl_xor_sync(0xffffffffu, ch, o);
    if (lane == 0 && ch) atomicAdd(&s_ch, ch);
    __syncthreads();
    if (threadIdx.x == 0 && s_ch) atomicAdd(changes, s_ch);
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
    const int TL = Rp % 128 == 0 ? 32 : (Rp % 64 == 0 ? 16 : 8);
    const int64_t teams = (int64_t)n * (Rp / (4 * TL));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((teams * TL + 255) / 256, (int64_t)g->sm_count * 8));
    float *cur = buf0, *nxt = buf1;
    for (int32_t k = 1; k <= T && n > 0; ++k) {
        if (TL == 32)
            k_hk_step<32><<<grid, 256, 0, s>>>(g->row_ptr, g->col, g->rows_sorted, n, R, Rp, eps_f, cur, nxt, d_ch + k);
        else if (TL == 16)
            k_hk_step<16><<<grid, 256, 0, s>>>(g->row_ptr, g->col, g->rows_sorted, n, R, Rp, eps_f, cur, nxt, d_ch + k);
        else
            k_hk_step<8><<<grid, 256, 0, s>>>(g->row_ptr, g->col, g->rows_sorted, n, R, Rp, eps_f, cur, nxt, d_ch + k);
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
