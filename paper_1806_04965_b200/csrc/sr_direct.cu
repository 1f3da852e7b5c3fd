// CUDA-core kernels of the frame update: the node update
//     x_v = sigma(b_v + sum_e f_e(theta_e, x_src(e)))          (paper Sec. A1.2)
// for every node of one launch group, in one launch.  They serve the fp32 mode, the dense heads and
// the few-channel nodes that are bound by memory traffic, and they are the reference engine the
// tensor-core kernel can be switched against.  Accumulation is fp32 in every mode.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "sr_input.cuh"
#include "sr_kernels.h"

namespace {

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void from_f(float* p, float v) { *p = v; }
__device__ __forceinline__ void from_f(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ void load4(const float* p, float (&v)[4])
{
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4])
{
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
    v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
}

// One value, or four, of a state; BESIDE: past L1 (see SrFollow).
template <bool BESIDE>
__device__ __forceinline__ float head_load1(const float* p) { return BESIDE ? sr_load_past_l1(p) : *p; }
template <bool BESIDE>
__device__ __forceinline__ float head_load1(const __nv_bfloat16* p)
{
    return BESIDE ? __uint_as_float((uint32_t)sr_load_past_l1(reinterpret_cast<const unsigned short*>(p)) << 16) : to_f(*p);
}
template <bool BESIDE>
__device__ __forceinline__ void head_load4(const float* p, float (&v)[4])
{
    if (!BESIDE) return load4(p, v);
    const float4 q = sr_load_past_l1(reinterpret_cast<const float4*>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <bool BESIDE>
__device__ __forceinline__ void head_load4(const __nv_bfloat16* p, float (&v)[4])
{
    if (!BESIDE) return load4(p, v);
    const uint2 q = sr_load_past_l1(reinterpret_cast<const uint2*>(p));
    v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
    v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
}

__device__ __forceinline__ void store4(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float (&v)[4])
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

constexpr int kItemSlices = 1 << 30;   // SrDirectItem::pad_: the block's warps share the pixels and take slices of the reduction
constexpr int kPix = 4;            // pixels per warp (conv nodes)
constexpr int kWarps = 4;          // warps per block
constexpr int kDenseB = 8;         // samples per warp (dense nodes)

// Conv node that conv_tile does not take (see sr_direct_untiled), or that has a weight which is not finite: a tap outside the image is
// left out here, while conv_tile multiplies it by zero.  A block covers kWarps*kPix consecutive pixels of one sample at a time; lanes
// run over output channels, so weight reads ([K][C_out] rows) and state writes (NHWC) are coalesced and the input
// reads are warp-uniform broadcasts.
template <typename T, bool ANY_ITEM>
__device__ void conv_item(const SrDevNode& nd, const SrDevEdge* edges, const SrDirectItem& it, int prev, int cur,
                          float* out_f32)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int HW = nd.H * nd.W;
    int b = it.b0, n_pix = kWarps * kPix, c_first = 0, c_end = nd.C;
    if (ANY_ITEM && nd.untiled == (sizeof(T) == 2 ? 2 : 4)) {                                                       // conv_tile's items: pixels and channels of their own
        const int qlog = (it.pad_ >> 24) & 15;
        b = it.b0 < 0 ? ~it.b0 : it.b0;
        n_pix = ((it.pad_ & kItemSlices ? 32 : kWarps * 32) >> qlog) * (it.b0 < 0 ? 4 : 1);
        c_first = it.pad_ & 0xFFFFFF;
        c_end = min(nd.C, c_first + (4 << qlog));
    }
    T* dst = static_cast<T*>(nd.state[cur]) + (size_t)b * HW * nd.C;
    const int p_end = min(HW, it.p0 + n_pix);
    for (int pbase = it.p0 + warp * kPix; pbase < p_end; pbase += kWarps * kPix) {
        int oy[kPix], ox[kPix];
        bool pv[kPix];
#pragma unroll
        for (int j = 0; j < kPix; ++j) {
            const int p = pbase + j;
            pv[j] = p < p_end;
            oy[j] = pv[j] ? p / nd.W : 0;
            ox[j] = pv[j] ? p % nd.W : 0;
        }
        for (int co0 = c_first; co0 < c_end; co0 += 32) {
            const int co = co0 + lane;
            const bool cv = co < c_end;
            float acc[kPix];
#pragma unroll
            for (int j = 0; j < kPix; ++j) acc[j] = 0.f;
            for (int ei = 0; ei < nd.n_edges; ++ei) {
                const SrDevEdge& e = edges[nd.first_edge + ei];
                const T* src = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)b * e.Hs * e.Ws * e.Cs;
                const bool vec = (e.Cs & 3) == 0;
                for (int ky = 0; ky < e.k; ++ky)
                    for (int kx = 0; kx < e.k; ++kx) {
                        const T* xp[kPix];
                        bool ok[kPix];
                        bool any = false;
#pragma unroll
                        for (int j = 0; j < kPix; ++j) {
                            const int iy = oy[j] * e.stride + ky - e.pad, ix = ox[j] * e.stride + kx - e.pad;
                            ok[j] = pv[j] && iy >= 0 && iy < e.Hs && ix >= 0 && ix < e.Ws;
                            xp[j] = src + ((size_t)(ok[j] ? iy : 0) * e.Ws + (ok[j] ? ix : 0)) * e.Cs;
                            any |= ok[j];
                        }
                        if (!any) continue;
                        const float* wp = e.w + (size_t)(ky * e.k + kx) * e.Cs * nd.C + co;
                        if (vec) {
                            for (int ci = 0; ci < e.Cs; ci += 4) {
                                float w[4];
#pragma unroll
                                for (int q = 0; q < 4; ++q) w[q] = cv ? wp[(size_t)(ci + q) * nd.C] : 0.f;
#pragma unroll
                                for (int j = 0; j < kPix; ++j) {
                                    if (!ok[j]) continue;
                                    float x[4];
                                    load4(xp[j] + ci, x);
#pragma unroll
                                    for (int q = 0; q < 4; ++q) acc[j] = fmaf(w[q], x[q], acc[j]);
                                }
                            }
                        } else {
                            for (int ci = 0; ci < e.Cs; ++ci) {
                                const float w = cv ? wp[(size_t)ci * nd.C] : 0.f;
#pragma unroll
                                for (int j = 0; j < kPix; ++j)
                                    if (ok[j]) acc[j] = fmaf(w, to_f(xp[j][ci]), acc[j]);
                            }
                        }
                    }
            }
            if (cv) {
                const float bias = nd.bias[co];
#pragma unroll
                for (int j = 0; j < kPix; ++j) {
                    if (!pv[j]) continue;
                    float z = acc[j] + bias;
                    if (nd.act == 1) z = fmaxf(z, 0.f);
                    from_f(dst + (size_t)(pbase + j) * nd.C + co, z);
                    if (out_f32) out_f32[((size_t)b * HW + pbase + j) * nd.C + co] = z;
                }
            }
        }
    }
}

// Conv node with a multiple of four channels.  A thread computes PX consecutive pixels of one sample x 4 channels; the threads of
// a block are 2^qb_log2 channel quads x pixel groups, so weight rows ([K][C_out]) and states (NHWC) are read and written in
// 16-byte vectors by neighbouring threads.  The reduction of an edge is one flat loop over a table in shared memory (offset
// inside the window, filter row and column): no branch per tap, so the loads of several steps are in flight together.  What
// bounds it is the latency of those loads for a small node and the load / store unit for a large one; PX = 4 loads a weight
// vector once for four pixels and is taken when that still leaves threads enough (see sr_direct_conv_items).
// SLICES: the warps of a block take the same 32 threads' worth of outputs and every fourth step of the reduction each, and the first one
// adds the sums, in order: a quarter of the chain of dependent loads, and four times the blocks.  Small CNN, fp32, us per frame before /
// now: at 1 / 16 / 64 / 128 samples 26.0 / 11.1, 42.6 / 24.0, 78.7 / 52.5, 113 / 95.2 (sequential at 1 / 64 / 128 56.6 / 28.3, 125 / 73,
// 176 / 117).
// Measured on B200 (was: a warp per four pixels, lanes over channels, a branch per tap), fp32, us per frame: MNIST net SR at 100
// samples 49 -> 17.5, at one 34 -> 12.6; small CNN at 128 samples 260 -> 114, at one 80 -> 27.
constexpr int kTab = 512;          // table entries at a time
constexpr int kTabSliced = (kWarps - 1) * 32 * 16 * 4 / (int)sizeof(int2);   // its place, where the sums of the slices go as well
template <typename T, int PX, bool SLICES>
__device__ void conv_tile(const SrDevNode& nd, const SrDevEdge* edges, const SrDirectItem& it, int prev, int cur, float* out_f32, int2* tab)
{
    constexpr int kStep = SLICES ? kWarps : 1;
    const int place = SLICES ? (int)threadIdx.x & 31 : (int)threadIdx.x, slice = SLICES ? (int)threadIdx.x >> 5 : 0;
    const int qlog = (it.pad_ >> 24) & 15, c = (it.pad_ & 0xFFFFFF) + 4 * (place & ((1 << qlog) - 1));
    const int HW = nd.H * nd.W, C = nd.C, p_first = it.p0 + (place >> qlog) * PX;
    const bool cv = c < C;
    int oy[PX], ox[PX];
    float acc[PX][4];
#pragma unroll
    for (int j = 0; j < PX; ++j) {
        const int p = p_first + j;
        oy[j] = p < HW ? p / nd.W : 1 << 30;                                     // (a pixel that does not exist lies outside every image)
        ox[j] = p % nd.W;
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
    }
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrDevEdge& e = edges[nd.first_edge + ei];
        const int Hs = e.Hs, Ws = e.Ws, Cs = e.Cs, k = e.k, vec = (Cs & 3) == 0 ? 4 : 1, n = e.K / vec, cg = Cs / vec;
        const T* src = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)it.b0 * Hs * Ws * Cs;
        const float* w = e.w + (cv ? c : 0);
        int y0[PX], x0[PX], o0[PX];
#pragma unroll
        for (int j = 0; j < PX; ++j) {
            y0[j] = (int)((unsigned)oy[j] * (unsigned)e.stride) - e.pad;
            x0[j] = ox[j] * e.stride - e.pad;
            o0[j] = oy[j] < (1 << 30) ? (y0[j] * Ws + x0[j]) * Cs : 0;
            if (oy[j] >= (1 << 30)) y0[j] = -(1 << 30);
        }
        for (int e0 = 0; e0 < n; e0 += kTab) {
            const int m = min(kTab, n - e0);
            __syncthreads();
            for (int i = threadIdx.x; i < m; i += kWarps * 32) {
                const int tap = (e0 + i) / cg, ci = ((e0 + i) % cg) * vec, dy = tap / k, dx = tap % k;
                tab[i] = make_int2((dy * Ws + dx) * Cs + ci, dy << 16 | dx);
            }
            __syncthreads();
            if (vec == 4) {
#pragma unroll 2
                for (int i = slice; i < m; i += kStep) {
                    const int2 t = tab[i];
                    const int dy = t.y >> 16, dx = t.y & 0xFFFF;
                    float4 wv[4];
                    float x[PX][4];
#pragma unroll
                    for (int j = 0; j < PX; ++j) {
                        x[j][0] = x[j][1] = x[j][2] = x[j][3] = 0.f;
                        if ((unsigned)(y0[j] + dy) < (unsigned)Hs && (unsigned)(x0[j] + dx) < (unsigned)Ws) load4(src + o0[j] + t.x, x[j]);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) wv[q] = __ldg(reinterpret_cast<const float4*>(w + (size_t)((e0 + i) * 4 + q) * C));
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int j = 0; j < PX; ++j) {
                            acc[j][0] = fmaf(wv[q].x, x[j][q], acc[j][0]); acc[j][1] = fmaf(wv[q].y, x[j][q], acc[j][1]);
                            acc[j][2] = fmaf(wv[q].z, x[j][q], acc[j][2]); acc[j][3] = fmaf(wv[q].w, x[j][q], acc[j][3]);
                        }
                }
            } else {
#pragma unroll 8
                for (int i = slice; i < m; i += kStep) {
                    const int2 t = tab[i];
                    const int dy = t.y >> 16, dx = t.y & 0xFFFF;
                    const float4 wv = __ldg(reinterpret_cast<const float4*>(w + (size_t)(e0 + i) * C));
#pragma unroll
                    for (int j = 0; j < PX; ++j) {
                        float x = 0.f;
                        if ((unsigned)(y0[j] + dy) < (unsigned)Hs && (unsigned)(x0[j] + dx) < (unsigned)Ws) x = to_f(src[o0[j] + t.x]);
                        acc[j][0] = fmaf(wv.x, x, acc[j][0]); acc[j][1] = fmaf(wv.y, x, acc[j][1]);
                        acc[j][2] = fmaf(wv.z, x, acc[j][2]); acc[j][3] = fmaf(wv.w, x, acc[j][3]);
                    }
                }
            }
        }
    }
    if (SLICES) {
        // (in the table's place: 32 threads x 4 * PX sums per warp but the first)
        static_assert(kTabSliced >= kTab, "the sums of the slices take the table's place");
        float4* sums = reinterpret_cast<float4*>(tab);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PX; ++j)
            if (slice > 0) sums[((slice - 1) * PX + j) * 32 + place] = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
        __syncthreads();
        if (slice > 0) return;
#pragma unroll
        for (int q = 0; q < kWarps - 1; ++q)
#pragma unroll
            for (int j = 0; j < PX; ++j) {
                const float4 a = sums[(q * PX + j) * 32 + place];
                acc[j][0] += a.x; acc[j][1] += a.y; acc[j][2] += a.z; acc[j][3] += a.w;
            }
    }
    if (!cv) return;
    const float4 b = *reinterpret_cast<const float4*>(nd.bias + c);
#pragma unroll
    for (int j = 0; j < PX; ++j) {
        const int p = p_first + j;
        if (p >= HW) continue;
        float z[4] = {acc[j][0] + b.x, acc[j][1] + b.y, acc[j][2] + b.z, acc[j][3] + b.w};
        if (nd.act == 1)
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = fmaxf(z[q], 0.f);
        const size_t o = ((size_t)it.b0 * HW + p) * C + c;
        store4(static_cast<T*>(nd.state[cur]) + o, z);
        if (out_f32) {
#pragma unroll
            for (int q = 0; q < 4; ++q) out_f32[o + q] = z[q];                  // (the caller's buffer: any alignment a float has)
        }
    }
}

// Dense node outside the limits of the head kernels: one warp per output channel and chunk of kDenseB samples; lanes stride over the
// reduction index (coalesced weight and state reads), partial sums meet in a shuffle reduction.
// A mean-dense edge is the dense edge whose weight index is k mod C_in, scaled by 1/(H*W).
template <typename T>
__device__ void dense_item(const SrDevNode& nd, const SrDevEdge* edges, const SrDirectItem& it, int prev, int cur,
                           int B, float* out_f32)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int co = it.p0 + warp;
    if (co >= nd.C) return;
    const int nb = min(kDenseB, B - it.b0);
    float acc[kDenseB];
#pragma unroll
    for (int j = 0; j < kDenseB; ++j) acc[j] = 0.f;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrDevEdge& e = edges[nd.first_edge + ei];
        const int Kx = e.Hs * e.Ws * e.Cs;                      // elements of one source sample
        const T* src = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)it.b0 * Kx;
        const float* wrow = e.w + (size_t)co * e.K;
        const float scale = (e.kind == SR_EDGE_MEAN_DENSE) ? 1.f / (float)(e.Hs * e.Ws) : 1.f;
        float part[kDenseB];
#pragma unroll
        for (int j = 0; j < kDenseB; ++j) part[j] = 0.f;
        for (int k = lane; k < Kx; k += 32) {
            const float w = wrow[(e.kind == SR_EDGE_MEAN_DENSE) ? (k % e.Cs) : k];
#pragma unroll
            for (int j = 0; j < kDenseB; ++j)
                if (j < nb) part[j] = fmaf(w, to_f(src[(size_t)j * Kx + k]), part[j]);
        }
#pragma unroll
        for (int j = 0; j < kDenseB; ++j) acc[j] += part[j] * scale;
    }
#pragma unroll
    for (int j = 0; j < kDenseB; ++j) {
        float v = acc[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        acc[j] = v;
    }
    if (lane == 0) {
        T* dst = static_cast<T*>(nd.state[cur]);
        const float b = nd.bias[co];
        for (int j = 0; j < nb; ++j) {
            float z = acc[j] + b;
            if (nd.act == 1) z = fmaxf(z, 0.f);
            from_f(dst + (size_t)(it.b0 + j) * nd.C + co, z);
            if (out_f32) out_f32[(size_t)(it.b0 + j) * nd.C + co] = z;
        }
    }
}


// Dense and mean-dense heads.  Bound by the latency of their loads, so as many as possible are in flight together, and
// everything a block needs to know arrives as a kernel parameter (tables in global memory cost a dependent round trip each:
// item, node, edge).
// Measured on B200, us per launch, before (one sample and up to 16 outputs per block of 128 threads, tables in global memory)
// -> now: 784 -> 128 fp32 at one sample 6.9 -> 2.5; 8192 -> 10 bf16 at one sample 18.3 -> 4.2, at 128 samples beside the
// tensor-core kernel 41 -> 20; mean of 8 x 8 x 256, then 256 -> 43, at 128 samples beside that kernel 71 -> 19.5.
constexpr int kHeadThreads = 256, kHeadWarps = kHeadThreads / 32;
constexpr int kHeadMaxC = 1024;    // channels of a node's mean-dense sources together

struct HeadParams {
    SrFrameArgs fr;
    SrInputPart in;                // the frame input's blocks come first (n_blocks = 0: none)
    int32_t n_nodes, B, follow, direct;      // direct: edges with R = 0 that leave an input node read the caller's frame (its
                                             // copy in the state buffer is being made by this launch)
    int32_t first_block[SR_HEAD_NODES + 1];
    SrHeadNode nodes[SR_HEAD_NODES];
};
static_assert(sizeof(HeadParams) <= 4000, "kernel parameters");

template <typename T>
__device__ __forceinline__ const T* head_source(const HeadParams& P, const SrFrame& F, const SrHeadEdge& e)
{
    const int prev = (int)(F.t & 1);
    if (P.direct && e.R == 0 && e.slot >= 0) return reinterpret_cast<const T*>(sr_frame_input(P.fr, F, e.slot));
    return static_cast<const T*>(e.src[e.R ? prev : prev ^ 1]);
}

// Nodes with dense edges only: a block takes CO outputs of S samples; its threads stride over the reduction index in vectors
// of four, every thread keeps S x CO partial sums (a weight vector serves S samples).  The sums of a warp meet by halving,
// those of the warps in shared memory in a fixed order.
template <typename T, int S, int CO, bool WithInput, bool BESIDE>
__global__ void __launch_bounds__(kHeadThreads) sr_head_kernel(const __grid_constant__ HeadParams P)
{
    __shared__ float red[kHeadWarps][32];
    __shared__ int2 tap[WithInput ? 128 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    sr_begin(P.follow);
    const SrFrame F = sr_frame(P.fr);
    int bx = (int)blockIdx.x, ni = 0;
    if (WithInput && (bx -= P.in.n_blocks) < 0) {
        sr_input_block<BESIDE>(P.in, P.fr, F, (int)blockIdx.x, tap);
        sr_end(P.follow);
        return;
    }
    while (ni + 1 < P.n_nodes && bx >= P.first_block[ni + 1]) ++ni;
    const SrHeadNode& nd = P.nodes[ni];
    const int co_blocks = (nd.C + CO - 1) / CO, bi = bx - P.first_block[ni], b0 = (bi / co_blocks) * S, co0 = (bi % co_blocks) * CO;
    const int nco = min(CO, nd.C - co0), cur = (int)((F.t + 1) & 1);
    float* const out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    float acc[S][CO];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int o = 0; o < CO; ++o) acc[s][o] = 0.f;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrHeadEdge& e = nd.edges[ei];
        const int K = e.K;
        const T* src = head_source<T>(P, F, e);
        const T* x[S];
        const float* w[CO];
#pragma unroll
        for (int s = 0; s < S; ++s) x[s] = src + (size_t)min(b0 + s, P.B - 1) * K;   // samples and rows beyond
#pragma unroll
        for (int o = 0; o < CO; ++o) w[o] = e.w + (size_t)(co0 + min(o, nco - 1)) * K;                                          // the last repeat it
        if ((K & 3) == 0) {
#pragma unroll(S == 1 ? 4 : 1)
            for (int k = 4 * tid; k < K; k += 4 * kHeadThreads) {
                float4 wv[CO];
                float xv[S][4];
#pragma unroll
                for (int s = 0; s < S; ++s) head_load4<BESIDE>(x[s] + k, xv[s]);
#pragma unroll
                for (int o = 0; o < CO; ++o) wv[o] = __ldg(reinterpret_cast<const float4*>(w[o] + k));
#pragma unroll
                for (int o = 0; o < CO; ++o)
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        acc[s][o] = fmaf(wv[o].x, xv[s][0], acc[s][o]); acc[s][o] = fmaf(wv[o].y, xv[s][1], acc[s][o]);
                        acc[s][o] = fmaf(wv[o].z, xv[s][2], acc[s][o]); acc[s][o] = fmaf(wv[o].w, xv[s][3], acc[s][o]);
                    }
            }
        } else {
            for (int k = tid; k < K; k += kHeadThreads)
#pragma unroll
                for (int o = 0; o < CO; ++o) {
                    const float wk = __ldg(w[o] + k);
#pragma unroll
                    for (int s = 0; s < S; ++s) acc[s][o] = fmaf(wk, head_load1<BESIDE>(x[s] + k), acc[s][o]);
                }
        }
    }
    // sums over the lanes: while more than one value is left, the step with distance d keeps the half that matches the lane's
    // bit d; then plain butterflies.  Lane l ends with value l / (32 / (S * CO)).
    constexpr int N = S * CO;
    static_assert(N <= 32 && (N & (N - 1)) == 0, "lane layout");
    float v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = acc[i / CO][i % CO];
#pragma unroll
    for (int d = 16, n = N; d > 0; d >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (lane & d) != 0;
#pragma unroll
            for (int i = 0; i < N / 2; ++i)
                if (i < n) {
                    const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
                }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
        }
    }
    if (lane % (32 / N) == 0) red[warp][lane / (32 / N)] = v[0];
    __syncthreads();
    if (tid < N) {
        const int b = b0 + tid / CO, o = tid % CO;
        if (o < nco && b < P.B) {
            float z = nd.bias[co0 + o];
#pragma unroll
            for (int q = 0; q < kHeadWarps; ++q) z += red[q][tid];
            if (nd.act == 1) z = fmaxf(z, 0.f);
            from_f(static_cast<T*>(nd.state[cur]) + (size_t)b * nd.C + co0 + o, z);
            if (out) out[(size_t)b * nd.C + co0 + o] = z;
        }
    }
    sr_end(P.follow);
}

// Nodes with a mean-dense edge: a block takes one sample and mean_q outputs per warp (see head_mean_outputs).  First the means of
// the sources (groups of Cs / 4 threads share the pixels, the groups' sums are added in group order), then every warp takes
// outputs by itself.  (With all outputs of a sample in one block, and dense edges read value by value, 64 channels of 8 x 8 by their
// mean and by all 4096 values to 100 outputs took 4472 us for 16 frames of one sample, fp32, so 174.)
template <typename T, bool BESIDE>
__global__ void __launch_bounds__(kHeadThreads) sr_mean_head_kernel(const __grid_constant__ HeadParams P)
{
    __shared__ __align__(16) float mean[kHeadMaxC];
    __shared__ __align__(16) float part[4 * kHeadThreads];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    sr_begin(P.follow);
    const SrFrame F = sr_frame(P.fr);
    int bx = (int)blockIdx.x, ni = 0;
    if ((bx -= P.in.n_blocks) < 0) {
        sr_input_block<BESIDE>(P.in, P.fr, F, (int)blockIdx.x, reinterpret_cast<int2*>(part));
        sr_end(P.follow);
        return;
    }
    while (ni + 1 < P.n_nodes && bx >= P.first_block[ni + 1]) ++ni;
    const SrHeadNode& nd = P.nodes[ni];
    const int per_block = kHeadWarps * nd.mean_q, co_blocks = (nd.C + per_block - 1) / per_block, bi = bx - P.first_block[ni];
    const int b = bi / co_blocks, o_first = (bi % co_blocks) * per_block, o_end = min(nd.C, o_first + per_block), cur = (int)((F.t + 1) & 1);
    float* const out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    int m_off = 0;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrHeadEdge& e = nd.edges[ei];
        if (e.kind != SR_EDGE_MEAN_DENSE) continue;
        const int vc = e.Cs / 4, groups = kHeadThreads / vc, col = tid % vc, grp = tid / vc;
        if (grp < groups) {
            const T* xs = head_source<T>(P, F, e) + (size_t)b * e.HW * e.Cs + 4 * col;
            float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
            for (int px = grp; px < e.HW; px += groups) {
                float x[4];
                head_load4<BESIDE>(xs + (size_t)px * e.Cs, x);
#pragma unroll
                for (int q = 0; q < 4; ++q) s4[q] += x[q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) part[grp * e.Cs + 4 * col + q] = s4[q];
        }
        __syncthreads();
        const float inv = 1.f / (float)e.HW;
        for (int c = tid; c < e.Cs; c += kHeadThreads) {
            float m = 0.f;
            for (int gq = 0; gq < groups; ++gq) m += part[gq * e.Cs + c];
            mean[m_off + c] = m * inv;
        }
        __syncthreads();
        m_off += e.Cs;
    }
    for (int o = o_first + warp; o < o_end; o += kHeadWarps) {
        float a = 0.f;
        m_off = 0;
        for (int ei = 0; ei < nd.n_edges; ++ei) {
            const SrHeadEdge& e = nd.edges[ei];
            const float* w = e.w + (size_t)o * e.K;
            if (e.kind == SR_EDGE_MEAN_DENSE) {
#pragma unroll 2
                for (int c = 4 * lane; c < e.Cs; c += 128) {
                    const float4 q = __ldg(reinterpret_cast<const float4*>(w + c)), m = *reinterpret_cast<const float4*>(mean + m_off + c);
                    a = fmaf(q.x, m.x, a); a = fmaf(q.y, m.y, a); a = fmaf(q.z, m.z, a); a = fmaf(q.w, m.w, a);
                }
                m_off += e.Cs;
            } else {
                const T* x = head_source<T>(P, F, e) + (size_t)b * e.K;
                if ((e.K & 3) == 0) {
#pragma unroll 4
                    for (int k = 4 * lane; k < e.K; k += 128) {
                        float v[4];
                        head_load4<BESIDE>(x + k, v);
                        const float4 q = __ldg(reinterpret_cast<const float4*>(w + k));
                        a = fmaf(q.x, v[0], a); a = fmaf(q.y, v[1], a); a = fmaf(q.z, v[2], a); a = fmaf(q.w, v[3], a);
                    }
                } else {
#pragma unroll 4
                    for (int k = lane; k < e.K; k += 32) a = fmaf(__ldg(w + k), head_load1<BESIDE>(x + k), a);
                }
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
        if (lane == 0) {
            float z = a + nd.bias[o];
            if (nd.act == 1) z = fmaxf(z, 0.f);
            from_f(static_cast<T*>(nd.state[cur]) + (size_t)b * nd.C + o, z);
            if (out) out[(size_t)b * nd.C + o] = z;
        }
    }
    sr_end(P.follow);
}

// Dense nodes that the two kernels above do not take: a mean-dense edge whose channels are no multiple of four or lie beyond kHeadMaxC
// with those of the node's other ones, or more than SR_HEAD_EDGES edges.  A block takes one sample and one or up to Q = kWideQ outputs
// per warp, whose weight rows are loaded side by side; edge by edge, a mean-dense one in pieces of kHeadMaxC channels: first the means
// of the piece (groups of threads share the pixels, the groups' sums are added in group order), then their products.
// Measured on B200, us per 16 frames, on dense_item (a warp per output and eight samples) -> here: means of 2 x 768 channels of 4 x 4
// to 100 outputs at 8 samples 7820 -> 249; mean of 10 channels of 32 x 32 to 10 outputs at 32 samples 3709 -> 133; eight
// means of 64 channels of 8 x 8 to 10 outputs at 8 samples 4433 -> 233.
constexpr int kWideQ = 8;

struct WideParams {
    SrFrameArgs fr;
    int32_t n_nodes, B, follow;
    int32_t first_block[SR_WIDE_NODES + 1];
    SrWideNode nodes[SR_WIDE_NODES];
    SrHeadEdge edges[SR_WIDE_EDGES];
};
static_assert(sizeof(WideParams) <= 4000, "kernel parameters");

// Adds w[row q * kHeadWarps] . x over n values, spread over the lanes, to acc[q] of the warp's n_q outputs.
template <int Q, typename X>
__device__ __forceinline__ void wide_dot(float (&acc)[Q], const float* w, size_t row, const X* x, int n, int n_q, bool vec, int lane)
{
    if (vec) {
#pragma unroll(Q == 1 ? 8 : 2)
        for (int k = 4 * lane; k < n; k += 128) {
            float xv[4];
            load4(x + k, xv);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q >= n_q) break;
                const float4 wv = __ldg(reinterpret_cast<const float4*>(w + q * kHeadWarps * row + k));
                acc[q] = fmaf(wv.x, xv[0], acc[q]); acc[q] = fmaf(wv.y, xv[1], acc[q]);
                acc[q] = fmaf(wv.z, xv[2], acc[q]); acc[q] = fmaf(wv.w, xv[3], acc[q]);
            }
        }
    } else {
#pragma unroll 4
        for (int k = lane; k < n; k += 32) {
            const float xv = to_f(x[k]);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q >= n_q) break;
                acc[q] = fmaf(__ldg(w + q * kHeadWarps * row + k), xv, acc[q]);
            }
        }
    }
}

template <typename T, int Q>
__global__ void __launch_bounds__(kHeadThreads) sr_wide_head_kernel(const __grid_constant__ WideParams P)
{
    __shared__ __align__(16) float mean[kHeadMaxC];
    __shared__ __align__(16) float part[4 * kHeadThreads];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    sr_begin(P.follow);
    sr_drop_old_lines(P.follow);
    const SrFrame F = sr_frame(P.fr);
    int ni = 0;
    while (ni + 1 < P.n_nodes && (int)blockIdx.x >= P.first_block[ni + 1]) ++ni;
    const SrWideNode& nd = P.nodes[ni];
    const int per_block = kHeadWarps * nd.q, co_blocks = (nd.C + per_block - 1) / per_block, bi = (int)blockIdx.x - P.first_block[ni];
    const int b = bi / co_blocks, o0 = (bi % co_blocks) * per_block + warp, o_end = min(nd.C, (bi % co_blocks + 1) * per_block);
    const int n_q = o0 < o_end ? (o_end - o0 + kHeadWarps - 1) / kHeadWarps : 0;       // outputs o0 + kHeadWarps * q
    const int prev = (int)(F.t & 1), cur = prev ^ 1;
    float* const out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    float acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = 0.f;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrHeadEdge& e = P.edges[nd.first_edge + ei];
        const T* src = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)b * e.HW * e.Cs;
        const float* w = e.w + (size_t)o0 * e.K;
        const bool vec = (e.K & 3) == 0;
        if (e.kind != SR_EDGE_MEAN_DENSE) {
            wide_dot(acc, w, e.K, src, e.K, n_q, vec, lane);
            continue;
        }
        const float inv = 1.f / (float)e.HW;
        for (int c0 = 0; c0 < e.Cs; c0 += kHeadMaxC) {
            const int n = min(kHeadMaxC, e.Cs - c0), cols = vec ? n / 4 : n, groups = max(1, kHeadThreads / cols);
            if (tid < groups * cols) {
                const int grp = tid / cols;
                for (int col = tid % cols; col < cols; col += kHeadThreads) {      // (more than one round: more columns than threads)
                    if (vec) {
                        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                        for (int px = grp; px < e.HW; px += groups) {
                            float x[4];
                            load4(src + c0 + 4 * col + (size_t)px * e.Cs, x);
#pragma unroll
                            for (int q = 0; q < 4; ++q) s4[q] += x[q];
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) part[grp * n + 4 * col + q] = s4[q];
                    } else {
                        float s1 = 0.f;
#pragma unroll 8
                        for (int px = grp; px < e.HW; px += groups) s1 += to_f(src[c0 + col + (size_t)px * e.Cs]);
                        part[grp * n + col] = s1;
                    }
                }
            }
            __syncthreads();
            for (int c = tid; c < n; c += kHeadThreads) {
                float m = 0.f;
                for (int gq = 0; gq < groups; ++gq) m += part[gq * n + c];
                mean[c] = m * inv;
            }
            __syncthreads();
            wide_dot(acc, w + c0, e.K, mean, n, n_q, vec, lane);
        }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        if (q >= n_q) break;
        float a = acc[q];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
        if (lane == 0) {
            const int o = o0 + q * kHeadWarps;
            float z = a + nd.bias[o];
            if (nd.act == 1) z = fmaxf(z, 0.f);
            from_f(static_cast<T*>(nd.state[cur]) + (size_t)b * nd.C + o, z);
            if (out) out[(size_t)b * nd.C + o] = z;
        }
    }
    sr_end(P.follow);
}

struct DirectParams {
    SrFrameArgs fr;
    const SrDevNode* nodes;
    const SrDevEdge* edges;
    const SrDirectItem* items;
    int32_t B, follow;
};

// NON_FINITE: nodes may have a weight that is not finite.  In fp32 a kernel of its own, because the compiler's choices for the tiled
// convolutions change with everything beside them (32 -> 32 channels of 32 x 32, 64 samples: 570 us for eight frames, 626 in the
// kernel that takes both); bf16 is as fast either way.  A launch that a caller recorded before the weight came keeps its kernel, and
// its tiles.
// SLICED: a kernel of its own, too, for launches with such items.
template <typename T, bool NON_FINITE, bool SLICED>
__global__ void __launch_bounds__(kWarps * 32) sr_direct_group_kernel(const __grid_constant__ DirectParams P)
{
    __shared__ __align__(16) int2 tab[SLICED ? kTabSliced : kTab];
    sr_begin(P.follow);
    sr_drop_old_lines(P.follow);
    const SrDirectItem it = P.items[blockIdx.x];
    const SrDevNode& nd = P.nodes[it.node];
    const SrFrame F = sr_frame(P.fr);
    const int prev = (int)(F.t & 1), cur = prev ^ 1;
    float* out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    if (nd.H == 1 && nd.W == 1 && P.edges[nd.first_edge].kind != SR_EDGE_CONV) dense_item<T>(nd, P.edges, it, prev, cur, P.B, out);
    // (As two tests joined by ||, or a mark in the item, this took the compiler from 96 registers to 128, and 3 -> 32 channels of
    // 32 x 32 at 64 samples, fp32, from 171 us for eight frames to 202.)
    else if ((nd.C | nd.untiled | (NON_FINITE && sizeof(T) == 4 ? nd.untiled >> 2 : 0)) % 4 != 0) conv_item<T, NON_FINITE>(nd, P.edges, it, prev, cur, out);
    else if (SLICED && it.b0 >= 0 && (it.pad_ & kItemSlices)) conv_tile<T, 1, true>(nd, P.edges, it, prev, cur, out, tab);
    else if (it.b0 >= 0) conv_tile<T, 1, false>(nd, P.edges, it, prev, cur, out, tab);
    else {
        SrDirectItem four = it;
        four.b0 = ~it.b0;
        if (SLICED && (it.pad_ & kItemSlices)) conv_tile<T, 4, true>(nd, P.edges, four, prev, cur, out, tab);
        else conv_tile<T, 4, false>(nd, P.edges, four, prev, cur, out, tab);
    }
    sr_end(P.follow);
}

}  // namespace

int sr_launch_direct_group(const sr_graph* g, int group, SrFollow how, cudaStream_t s)
{
    const int n = g->group_item_count[group];
    if (n == 0) return 0;
    DirectParams P;
    P.fr = g->frame;
    P.nodes = reinterpret_cast<const SrDevNode*>(g->ws + g->r_nodes.offset);
    P.edges = reinterpret_cast<const SrDevEdge*>(g->ws + g->r_edges.offset);
    P.items = reinterpret_cast<const SrDirectItem*>(g->ws + g->r_items.offset) + g->group_item_offset[group];
    P.B = g->batch;
    P.follow = how.flags();
    bool finite = true;
    for (int v : g->groups[group]) finite = finite && g->nodes[v].w_finite;
    auto kernel = [&](auto sliced) {
        return g->dtype == SR_DTYPE_BF16 ? sr_direct_group_kernel<__nv_bfloat16, true, sliced>
                                         : finite ? sr_direct_group_kernel<float, false, sliced> : sr_direct_group_kernel<float, true, sliced>;
    };
    sr_launch(g->group_sliced[group] ? kernel(std::true_type()) : kernel(std::false_type()), n, kWarps * 32, 0, s, how.early, P);
    return 1;
}

// Dense nodes: with 16 samples or more a block takes 4 x 8 (samples x outputs), with fewer 1 x 2, which spreads a small batch over
// more blocks and keeps four steps of the reduction in flight.
static bool head_wide(const sr_graph* g) { return g->batch >= 16; }

// Outputs per warp of a node with a mean-dense edge (at most `most`): few, because a warp takes them one after the other, as long as
// the blocks number 500 at most, from where on they queue and every one computes the sample's means again; a batch that has a
// block for every SM anyway does not part two outputs.  Measured on B200, us per 16 frames with 1 / 2 / 3 / 8 / 16 outputs per
// warp and with all: 256 channels of 8 x 8 to 1000 outputs at one sample 92 / 104 / 115 / 179 / 280 / 1617, at 32 samples 466 /
// 311 / 258 / 230 / 324 / 1710 (this rule: 9); 32 channels of 16 x 16 to 43 outputs at 8 samples 75 / 85 / 96 / 125 with six, at
// 128 samples 131 / 111 / 113 / 140; 256 channels of 8 x 8 to 10 outputs at 256 samples, fp32, 311 / 300.
static int head_mean_outputs(const sr_graph* g, int channels, int most)
{
    const int all = (channels + kHeadWarps - 1) / kHeadWarps;
    int q = g->batch >= g->sm_count ? std::min(2, all) : 1;
    while (q < all && q < most && (long long)g->batch * ((channels + kHeadWarps * q - 1) / (kHeadWarps * q)) > 500) ++q;
    return q;
}

static int head_blocks(const sr_graph* g, const SrHeadNode& h)
{
    if (h.has_mean) return g->batch * ((h.C + kHeadWarps * h.mean_q - 1) / (kHeadWarps * h.mean_q));
    const int S = head_wide(g) ? 4 : 1, CO = head_wide(g) ? 8 : 2;
    return (g->batch + S - 1) / S * ((h.C + CO - 1) / CO);
}

// The frame input goes with the heads of a group if there is one launch of them (not of the wide kind, whose registers leave
// room for one block beside the tensor-core kernel), and input and heads together are one block per SM at most: a launch less
// counts where a frame takes microseconds, while a large input is better off with small blocks of its own.
bool sr_heads_take_input(const sr_graph* g, int group, const SrFrameArgs& fr, unsigned copies, unsigned stems_R)
{
    const std::vector<SrHeadNode>& heads = g->group_heads[group];
    const std::vector<const SrStem*>& stems = sr_stems(g, stems_R);
    if (heads.empty() || heads.size() > SR_HEAD_NODES || !g->group_wide[group].empty() || stems.size() > kStemsPerLaunch) return false;
    int blocks = 0, mean = 0;
    for (const SrHeadNode& h : heads) {
        blocks += head_blocks(g, h);
        mean += h.has_mean;
    }
    if (mean != 0 && mean != (int)heads.size()) return false;
    if (mean == 0 && head_wide(g)) return false;
    if (g->input_feeds_same_frame) {
        // then the heads read the caller's frame itself, in vectors of four elements
        if (fr.ctl || !stems.empty()) return false;
        for (size_t i = 0; i < g->input_nodes.size(); ++i)
            if (reinterpret_cast<uintptr_t>(fr.v.in_base[i]) & 15 || fr.v.in_stride_bytes[i] & 15) return false;
    }
    size_t next = 0;
    return blocks + sr_plan_input(g, copies, stems, next, true).n_blocks <= g->sm_count;
}

int sr_launch_heads(const sr_graph* g, int group, bool with_input, unsigned copies, unsigned stems_R, SrFollow how, cudaStream_t s)
{
    int launches = 0;
    for (int cls = 0; cls < 2; ++cls) {                                      // 0: nodes with a mean-dense edge, 1: without
        const bool wide = head_wide(g);
        HeadParams P;
        P.fr = g->frame;
        P.B = g->batch;
        P.direct = with_input && g->input_feeds_same_frame ? 1 : 0;
        P.in.n_blocks = 0;
        P.n_nodes = 0;
        int blocks = 0;
        auto flush = [&]() {
            if (P.n_nodes == 0) return;
            if (with_input) {
                size_t next = 0;
                P.in = sr_plan_input(g, copies, sr_stems(g, stems_R), next, true);
            }
            P.follow = how.flags();
            auto kernel = [&](auto beside) {
                const bool bf = g->dtype == SR_DTYPE_BF16;
                if (cls == 0) return bf ? sr_mean_head_kernel<__nv_bfloat16, beside> : sr_mean_head_kernel<float, beside>;
                if (wide) return bf ? sr_head_kernel<__nv_bfloat16, 4, 8, false, beside> : sr_head_kernel<float, 4, 8, false, beside>;
                return bf ? sr_head_kernel<__nv_bfloat16, 1, 2, true, beside> : sr_head_kernel<float, 1, 2, true, beside>;
            };
            sr_launch(how.beside ? kernel(std::true_type()) : kernel(std::false_type()), P.in.n_blocks + blocks, kHeadThreads, 0, s, how.early, P);
            ++launches;
            how.early = true;
            P.n_nodes = 0;
            blocks = 0;
        };
        for (const SrHeadNode& h : g->group_heads[group]) {
            if ((h.has_mean ? 0 : 1) != cls) continue;
            P.nodes[P.n_nodes] = h;
            P.first_block[P.n_nodes++] = blocks;
            blocks += head_blocks(g, h);
            P.first_block[P.n_nodes] = blocks;
            if (P.n_nodes == SR_HEAD_NODES) flush();
        }
        flush();
    }
    for (int few = 0; few < 2; ++few) {                                      // 1: nodes of one output per warp
        WideParams P;
        P.fr = g->frame;
        P.B = g->batch;
        P.n_nodes = 0;
        int blocks = 0, n_edges = 0;
        auto flush = [&]() {
            if (P.n_nodes == 0) return;
            P.follow = how.flags();
            auto kernel = [&](auto q) { return g->dtype == SR_DTYPE_BF16 ? sr_wide_head_kernel<__nv_bfloat16, q> : sr_wide_head_kernel<float, q>; };
            sr_launch(few ? kernel(std::integral_constant<int, 1>()) : kernel(std::integral_constant<int, kWideQ>()), blocks, kHeadThreads, 0, s, how.early, P);
            ++launches;
            how.early = true;
            P.n_nodes = blocks = n_edges = 0;
        };
        for (const SrWideNode& h : g->group_wide[group]) {
            if ((h.q == 1) != (few == 1)) continue;
            if (P.n_nodes == SR_WIDE_NODES || n_edges + h.n_edges > SR_WIDE_EDGES) flush();
            std::copy_n(g->group_wide_edges[group].begin() + h.first_edge, h.n_edges, P.edges + n_edges);
            P.nodes[P.n_nodes] = h;
            P.nodes[P.n_nodes].first_edge = n_edges;
            P.first_block[P.n_nodes++] = blocks;
            n_edges += h.n_edges;
            blocks += g->batch * ((h.C + kHeadWarps * h.q - 1) / (kHeadWarps * h.q));
            P.first_block[P.n_nodes] = blocks;
        }
        flush();
    }
    return launches;
}

// Does a convolutional node run on conv_item?  conv_tile takes channels in vectors of four and counts the elements of a source
// sample in 32 bits (from the corner of a window that leaves the image, hence the margin).
bool sr_direct_untiled(const sr_graph* g, int v)
{
    bool tile = g->nodes[v].d.c % 4 == 0 && g->nodes[v].d.c < 1 << 24;
    for (int e : g->nodes[v].in_edges) {
        const SrHostEdge& he = g->edges[e];
        const sr_node_desc& s = g->nodes[he.d.src].d;
        tile = tile && (double)(s.h + 2 * he.k_eff) * (s.w + 2 * he.k_eff) * s.c < 2147483648.0;
    }
    return !tile;
}

// The work items of a convolutional node on the CUDA cores.
void sr_direct_conv_items(const sr_graph* g, int v, std::vector<SrDirectItem>& items)
{
    const sr_node_desc& d = g->nodes[v].d;
    const int HW = d.h * d.w;
    if (sr_direct_untiled(g, v)) {
        for (int b = 0; b < g->batch; ++b)
            for (int p0 = 0; p0 < HW; p0 += kWarps * kPix) items.push_back(SrDirectItem{v, b, p0, 0});
        return;
    }
    int qlog = 0;
    while (qlog < 5 && (4 << qlog) < d.c) ++qlog;
    // Four pixels per thread once that still gives every SM 256 threads; marked by the complement of the sample.  Measured on
    // B200, fp32, us per frame with one / four pixels everywhere: small CNN (28 x 28 x 32, 14 x 14 x 32, 7 x 7 x 64) at 128
    // samples 161 / 133 (this rule: 114), at 32 samples (sequential) 90 / 144, at one 27 / 51; MNIST net at 256 samples 35 / 53.
    // Slices of a reduction of 128 values or more (32 steps where the source's channels come in fours) until there are 512 threads per SM without them (256: sequential at 128 samples 146
    // instead of 117 us a frame); with four pixels per thread where a pixel per thread would make 64 threads per SM (256: 29.8 instead
    // of 24.0 us at 16 samples, 49.2 instead of 39.9 at 48; never: 27.0 and 62.1).
    const size_t quads = (size_t)g->batch * HW * (d.c / 4), sms = (size_t)g->sm_count;
    int K = 0;
    for (int e : g->nodes[v].in_edges) K += g->edges[e].K;
    const bool slices = K >= 128 && quads / 4 < sms * 512 && g->compact == 0, four = quads / 4 >= sms * 256 || (slices && quads >= sms * 64);
    const int px = ((slices ? 32 : kWarps * 32) >> qlog) * (four ? 4 : 1);
    for (int b = 0; b < g->batch; ++b)
        for (int p0 = 0; p0 < HW; p0 += px)
            for (int c0 = 0; c0 < d.c; c0 += 4 << qlog) items.push_back(SrDirectItem{v, four ? ~b : b, p0, c0 | qlog << 24 | (slices ? kItemSlices : 0)});
}
bool sr_direct_sliced(const SrDirectItem& it) { return (it.pad_ & kItemSlices) != 0; }
int sr_direct_dense_outputs_per_block() { return kWarps; }
int sr_direct_dense_samples_per_block() { return kDenseB; }

// Which head kernel takes the node: 1: sr_head_kernel or sr_mean_head_kernel, 2: sr_wide_head_kernel, 0: none.
int sr_head_class(const sr_graph* g, int v)
{
    const SrHostNode& n = g->nodes[v];
    if (n.in_edges.size() > SR_WIDE_EDGES) return 0;
    int channels = 0;
    for (int e : n.in_edges) {
        const SrHostEdge& he = g->edges[e];
        if (he.d.kind != SR_EDGE_MEAN_DENSE) continue;
        const int cs = g->nodes[he.d.src].d.c;
        if (cs % 4 != 0 || cs > kHeadMaxC) return 2;
        channels += cs;
    }
    return n.in_edges.size() > SR_HEAD_EDGES || channels > kHeadMaxC ? 2 : 1;
}

// Fills g's lists of the group's head nodes for the workspace that is being bound.
void sr_describe_heads(sr_graph* g, int group)
{
    char* const ws = g->ws;
    for (int v : g->group_head_nodes[group]) {
        const SrHostNode& n = g->nodes[v];
        std::vector<SrHeadEdge> edges;
        bool has_mean = false;
        for (int e : n.in_edges) {
            const SrHostEdge& he = g->edges[e];
            const SrHostNode& s = g->nodes[he.d.src];
            SrHeadEdge x{};
            x.src[0] = ws + s.state[0].offset;
            x.src[1] = ws + s.state[1].offset;
            x.w = reinterpret_cast<const float*>(ws + he.w_direct.offset);
            x.HW = s.d.h * s.d.w; x.Cs = s.d.c; x.kind = he.d.kind; x.R = he.R; x.K = he.K;
            x.slot = s.input_slot;
            has_mean |= he.d.kind == SR_EDGE_MEAN_DENSE;
            edges.push_back(x);
        }
        auto describe = [&](auto& h) {
            h.state[0] = ws + n.state[0].offset;
            h.state[1] = ws + n.state[1].offset;
            h.bias = reinterpret_cast<const float*>(ws + n.bias.offset);
            h.C = n.d.c; h.act = n.d.act;
            h.is_output = v == g->info.output_node;
            h.n_edges = (int)edges.size();
        };
        if (sr_head_class(g, v) == 1) {
            SrHeadNode h{};
            describe(h);
            h.has_mean = has_mean;
            if (has_mean) h.mean_q = head_mean_outputs(g, h.C, h.C);
            std::copy(edges.begin(), edges.end(), h.edges);
            g->group_heads[group].push_back(h);
        } else {
            SrWideNode h{};
            describe(h);
            h.q = head_mean_outputs(g, h.C, kWideQ);
            h.first_edge = (int)g->group_wide_edges[group].size();
            g->group_wide_edges[group].insert(g->group_wide_edges[group].end(), edges.begin(), edges.end());
            g->group_wide[group].push_back(h);
        }
    }
}

bool sr_direct_share_sm()
{
    auto ask = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess; };
    auto heads = [&](auto beside) {
        return ask(sr_head_kernel<__nv_bfloat16, 4, 8, false, beside>) && ask(sr_head_kernel<__nv_bfloat16, 1, 2, true, beside>) &&
               ask(sr_mean_head_kernel<__nv_bfloat16, beside>);
    };
    return heads(std::false_type()) && heads(std::true_type()) && ask(sr_wide_head_kernel<__nv_bfloat16, 1>) &&
           ask(sr_wide_head_kernel<__nv_bfloat16, kWideQ>) && ask(sr_direct_group_kernel<__nv_bfloat16, true, false>) && ask(sr_direct_group_kernel<__nv_bfloat16, true, true>);
}
