// CUDA-core kernels of the frame update: the node update
//     x_v = sigma(b_v + sum_e f_e(theta_e, x_src(e)))          (paper Sec. A1.2)
// for every node of one launch group, in one launch.  They serve the fp32 mode, the dense heads and
// the few-channel nodes that are bound by memory traffic, and they are the reference engine the
// tensor-core kernel can be switched against.  Accumulation is fp32 in every mode.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "sr_internal.h"
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

constexpr int kPix = 4;            // pixels per warp (conv nodes)
constexpr int kWarps = 4;          // warps per block
constexpr int kDenseB = 8;         // samples per warp (dense nodes)

// Conv node: a block covers kWarps*kPix consecutive pixels of one sample; lanes run over output
// channels, so weight reads ([K][C_out] rows) and state writes (NHWC) are coalesced and the input
// reads are warp-uniform broadcasts.
template <typename T>
__device__ void conv_item(const SrDevNode& nd, const SrDevEdge* edges, const SrDirectItem& it, int prev, int cur,
                          float* out_f32)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int HW = nd.H * nd.W;
    const int pbase = it.p0 + warp * kPix;
    int oy[kPix], ox[kPix];
    bool pv[kPix];
#pragma unroll
    for (int j = 0; j < kPix; ++j) {
        const int p = pbase + j;
        pv[j] = p < HW;
        oy[j] = pv[j] ? p / nd.W : 0;
        ox[j] = pv[j] ? p % nd.W : 0;
    }
    T* dst = static_cast<T*>(nd.state[cur]) + (size_t)it.b0 * HW * nd.C;
    for (int co0 = 0; co0 < nd.C; co0 += 32) {
        const int co = co0 + lane;
        const bool cv = co < nd.C;
        float acc[kPix];
#pragma unroll
        for (int j = 0; j < kPix; ++j) acc[j] = 0.f;
        for (int ei = 0; ei < nd.n_edges; ++ei) {
            const SrDevEdge& e = edges[nd.first_edge + ei];
            const T* src = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)it.b0 * e.Hs * e.Ws * e.Cs;
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
            const float b = nd.bias[co];
#pragma unroll
            for (int j = 0; j < kPix; ++j) {
                if (!pv[j]) continue;
                float z = acc[j] + b;
                if (nd.act == 1) z = fmaxf(z, 0.f);
                from_f(dst + (size_t)(pbase + j) * nd.C + co, z);
                if (out_f32) out_f32[((size_t)it.b0 * HW + pbase + j) * nd.C + co] = z;
            }
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
    int32_t n_nodes, B;
    int32_t first_block[SR_HEAD_NODES + 1];
    SrHeadNode nodes[SR_HEAD_NODES];
};
static_assert(sizeof(HeadParams) <= 4000, "kernel parameters");

// Nodes with dense edges only: a block takes CO outputs of S samples; its threads stride over the reduction index in vectors
// of four, every thread keeps S x CO partial sums (a weight vector serves S samples).  The sums of a warp meet by halving,
// those of the warps in shared memory in a fixed order.
template <typename T, int S, int CO>
__global__ void __launch_bounds__(kHeadThreads) sr_head_kernel(const __grid_constant__ HeadParams P)
{
    __shared__ float red[kHeadWarps][32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const SrFrame F = sr_frame(P.fr);
    int ni = 0;
    while (ni + 1 < P.n_nodes && (int)blockIdx.x >= P.first_block[ni + 1]) ++ni;
    const SrHeadNode& nd = P.nodes[ni];
    const int co_blocks = (nd.C + CO - 1) / CO, bi = (int)blockIdx.x - P.first_block[ni], b0 = (bi / co_blocks) * S, co0 = (bi % co_blocks) * CO;
    const int nco = min(CO, nd.C - co0), prev = (int)(F.t & 1), cur = prev ^ 1;
    float* const out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    float acc[S][CO];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int o = 0; o < CO; ++o) acc[s][o] = 0.f;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrHeadEdge& e = nd.edges[ei];
        const int K = e.K;
        const T* x[S];
        const float* w[CO];
#pragma unroll
        for (int s = 0; s < S; ++s) x[s] = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)min(b0 + s, P.B - 1) * K;   // samples and rows beyond
#pragma unroll
        for (int o = 0; o < CO; ++o) w[o] = e.w + (size_t)(co0 + min(o, nco - 1)) * K;                                          // the last repeat it
        if ((K & 3) == 0) {
#pragma unroll(S == 1 ? 4 : 1)
            for (int k = 4 * tid; k < K; k += 4 * kHeadThreads) {
                float4 wv[CO];
                float xv[S][4];
#pragma unroll
                for (int s = 0; s < S; ++s) load4(x[s] + k, xv[s]);
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
                    for (int s = 0; s < S; ++s) acc[s][o] = fmaf(wk, to_f(x[s][k]), acc[s][o]);
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
}

// Nodes with a mean-dense edge: a block takes one sample.  First the means of the sources (groups of Cs / 4 threads share the
// pixels, the groups' sums are added in group order), then every warp takes outputs by itself.
template <typename T>
__global__ void __launch_bounds__(kHeadThreads) sr_mean_head_kernel(const __grid_constant__ HeadParams P)
{
    __shared__ __align__(16) float mean[kHeadMaxC];
    __shared__ float part[4 * kHeadThreads];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const SrFrame F = sr_frame(P.fr);
    int ni = 0;
    while (ni + 1 < P.n_nodes && (int)blockIdx.x >= P.first_block[ni + 1]) ++ni;
    const SrHeadNode& nd = P.nodes[ni];
    const int b = (int)blockIdx.x - P.first_block[ni], prev = (int)(F.t & 1), cur = prev ^ 1;
    float* const out = nd.is_output ? sr_frame_output(P.fr, F) : nullptr;
    int m_off = 0;
    for (int ei = 0; ei < nd.n_edges; ++ei) {
        const SrHeadEdge& e = nd.edges[ei];
        if (e.kind != SR_EDGE_MEAN_DENSE) continue;
        const int vc = e.Cs / 4, groups = kHeadThreads / vc, col = tid % vc, grp = tid / vc;
        if (grp < groups) {
            const T* xs = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)b * e.HW * e.Cs + 4 * col;
            float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
            for (int px = grp; px < e.HW; px += groups) {
                float x[4];
                load4(xs + (size_t)px * e.Cs, x);
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
    for (int o = warp; o < nd.C; o += kHeadWarps) {
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
                const T* x = static_cast<const T*>(e.src[e.R ? prev : cur]) + (size_t)b * e.K;
#pragma unroll 4
                for (int k = lane; k < e.K; k += 32) a = fmaf(__ldg(w + k), to_f(x[k]), a);
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
}

template <typename T>
__global__ void __launch_bounds__(kWarps * 32)
sr_direct_group_kernel(const SrDevNode* __restrict__ nodes, const SrDevEdge* __restrict__ edges,
                       const SrDirectItem* __restrict__ items, const __grid_constant__ SrFrameArgs fr, int B)
{
    const SrDirectItem it = items[blockIdx.x];
    const SrDevNode& nd = nodes[it.node];
    const SrFrame F = sr_frame(fr);
    const int prev = (int)(F.t & 1), cur = prev ^ 1;
    float* out = nd.is_output ? sr_frame_output(fr, F) : nullptr;
    if (nd.H == 1 && nd.W == 1 && edges[nd.first_edge].kind != SR_EDGE_CONV) dense_item<T>(nd, edges, it, prev, cur, B, out);
    else conv_item<T>(nd, edges, it, prev, cur, out);
}

}  // namespace

int sr_launch_direct_group(const sr_graph* g, int group, cudaStream_t s)
{
    const int n = g->group_item_count[group];
    if (n == 0) return 0;
    const SrDevNode* nodes = reinterpret_cast<const SrDevNode*>(g->ws + g->r_nodes.offset);
    const SrDevEdge* edges = reinterpret_cast<const SrDevEdge*>(g->ws + g->r_edges.offset);
    const SrDirectItem* items = reinterpret_cast<const SrDirectItem*>(g->ws + g->r_items.offset) + g->group_item_offset[group];
    if (g->dtype == SR_DTYPE_BF16)
        sr_direct_group_kernel<__nv_bfloat16><<<n, kWarps * 32, 0, s>>>(nodes, edges, items, g->frame, g->batch);
    else
        sr_direct_group_kernel<float><<<n, kWarps * 32, 0, s>>>(nodes, edges, items, g->frame, g->batch);
    return 1;
}

int sr_launch_heads(const sr_graph* g, int group, cudaStream_t s)
{
    int launches = 0;
    for (int cls = 0; cls < 2; ++cls) {                                      // 0: nodes with a mean-dense edge, 1: without
        // Dense nodes: with 16 samples or more a block takes 4 x 8 (samples x outputs), with fewer 1 x 2, which spreads a small
        // batch over more blocks and keeps four steps of the reduction in flight.
        const bool wide = g->batch >= 16;
        const int S = cls == 0 ? 1 : (wide ? 4 : 1), CO = cls == 0 ? 1 << 30 : (wide ? 8 : 2);
        HeadParams P;
        P.B = g->batch;
        P.fr = g->frame;
        P.n_nodes = 0;
        int blocks = 0;
        auto flush = [&]() {
            if (P.n_nodes == 0) return;
            const bool bf = g->dtype == SR_DTYPE_BF16;
            if (cls == 0) {
                if (bf) sr_mean_head_kernel<__nv_bfloat16><<<blocks, kHeadThreads, 0, s>>>(P);
                else sr_mean_head_kernel<float><<<blocks, kHeadThreads, 0, s>>>(P);
            } else if (wide) {
                if (bf) sr_head_kernel<__nv_bfloat16, 4, 8><<<blocks, kHeadThreads, 0, s>>>(P);
                else sr_head_kernel<float, 4, 8><<<blocks, kHeadThreads, 0, s>>>(P);
            } else {
                if (bf) sr_head_kernel<__nv_bfloat16, 1, 2><<<blocks, kHeadThreads, 0, s>>>(P);
                else sr_head_kernel<float, 1, 2><<<blocks, kHeadThreads, 0, s>>>(P);
            }
            ++launches;
            P.n_nodes = 0;
            blocks = 0;
        };
        for (const SrHeadNode& h : g->group_heads[group]) {
            if ((h.has_mean ? 0 : 1) != cls) continue;
            P.nodes[P.n_nodes] = h;
            P.first_block[P.n_nodes++] = blocks;
            blocks += (g->batch + S - 1) / S * (cls == 0 ? 1 : (h.C + CO - 1) / CO);
            P.first_block[P.n_nodes] = blocks;
            if (P.n_nodes == SR_HEAD_NODES) flush();
        }
        flush();
    }
    return launches;
}

int sr_direct_conv_pixels_per_block() { return kWarps * kPix; }
int sr_direct_dense_outputs_per_block() { return kWarps; }
int sr_direct_dense_samples_per_block() { return kDenseB; }

// Can the head kernels take the node?
bool sr_head_takes(const sr_graph* g, int v)
{
    const SrHostNode& n = g->nodes[v];
    if (n.in_edges.size() > SR_HEAD_EDGES) return false;
    int channels = 0;
    for (int e : n.in_edges) {
        const SrHostEdge& he = g->edges[e];
        if (he.d.kind != SR_EDGE_MEAN_DENSE) continue;
        const int cs = g->nodes[he.d.src].d.c;
        if (cs % 4 != 0) return false;
        channels += cs;
    }
    return channels <= kHeadMaxC;
}

bool sr_direct_share_sm()
{
    auto ask = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess; };
    return ask(sr_head_kernel<__nv_bfloat16, 4, 8>) && ask(sr_head_kernel<__nv_bfloat16, 1, 2>) && ask(sr_mean_head_kernel<__nv_bfloat16>) &&
           ask(sr_direct_group_kernel<__nv_bfloat16>);
}
