// Frame input: the input nodes' state takes the caller's frame, and few-channel input edges are staged, in one launch.
//
// A staged edge (C_in * k * k <= 128, C_in not a multiple of 16) feeds the tensor-core kernel im2col rows: row (b, oy, ox)
// holds the k * k * C_in receptive field of that output pixel (zero outside the image, zero padded to Kp), so that the edge
// becomes an ordinary K-block.
//
// Bound by the latency of its loads and, for large batches, by the bytes staged.  A thread makes one 16-byte chunk (eight
// values) at a time: neighbouring threads write neighbouring chunks, and a single sample still fills many blocks.  Chunks
// that hold padding only are never written (the staging buffers are zeroed when a workspace is bound).
// Measured on B200, us, input copy + staging before (two launches, a thread per pixel) -> now: one 32 x 32 x 3 sample through a
// 5 x 5 filter 1.6 + 8.4 -> 2.6; 37 samples of 28 x 28 x 3 through 3 x 3 2.1 + 5.7 -> 4.4; 128 samples through 5 x 5 beside the
// tensor-core kernel 2.9 + 54 -> 40.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "sr_internal.h"
#include "sr_kernels.h"

namespace {

constexpr int kThreads = 256;
constexpr int kStemsPerLaunch = 8;

struct CopyPart { void* dst[2]; size_t bytes; int32_t slot, first_block; };
struct StemPart { void* dst[2]; int32_t slot, first_block, Hs, Ws, Cs, Ho, Wo, k, stride, pad, Kp, K; };

struct InputParams {
    SrFrameArgs fr;                 // the frame: fr.in(slot) of this update; it goes to the buffers of parity (t + 1) & 1
    int32_t n_copy, n_stem, n_blocks, B;
    CopyPart copy[SR_MAX_INPUTS];
    StemPart stem[kStemsPerLaunch];
};
static_assert(sizeof(InputParams) <= 4000, "kernel parameters");

// (Registers for six blocks per SM: three of them fit beside a CTA of the tensor-core kernel.)
__global__ void __launch_bounds__(kThreads, 6) sr_input_kernel(const __grid_constant__ InputParams P)
{
    __shared__ int2 tap[128];       // per element of a window: offset from the (unpadded) window origin; dy << 16 | dx
    const SrFrame F = sr_frame(P.fr);
    const int cur = (int)((F.t + 1) & 1), bx = (int)blockIdx.x;
    const int first_stem = P.n_stem ? P.stem[0].first_block : P.n_blocks;
    if (bx < first_stem) {
        int i = 0;
        while (i + 1 < P.n_copy && bx >= P.copy[i + 1].first_block) ++i;
        const CopyPart& c = P.copy[i];
        const int blocks = (i + 1 < P.n_copy ? P.copy[i + 1].first_block : first_stem) - c.first_block;
        const char* src = sr_frame_input(P.fr, F, c.slot);
        char* dst = static_cast<char*>(c.dst[cur]);
        const size_t tid = (size_t)(bx - c.first_block) * kThreads + threadIdx.x, nth = (size_t)blocks * kThreads;
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            const size_t nv = c.bytes / 16;
            for (size_t j = tid; j < nv; j += nth) reinterpret_cast<uint4*>(dst)[j] = reinterpret_cast<const uint4*>(src)[j];
            for (size_t j = nv * 16 + tid; j < c.bytes; j += nth) dst[j] = src[j];
        } else {
            for (size_t j = tid; j < c.bytes; j += nth) dst[j] = src[j];
        }
        return;
    }
    int i = 0;
    while (i + 1 < P.n_stem && bx >= P.stem[i + 1].first_block) ++i;
    const StemPart& st = P.stem[i];
    const unsigned blocks = (unsigned)((i + 1 < P.n_stem ? P.stem[i + 1].first_block : P.n_blocks) - st.first_block);
    const int Hs = st.Hs, Ws = st.Ws, Cs = st.Cs, k = st.k, K = st.K;
    for (int kk = threadIdx.x; kk < 128; kk += kThreads) {
        int2 q = make_int2(0, 0);
        if (kk < K) {
            const int ci = kk % Cs, tp = kk / Cs, dx = tp % k, dy = tp / k;
            q = make_int2((dy * Ws + dx) * Cs + ci, dy << 16 | dx);
        }
        tap[kk] = q;
    }
    __syncthreads();
    const unsigned short* src = reinterpret_cast<const unsigned short*>(sr_frame_input(P.fr, F, st.slot));
    uint4* dst = static_cast<uint4*>(st.dst[cur]);
    const unsigned used = (unsigned)(K + 7) / 8, all = (unsigned)st.Kp / 8, Wo = (unsigned)st.Wo, Ho = (unsigned)st.Ho;
    const unsigned n = (unsigned)P.B * Ho * Wo * used;
    for (unsigned j = ((unsigned)bx - (unsigned)st.first_block) * kThreads + threadIdx.x; j < n; j += blocks * kThreads) {
        const unsigned p = j / used, c = j - p * used, r = p / Wo, ox = p - r * Wo, b = r / Ho, oy = r - b * Ho;
        const int y0 = (int)oy * st.stride - st.pad, x0 = (int)ox * st.stride - st.pad;
        const unsigned short* base = src + (((long long)b * Hs + y0) * Ws + x0) * Cs;
        const int k0 = (int)c * 8;
        uint32_t v[4];
        if (y0 >= 0 && x0 >= 0 && y0 + k <= Hs && x0 + k <= Ws) {              // the whole window lies in the image
            unsigned short e[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) e[q] = base[tap[k0 + q].x];             // (elements beyond K read the window's first)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = (k0 + 2 * q < K ? (uint32_t)e[2 * q] : 0u) | (k0 + 2 * q + 1 < K ? (uint32_t)e[2 * q + 1] << 16 : 0u);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = 0u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int2 t = tap[k0 + 2 * q + h];
                    const int y = y0 + (t.y >> 16), x = x0 + (t.y & 0xFFFF);
                    if (k0 + 2 * q + h < K && y >= 0 && y < Hs && x >= 0 && x < Ws) v[q] |= (uint32_t)base[t.x] << (16 * h);
                }
            }
        }
        dst[(size_t)p * all + c] = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

__global__ void sr_set_ctl_kernel(SrFrameCtl* ctl, SrFrameCtl v) { *ctl = v; }

__global__ void sr_advance_kernel(SrFrameCtl* ctl, int n)
{
    ctl->t += n;
    ctl->run_t += n;
}

}  // namespace

// Queues the input of the frame that `fr` describes.  copies: bit i = input node i's state takes it; stems_R: which staged edges
// (bit 0: those that read it within the frame, R = 0; bit 1: those that read it a frame later, R = 1); beside: it runs on a
// stream of its own beside the frame's other launches.  Returns launches.
int sr_launch_input(const sr_graph* g, const SrFrameArgs& fr, unsigned copies, unsigned stems_R, bool beside, cudaStream_t s)
{
    // Beside a tensor-core kernel: few blocks (every SM has threads left for that kernel's CTA at once; with a grid that fills
    // the SMs it started up to 15 us late), else as many as there is work.
    const size_t per_part = beside ? 148 * 2 : 148 * 16;
    int launches = 0;
    std::vector<const SrStem*> stems;
    for (const SrStem& st : g->stems)
        if ((stems_R >> st.R) & 1u) stems.push_back(&st);
    size_t next = 0;
    do {
        InputParams P;
        P.fr = fr;
        P.B = g->batch;
        P.n_copy = P.n_stem = 0;
        int blocks = 0;
        if (launches == 0)
            for (size_t i = 0; i < g->input_nodes.size(); ++i) {
                if (!((copies >> i) & 1u)) continue;
                const SrHostNode& n = g->nodes[g->input_nodes[i]];
                CopyPart& c = P.copy[P.n_copy++];
                c.dst[0] = g->ws + n.state[0].offset;
                c.dst[1] = g->ws + n.state[1].offset;
                c.bytes = (size_t)g->batch * n.d.h * n.d.w * n.d.c * g->elem;
                c.slot = (int)i;
                c.first_block = blocks;
                blocks += (int)std::min<size_t>(beside ? 148 : 296, (c.bytes / 16 + kThreads - 1) / kThreads + 1);
            }
        for (; next < stems.size() && P.n_stem < kStemsPerLaunch; ++next) {
            const SrStem& st = *stems[next];
            StemPart& d = P.stem[P.n_stem++];
            d.dst[0] = st.dst[0]; d.dst[1] = st.dst[1];
            d.slot = st.slot;
            d.Hs = st.Hs; d.Ws = st.Ws; d.Cs = st.Cs; d.Ho = st.Ho; d.Wo = st.Wo;
            d.k = st.k; d.stride = st.stride; d.pad = st.pad; d.Kp = st.Kp; d.K = st.K;
            d.first_block = blocks;
            const size_t chunks = (size_t)g->batch * st.Ho * st.Wo * ((st.K + 7) / 8);
            blocks += (int)std::min<size_t>(per_part, (chunks + kThreads - 1) / kThreads);
        }
        P.n_blocks = blocks;
        if (blocks == 0) break;
        sr_input_kernel<<<blocks, kThreads, 0, s>>>(P);
        ++launches;
    } while (next < stems.size());
    return launches;
}

void sr_launch_set_ctl(const sr_graph* g, const SrFrameCtl& v, cudaStream_t s)
{
    sr_set_ctl_kernel<<<1, 1, 0, s>>>(reinterpret_cast<SrFrameCtl*>(g->ws + g->r_ctl.offset), v);
}

void sr_launch_advance(const sr_graph* g, int n, cudaStream_t s)
{
    sr_advance_kernel<<<1, 1, 0, s>>>(reinterpret_cast<SrFrameCtl*>(g->ws + g->r_ctl.offset), n);
}

// The kernels that run beside the tensor-core kernel ask for the partition of the SM that it needs (all of it shared memory): an
// SM changes its partition only when it is empty, so with another one the tensor-core kernel waits for them to drain.
bool sr_input_share_sm()
{
    return cudaFuncSetAttribute(sr_input_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess;
}
