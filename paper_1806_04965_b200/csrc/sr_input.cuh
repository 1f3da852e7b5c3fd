// Frame input: the input nodes' state takes the caller's frame, and few-channel input edges are staged, in one launch (of its
// own, or together with the dense heads of a small frame).
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
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "sr_internal.h"

constexpr int kInputThreads = 256;
constexpr int kStemsPerLaunch = 8;

struct SrCopyPart { void* dst[2]; size_t bytes; int32_t slot, first_block; };
struct SrStemPart { void* dst[2]; int32_t slot, first_block, Hs, Ws, Cs, Ho, Wo, k, stride, pad, Kp, K; };

// The frame goes to the buffers of parity (t + 1) & 1.
struct SrInputPart {
    int32_t n_copy, n_stem, n_blocks, B;
    SrCopyPart copy[SR_MAX_INPUTS];
    SrStemPart stem[kStemsPerLaunch];
};

// Block bx of the input's n_blocks.  tap: 128 words of shared memory; per element of a window: offset from the (unpadded) window
// origin; dy << 16 | dx.  BESIDE: for a launch that does not wait for the one before it (see SrFollow).
template <bool BESIDE>
__device__ __forceinline__ void sr_input_block(const SrInputPart& P, const SrFrameArgs& fr, const SrFrame& F, int bx, int2* tap)
{
    const int cur = (int)((F.t + 1) & 1);
    const int first_stem = P.n_stem ? P.stem[0].first_block : P.n_blocks;
    if (bx < first_stem) {
        int i = 0;
        while (i + 1 < P.n_copy && bx >= P.copy[i + 1].first_block) ++i;
        const SrCopyPart& c = P.copy[i];
        const int blocks = (i + 1 < P.n_copy ? P.copy[i + 1].first_block : first_stem) - c.first_block;
        const char* src = sr_frame_input(fr, F, c.slot);
        char* dst = static_cast<char*>(c.dst[cur]);
        const size_t tid = (size_t)(bx - c.first_block) * kInputThreads + threadIdx.x, nth = (size_t)blocks * kInputThreads;
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            const size_t nv = c.bytes / 16;
            const uint4* v = reinterpret_cast<const uint4*>(src);
            for (size_t j = tid; j < nv; j += nth) reinterpret_cast<uint4*>(dst)[j] = BESIDE ? sr_load_past_l1(v + j) : v[j];
            if (BESIDE && nv * 16 < c.bytes) __threadfence();
            for (size_t j = nv * 16 + tid; j < c.bytes; j += nth) dst[j] = src[j];
        } else {
            if (BESIDE) __threadfence();
            for (size_t j = tid; j < c.bytes; j += nth) dst[j] = src[j];
        }
        return;
    }
    if (BESIDE) __threadfence();
    int i = 0;
    while (i + 1 < P.n_stem && bx >= P.stem[i + 1].first_block) ++i;
    const SrStemPart& st = P.stem[i];
    const unsigned blocks = (unsigned)((i + 1 < P.n_stem ? P.stem[i + 1].first_block : P.n_blocks) - st.first_block);
    const int Hs = st.Hs, Ws = st.Ws, Cs = st.Cs, k = st.k, K = st.K;
    for (int kk = threadIdx.x; kk < 128; kk += kInputThreads) {
        int2 q = make_int2(0, 0);
        if (kk < K) {
            const int ci = kk % Cs, tp = kk / Cs, dx = tp % k, dy = tp / k;
            q = make_int2((dy * Ws + dx) * Cs + ci, dy << 16 | dx);
        }
        tap[kk] = q;
    }
    __syncthreads();
    const unsigned short* src = reinterpret_cast<const unsigned short*>(sr_frame_input(fr, F, st.slot));
    uint4* dst = static_cast<uint4*>(st.dst[cur]);
    const unsigned used = (unsigned)(K + 7) / 8, all = (unsigned)st.Kp / 8, Wo = (unsigned)st.Wo, Ho = (unsigned)st.Ho;
    const unsigned n = (unsigned)P.B * Ho * Wo * used;
    for (unsigned j = ((unsigned)bx - (unsigned)st.first_block) * kInputThreads + threadIdx.x; j < n; j += blocks * kInputThreads) {
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

// Host: the blocks that copy the inputs named in `copies` and stage `stems` [next, ...), as many as fit; advances next.
inline SrInputPart sr_plan_input(const sr_graph* g, unsigned copies, const std::vector<const SrStem*>& stems, size_t& next, bool beside)
{
    // Beside a tensor-core kernel: few blocks (every SM has threads and registers left for all of them), else as many as there
    // is work for.
    const size_t sms = (size_t)g->sm_count, per_part = beside ? sms * 2 : sms * 16;
    SrInputPart P;
    P.B = g->batch;
    P.n_copy = P.n_stem = 0;
    int blocks = 0;
    for (size_t i = 0; i < g->input_nodes.size(); ++i) {
        if (!((copies >> i) & 1u)) continue;
        const SrHostNode& n = g->nodes[g->input_nodes[i]];
        SrCopyPart& c = P.copy[P.n_copy++];
        c.dst[0] = g->ws + n.state[0].offset;
        c.dst[1] = g->ws + n.state[1].offset;
        c.bytes = (size_t)g->batch * n.d.h * n.d.w * n.d.c * g->elem;
        c.slot = (int)i;
        c.first_block = blocks;
        blocks += (int)std::min<size_t>(beside ? sms : sms * 2, (c.bytes / 16 + kInputThreads - 1) / kInputThreads + 1);
    }
    for (; next < stems.size() && P.n_stem < kStemsPerLaunch; ++next) {
        const SrStem& st = *stems[next];
        SrStemPart& d = P.stem[P.n_stem++];
        d.dst[0] = st.dst[0]; d.dst[1] = st.dst[1];
        d.slot = st.slot;
        d.Hs = st.Hs; d.Ws = st.Ws; d.Cs = st.Cs; d.Ho = st.Ho; d.Wo = st.Wo;
        d.k = st.k; d.stride = st.stride; d.pad = st.pad; d.Kp = st.Kp; d.K = st.K;
        d.first_block = blocks;
        const size_t chunks = (size_t)g->batch * st.Ho * st.Wo * ((st.K + 7) / 8);
        blocks += (int)std::min<size_t>(per_part, (chunks + kInputThreads - 1) / kInputThreads);
    }
    P.n_blocks = blocks;
    return P;
}

// The staged edges that stems_R names (bit 0: those that read the frame's input within the frame, R = 0; bit 1: a frame later).
inline const std::vector<const SrStem*>& sr_stems(const sr_graph* g, unsigned stems_R) { return g->stems_of[stems_R & 3u]; }
