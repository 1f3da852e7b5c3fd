// Dense resident engine: the frame update  x_v = sigma(b_v + sum_e f_e(theta_e, x_src(e)))  (paper Sec. A1.2) of a small network
// whose edges are dense, or small convolutions, for all T frames of a run in ONE launch.  Arithmetic is fp32; bf16 states are
// rounded when they are stored and lie in shared memory as fp32.
//
// Such a network (the paper's H2 / O layers, a tiny MLP) moves a few hundred kilobytes of weights per frame and does a
// million multiply-adds: launched frame by frame it is pure launch latency.  Here a cluster of eight or sixteen CTAs
// keeps ALL weights in shared memory, split by output rows, and walks the frames of two, four or eight sequences by itself:
//   - every CTA holds a full copy of every node state of its sequences (two buffers by frame parity; input
//     nodes three, because the next input frame is fetched with cp.async while the current update still reads the
//     previous one);
//   - a work unit is up to four output rows of one node; a warp takes a unit, its lanes stride over the reduction
//     index with 16-byte loads (one weight vector per row, one state vector per sequence), multiply-adds are two to an
//     instruction (fma.rn.f32x2 on neighbouring elements of the vectors), shuffles sum the
//     lanes (halving the number of values per step until a group of lanes holds the four rows of one sequence), and the
//     results (bias, ReLU) are written as one 16-byte word into the state copies of ALL CTAs of the cluster; warps never wait
//     for each other inside a level.  (Measured alternative: four-row units cut along the reduction index into parts on up to
//     fourteen warps that hand their partial sums on through shared memory, 3.1 against 2.8 us per frame at the time: the
//     shared-memory traffic stays the same and every part pays the reduction over the lanes.)
//   - units are given to the warps longest first (host side); the warps left without a unit in the first level fetch
//     the next input frame;
//   - a tableau level (Eq. 4) ends when its new states have arrived: the stores into the other CTAs (st.async) count their
//     bytes on a barrier there, one per level and frame parity, which every warp waits for (bounded: on expiry the kernel
//     records an error and returns).  No cluster-wide barrier per frame.
// What bounds it: latency.  On the 784-128-128-10 network, B = 8, 256 frames took 721 us (2.70 per further frame) with eight
// sequences per cluster, sixteen warps, scalar multiply-adds and a cluster barrier per frame, 656 us (2.49) with the packed
// multiply-adds and the counted stores, whose shared-memory loads per step stayed the same, and take 388 us (1.45) with two
// sequences per cluster.
// Convolutions (a few thousand weights, the paper's H1 of the MNIST networks): every CTA keeps all weights of the edge, [K][C].  A work
// unit is eight quads (a pixel and four neighbouring channels each) for up to four sequences; a lane takes a quad and a quarter of the
// reduction, taps outside the image left out, and after a sum over the quarters writes four channels of one sequence.  A rank computes
// a run of quads; the sequences lie quad by quad side by side (and an unused one, against bank conflicts), so what a rank has computed
// is one piece, which goes to every other CTA as one bulk copy when its last unit is done.  MNIST network SR, fp32, 100 sequences, us
// per frame: 12.1 launched, 8.1 here (sequential 19.2 and 9.3).  Bound by the instructions around the multiply-adds with two warps
// per scheduler; walked tap by tap instead of row by row it took 11.2.
// The sums run in a fixed order, so results are reproducible bit for bit.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "sr_dense.h"
#include "sr_resident.h"

namespace {

constexpr int kDnMaxNodes = 16, kDnMaxEdges = 32, kDnMaxLevels = 16, kDnMaxUnits = 128;
constexpr int kDnMaxSamples = 8;       // sequences per cluster, most
constexpr int kDnMoreThanHalf = 120 * 1024;   // of an SM's shared memory, bytes
constexpr int kDnMaxCluster = 16;      // CTAs per cluster: 8, or 16 (a non-portable size) for rollouts with one level per frame
constexpr int kDnWarps = 8;            // 256 threads: a work unit keeps 64 registers of packed accumulators and its operands
constexpr int kDnRows = 4;             // output rows per work unit
constexpr int kDnHeld = 8;             // vectors of a bf16 input frame that a fetching thread has on their way at a time
// Multiply-adds per sample and frame of all convolutions, most.  Of the networks measured (28 x 28 x 1 to 7 x 7 x 16..108, 14 x 14 x 4 to a
// recurrent 7 x 7 x 8..40) those with more did not fit the shared memory, but for one of 296 thousand at up to 16 sequences (launched /
// here 6.8 / 3.5 us per frame at one); at 211 thousand it is 6.4 / 3.6, 11.7 / 8.2 at 64.
constexpr int kDnConvWork = 1 << 18;
constexpr int kDnSmemMax = 226 * 1024;

struct DnNode {
    void* gstate[2];                   // state buffers in global memory, [B][C], by frame parity
    const float* bias;
    int32_t C, Cpad, act, is_input, input_slot, is_output;   // C: values of a sample
    int32_t n_bias, step, seq;         // in shared memory: floats from one vector of four values to the next, from one sequence to the next
    int32_t buf[3];                    // float offsets of the shared-memory state buffers: frame f lives in buf[f % 3] (input
                                       // nodes) or buf[f & 1] (others)
    int32_t bias_off;                  // float offset of the node's bias copy in shared memory
};

struct DnEdge { int32_t src, tgt, R, Kpad; };

// One incoming edge of a work unit, ready to use (32 bytes): where the unit's weight rows start (floats from the
// rank's first weight), the padded reduction length = row pitch of the weights, the row pitch of the source state,
// the frames the edge looks back (Eq. 2), and the source's shared-memory buffers (three for an input node).
struct DnTerm { int32_t w_off, Kpad, xp, R, n_buf, buf[3]; };   // n_buf: also, << 8, floats from one vector of four to the next
static_assert(sizeof(DnTerm) == 32, "read as two 16-byte words");

// The second term of an edge of a convolution unit; there Kpad = k | stride << 8 | pad << 16.
struct DnConv { int32_t Hs, Ws, Cs, pad_[5]; };
static_assert(sizeof(DnConv) == sizeof(DnTerm), "lies among the terms");

// Up to four rows of a node with everything a warp needs (48 bytes).  nrows = 0: no unit (a gap in a warp's list).  A convolution unit:
// nrows = quads, row0 = the first of them, Cpad = floats from one to the next, channels, width, first = channels and width of the node,
// first sequence.
struct DnUnit {
    int32_t nrows, row0, term0, n_terms;
    int32_t bias_off, Cpad, C, flags;                        // flags: 1 = ReLU, 2 = the output node, 4 = a convolution
    int32_t buf[2];                                          // the node's two shared-memory buffers by frame parity
    int16_t channels, width, first, pad_;
};
static_assert(sizeof(DnUnit) == 48, "read as three 16-byte words");

constexpr int kDnMaxTerms = 256;
constexpr int kDnMaxSlices = kDnMaxNodes;

// What a rank computes of a convolution node: in both buffers of the node, the same place in every CTA's copy.
struct DnSlice { int32_t off[2], bytes, pad_; };

struct DnBlobHdr {                     // head of a rank's blob; the rank's weight slices follow
    int32_t n_units, fetch_mask, idle, pad_;                 // fetch_mask: warps that fetch input frames; idle: the rank has no unit
    int32_t level_begin[kDnMaxLevels + 1];                   // units of level l: [level_begin[l-1], level_begin[l]); warp w
    int32_t pad2_[3];                                        // takes entries w, w + kDnWarps, ... of a level
    int32_t level_bytes[kDnMaxLevels];                       // bytes of a level's new states that arrive from elsewhere (or are
                                                             // sent to the rank itself)
    int32_t conv_units[kDnMaxLevels], first_slice[kDnMaxLevels + 4];      // convolution units of a level, and slices
    DnSlice slices[kDnMaxSlices];
    DnUnit units[kDnMaxUnits];
    DnTerm terms[kDnMaxTerms];
};
static_assert(sizeof(DnBlobHdr) % 16 == 0, "the weights that follow are read with 16-byte loads");
static_assert(offsetof(DnBlobHdr, units) % 16 == 0 && offsetof(DnBlobHdr, terms) % 16 == 0, "tables are read with 16-byte loads");

struct DnParams {
    int32_t n_nodes, n_edges, n_levels, B;
    int32_t blob_bytes, hdr_floats, total_floats, n_idle;    // n_idle: ranks without a unit
    int32_t* error;                                          // device-side error code
    long long wait_limit;                                    // cycles after which a wait gives up
    const unsigned char* blobs;        // one blob of blob_bytes per rank of the cluster
    DnNode nodes[kDnMaxNodes];
    DnEdge edges[kDnMaxEdges];
    int32_t first_edge[kDnMaxNodes + 1];                     // edges are sorted by target node
};

__device__ __forceinline__ void dn_cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void dn_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dn_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t dn_map_rank(uint32_t local, uint32_t rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
// Stores into another CTA's shared memory that count their bytes on a barrier there: whoever waits for the barrier sees them.
__device__ __forceinline__ void dn_st_async(uint32_t cell, uint32_t bar, uint32_t rank, float v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];"
                 ::"r"(dn_map_rank(cell, rank)), "f"(v), "r"(dn_map_rank(bar, rank)) : "memory");
}
__device__ __forceinline__ void dn_st_async4(uint32_t cell, uint32_t bar, uint32_t rank, const float (&v)[4])
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(dn_map_rank(cell, rank)), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(dn_map_rank(bar, rank)) : "memory");
}
__device__ __forceinline__ bool dn_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for a phase of a barrier that other CTAs' stores complete.
__device__ __forceinline__ bool dn_wait(uint32_t bar, uint32_t parity, volatile int* gave_up, long long limit)
{
    long long t0 = 0;
    for (int i = 0;; ++i) {
        if (dn_try_wait(bar, parity)) return true;
        if ((i & 31) == 31) {
            const long long t = clock64();
            if (t0 == 0) t0 = t;
            if (*gave_up || t - t0 > limit) {
                *gave_up = 1;
                return false;
            }
        }
    }
}

// Fetch `n` floats (a multiple of 4, 16-byte aligned on both sides) with cp.async.
__device__ __forceinline__ void dn_fetch(float* dst, const float* src, int n, int tid, int nthr)
{
    for (int i = tid * 4; i < n; i += nthr * 4) dn_cp_async16(dst + i, src + i);
}

// Two fp32 multiply-adds in one instruction: (acc.lo, acc.hi) += (a.lo * x.lo, a.hi * x.hi).
__device__ __forceinline__ void dn_fma2(unsigned long long& acc, unsigned long long a, unsigned long long x)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(x));
}
// acc[r][b0 + b] += a[r] . x[b] for G sequences: the even and the odd elements of the vectors are summed side by side.  Written
// component by component so that consecutive multiply-adds are independent of each other.
template <int R, int S, int G>
__device__ __forceinline__ void dn_fma(unsigned long long (&acc)[R][S], const ulonglong2 (&a)[R], const ulonglong2 (&x)[G], int b0)
{
#pragma unroll
    for (int b = 0; b < G; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) dn_fma2(acc[r][b0 + b], a[r].x, x[b].x);
#pragma unroll
    for (int b = 0; b < G; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) dn_fma2(acc[r][b0 + b], a[r].y, x[b].y);
}

// One halving step of the sum over the lanes: with distance D a lane keeps the half of its N values per row that matches its bit D
// and adds the partner's.
template <int R, int N, int D>
__device__ __forceinline__ void dn_halve(float (&out)[R][N / 2], const float (&v)[R][N], int lane)
{
    const bool up = (lane & D) != 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < N / 2; ++j) {
            const float keep = up ? v[r][j + N / 2] : v[r][j], send = up ? v[r][j] : v[r][j + N / 2];
            out[r][j] = keep + __shfl_xor_sync(0xffffffffu, send, D);
        }
}

// A value as a state of type T holds it.
template <typename T>
__device__ __forceinline__ float dn_rounded(float v) { return sizeof(T) == 2 ? __bfloat162float(__float2bfloat16_rn(v)) : v; }

// One work unit: up to R rows of a node for the S sequences of the cluster, relative frame f -> f + 1.
// The loads of a reduction step are issued ahead of the multiply-adds that use them: the weights and the first four
// sequences of step i + 1 while the last four sequences of step i are still being multiplied.
// (MIXED: a source may be a convolution, whose vectors of four lie further apart.)
template <int R, int CL, int S, typename T, bool MIXED>
__device__ __forceinline__ void dn_unit(const DnBlobHdr* H, const DnUnit& un, float* dn_mem, const float* wsm,
                                        const SrFrameCtl& init, int f, int lane, int b0, int nb, long long run0, uint32_t bar)
{
    unsigned long long acc2[R][S];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int b = 0; b < S; ++b) acc2[r][b] = 0ull;
    for (int ti = un.term0; ti < un.term0 + un.n_terms; ++ti) {
        const DnTerm tm = H->terms[ti];
        const int sf = f + 1 - tm.R;                                  // Eq. 2: the source frame
        const int bi = (tm.n_buf & 0xFF) == 3 ? sf % 3 : (sf & 1), step = MIXED ? tm.n_buf >> 8 : 4;
        const float* xs = dn_mem + (bi == 0 ? tm.buf[0] : (bi == 1 ? tm.buf[1] : tm.buf[2])) + lane * step;
        const float* w0 = wsm + tm.w_off + lane * 4;
        int ro[R];                                                    // rows the unit does not have repeat row 0 (their sums are dropped)
#pragma unroll
        for (int r = 0; r < R; ++r) ro[r] = r < un.nrows ? r * tm.Kpad : 0;
        const int xp = tm.xp, n_k = tm.Kpad - lane * 4;               // this lane's steps: k = 0, 128, ... < n_k
        if (n_k <= 0) continue;
        constexpr int G = S < 4 ? S : 4;                              // sequences whose loads are issued together
        ulonglong2 a[R], xa[G];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = *reinterpret_cast<const ulonglong2*>(w0 + ro[r]);
#pragma unroll
        for (int b = 0; b < G; ++b) xa[b] = *reinterpret_cast<const ulonglong2*>(xs + b * xp);
        for (int k = 0, x = 0; k < n_k; k += 128, x += 32 * step) {
            ulonglong2 an[R], xb[G];
            const int kn = k + 128 < n_k ? k + 128 : k;               // the last step re-reads itself (no branch)
            const int xn = MIXED ? (k + 128 < n_k ? x + 32 * step : x) : kn;
            if (S > G) {
#pragma unroll
                for (int b = 0; b < G; ++b) xb[b] = *reinterpret_cast<const ulonglong2*>(xs + (b + G) * xp + (MIXED ? x : k));
                dn_fma<R, S, G>(acc2, a, xa, 0);
#pragma unroll
                for (int r = 0; r < R; ++r) an[r] = *reinterpret_cast<const ulonglong2*>(w0 + ro[r] + kn);
#pragma unroll
                for (int b = 0; b < G; ++b) xa[b] = *reinterpret_cast<const ulonglong2*>(xs + b * xp + xn);
                dn_fma<R, S, G>(acc2, a, xb, S - G);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) an[r] = *reinterpret_cast<const ulonglong2*>(w0 + ro[r] + kn);
#pragma unroll
                for (int b = 0; b < G; ++b) xb[b] = *reinterpret_cast<const ulonglong2*>(xs + b * xp + xn);
                dn_fma<R, S, G>(acc2, a, xa, 0);
#pragma unroll
                for (int b = 0; b < G; ++b) xa[b] = xb[b];
            }
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = an[r];
        }
    }
    float acc[R][S];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int b = 0; b < S; ++b) acc[r][b] = __uint_as_float((uint32_t)acc2[r][b]) + __uint_as_float((uint32_t)(acc2[r][b] >> 32));
    // Sum over the lanes: halving steps until a lane holds the R rows of ONE sequence, lane / (32 / S), then plain butterflies
    // among the 32 / S lanes that hold the same one.
    float z[R];
    if constexpr (S == 8) {
        float v4[R][4], v2[R][2], v1[R][1];
        dn_halve<R, 8, 16>(v4, acc, lane);
        dn_halve<R, 4, 8>(v2, v4, lane);
        dn_halve<R, 2, 4>(v1, v2, lane);
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = v1[r][0];
    } else if constexpr (S == 4) {
        float v2[R][2], v1[R][1];
        dn_halve<R, 4, 16>(v2, acc, lane);
        dn_halve<R, 2, 8>(v1, v2, lane);
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = v1[r][0];
    } else {
        float v1[R][1];
        dn_halve<R, 2, 16>(v1, acc, lane);
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = v1[r][0];
    }
#pragma unroll
    for (int d = 16 / S; d > 0; d >>= 1)
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] += __shfl_xor_sync(0xffffffffu, z[r], d);
    constexpr int kLanes = 32 / S;                                    // lanes that hold the same sequence
    const int b = lane / kLanes;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        z[r] += dn_mem[un.bias_off + un.row0 + (r < un.nrows ? r : 0)];
        if (un.flags & 1) z[r] = fmaxf(z[r], 0.f);
    }
    float y[R];                                                       // as the state holds them
#pragma unroll
    for (int r = 0; r < R; ++r) y[r] = dn_rounded<T>(z[r]);
    const uint32_t cell = dn_smem(dn_mem + (((f + 1) & 1) ? un.buf[1] : un.buf[0]) + b * un.Cpad + un.row0);
    constexpr uint32_t kPerLane = CL > kLanes ? CL / kLanes : 1;      // ranks that each of them serves
    const uint32_t q = (uint32_t)(lane % kLanes) * kPerLane;
    if (q >= CL) {
        // (more lanes than ranks: nothing to send)
    } else if (R == 4 && un.nrows == 4 && (un.row0 & 3) == 0) {
        const float z4[4] = {y[0], y[1], y[2 % R], y[3 % R]};
#pragma unroll
        for (uint32_t i = 0; i < kPerLane; ++i) dn_st_async4(cell, bar, q + i, z4);
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < un.nrows) {
#pragma unroll
                for (uint32_t i = 0; i < kPerLane; ++i) dn_st_async(cell + 4 * r, bar, q + i, y[r]);
            }
    }
    if ((un.flags & 2) && init.out_base && lane % kLanes == 0 && b < nb) {
        float* o = init.out_base + (run0 + f) * init.out_stride + (long long)(b0 + b) * un.C + un.row0;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < un.nrows) o[r] = z[r];
    }
}

// A convolution unit (see the file comment): eight quads, four slices of the reduction (lane / 8), N sequences.
template <int CL, int N, typename T>
__device__ __forceinline__ void dn_conv_unit(const DnBlobHdr* H, const DnUnit& un, float* dn_mem, const float* wsm,
                                             const SrFrameCtl& init, int f, int lane, int b0, int nb, long long run0, uint32_t bar,
                                             int level, uint32_t rank, int* done)
{
    const int slice = lane >> 3, at = min(lane & 7, un.nrows - 1);
    const int quads = un.channels >> 2, idx = un.row0 + at, C = un.channels;
    const int px = idx / quads, ch = (idx - px * quads) * 4, oy = px / un.width, ox = px - oy * un.width;
    unsigned long long acc[N][2];
#pragma unroll
    for (int s = 0; s < N; ++s) acc[s][0] = acc[s][1] = 0ull;
    auto pair = [](float v) {
        unsigned long long r;
        asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
        return r;
    };
    for (int ti = un.term0; ti < un.term0 + 2 * un.n_terms; ti += 2) {
        const DnTerm tm = H->terms[ti];
        const DnConv cv = *reinterpret_cast<const DnConv*>(&H->terms[ti + 1]);
        const int k = tm.Kpad & 0xFF, stride = (tm.Kpad >> 8) & 0xFF, pad = tm.Kpad >> 16, Cs = cv.Cs, xp = tm.xp;
        const int sf = f + 1 - tm.R;                                  // Eq. 2: the source frame
        const int bi = (tm.n_buf & 0xFF) == 3 ? sf % 3 : (sf & 1), step = tm.n_buf >> 8;
        const int y0 = oy * stride - pad, x0 = ox * stride - pad;
        const float* xs = dn_mem + (bi == 0 ? tm.buf[0] : (bi == 1 ? tm.buf[1] : tm.buf[2])) + un.first * xp;
        const int origin = (y0 * cv.Ws + x0) * Cs;
        const float* w0 = wsm + tm.w_off + ch;
        // a filter row is one run of values; the slices take its values (in fours where the source has whole vectors) in turn
        const int kx0 = max(0, -x0), kx1 = min(k, cv.Ws - x0);
        for (int ky = max(0, -y0); ky < min(k, cv.Hs - y0); ++ky) {
            const int at0 = origin + ky * cv.Ws * Cs;
            const float* w = w0 + ky * k * Cs * C;
            if ((Cs & 3) == 0) {
                const int e0 = kx0 * Cs >> 2, e1 = kx1 * Cs >> 2;
                int e = e0 + ((slice - e0) & 3);
                const float* x = xs + ((at0 >> 2) + e) * step;
                const float* wp = w + 4 * e * C;
#pragma unroll 2
                for (; e < e1; e += 4, x += 4 * step, wp += 16 * C) {
                    float4 v[N];
                    ulonglong2 wv[4];
#pragma unroll
                    for (int s = 0; s < N; ++s) v[s] = *reinterpret_cast<const float4*>(x + s * xp);
#pragma unroll
                    for (int q = 0; q < 4; ++q) wv[q] = *reinterpret_cast<const ulonglong2*>(wp + q * C);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int s = 0; s < N; ++s) {
                            const unsigned long long xx = pair(q == 0 ? v[s].x : q == 1 ? v[s].y : q == 2 ? v[s].z : v[s].w);
                            dn_fma2(acc[s][0], wv[q].x, xx);
                            dn_fma2(acc[s][1], wv[q].y, xx);
                        }
                }
            } else {
                const int e0 = kx0 * Cs, e1 = kx1 * Cs;
                int e = e0 + ((slice - e0) & 3);
                const float* x = xs + at0 + e;
                const float* wp = w + e * C;
#pragma unroll 2
                for (; e < e1; e += 4, x += 4, wp += 4 * C) {
                    const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(wp);
#pragma unroll
                    for (int s = 0; s < N; ++s) {
                        const unsigned long long xx = pair(x[s * xp]);
                        dn_fma2(acc[s][0], wv.x, xx);
                        dn_fma2(acc[s][1], wv.y, xx);
                    }
                }
            }
        }
    }
    __syncwarp();
    // Sum over the slices: halving steps until a lane holds the four channels of one sequence (N = 4: sequence `slice`; N = 2: sequence
    // slice / 2, in two lanes).
    float a[4][N], z[4];
#pragma unroll
    for (int s = 0; s < N; ++s) {
        a[0][s] = __uint_as_float((uint32_t)acc[s][0]); a[1][s] = __uint_as_float((uint32_t)(acc[s][0] >> 32));
        a[2][s] = __uint_as_float((uint32_t)acc[s][1]); a[3][s] = __uint_as_float((uint32_t)(acc[s][1] >> 32));
    }
    float h[4][N / 2];
    dn_halve<4, N, 16>(h, a, lane);
    if constexpr (N == 4) {
        float h1[4][1];
        dn_halve<4, 2, 8>(h1, h, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = h1[i][0];
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = h[i][0] + __shfl_xor_sync(0xffffffffu, h[i][0], 8);
    }
    const int b = un.first + (N == 4 ? slice : slice >> 1);
    const float4 bias = *reinterpret_cast<const float4*>(dn_mem + un.bias_off + ch);
    z[0] += bias.x; z[1] += bias.y; z[2] += bias.z; z[3] += bias.w;
    if (un.flags & 1)
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = fmaxf(z[i], 0.f);
    if ((lane & 7) < un.nrows) {
        if ((un.flags & 2) && init.out_base && b < nb && (N == 4 || (slice & 1) == 0)) {
            float* o = init.out_base + (run0 + f) * init.out_stride + (long long)(b0 + b) * un.C + idx * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = z[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = dn_rounded<T>(z[i]);
        if (N == 4 || (slice & 1) == 0)
            *reinterpret_cast<float4*>(dn_mem + (((f + 1) & 1) ? un.buf[1] : un.buf[0]) + idx * un.Cpad + b * 4) = make_float4(z[0], z[1], z[2], z[3]);
    }
    // the unit that is the rank's last of its level sends what the rank has computed
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __threadfence_block();
    __syncwarp();
    int last = 0;
    if (lane == 0) last = atomicAdd(done, 1) == H->conv_units[level] - 1;
    if (__shfl_sync(0xffffffffu, last, 0)) {
        __threadfence_block();
        if (lane == 0) {
            *done = 0;
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (lane < CL && lane != (int)rank)
            for (int i = H->first_slice[level]; i < H->first_slice[level + 1]; ++i) {
                const uint32_t src = dn_smem(dn_mem + H->slices[i].off[(f + 1) & 1]);
                asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(dn_map_rank(src, (uint32_t)lane)), "r"(src), "r"(H->slices[i].bytes), "r"(dn_map_rank(bar, (uint32_t)lane)) : "memory");
            }
    }
    __syncwarp();
}

// `n` values (a multiple of 4) of a state in global memory into shared memory, as fp32.
__device__ __forceinline__ void dn_load(float* dst, const float* src, int n, int tid, int nthr) { dn_fetch(dst, src, n, tid, nthr); }
__device__ __forceinline__ void dn_load(float* dst, const __nv_bfloat16* src, int n, int tid, int nthr)
{
#pragma unroll 4
    for (int i = tid * 4; i < n; i += nthr * 4) {
        const uint2 q = *reinterpret_cast<const uint2*>(src + i);
        *reinterpret_cast<float4*>(dst + i) = make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u),
                                                          __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xFFFF0000u));
    }
}
__device__ __forceinline__ float4 dn_widen(uint2 q)
{
    return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u), __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xFFFF0000u));
}
__device__ __forceinline__ float dn_value(float v) { return v; }
__device__ __forceinline__ float dn_value(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void dn_store(float* p, float v) { *p = v; }
__device__ __forceinline__ void dn_store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void dn_store4(float* p, const float* v) { *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(v); }
__device__ __forceinline__ void dn_store4(__nv_bfloat16* p, const float* v)
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

template <int CL, int S, typename T, bool CONV>
__global__ void __launch_bounds__(kDnWarps * 32, 1)
sr_dense_kernel(const DnParams P, const SrFrameCtl init, int n_frames)
{
    extern __shared__ __align__(16) float dn_mem[];
    // the input nodes as the fetching warps need them: first float of this cluster's sequences in the caller's frame 0
    // of the run, floats from one frame to the next, floats per frame, the three shared-memory buffers
    __shared__ const T* in_src[SR_MAX_INPUTS];
    __shared__ long long in_step[SR_MAX_INPUTS];
    __shared__ int in_len[SR_MAX_INPUTS], in_buf[SR_MAX_INPUTS][3], n_in, n_vectors;   // n_vectors: of four values, in a frame of all inputs
    __shared__ uint64_t bars[kDnMaxLevels][2];               // per level and frame parity: the level's new states have arrived
    __shared__ int gave_up, conv_done;
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
    sr_let_successor_start();
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int b0 = (int)(blockIdx.x / CL) * S;
    const int nb = min(S, P.B - b0);
    const DnBlobHdr* H = reinterpret_cast<const DnBlobHdr*>(dn_mem);
    const float* wsm = dn_mem + P.hdr_floats;

    // this rank's tables and weight slices, and zeros in every state buffer (padding columns and unused sequences stay zero)
    {
        const float* blob = reinterpret_cast<const float*>(P.blobs + (size_t)rank * P.blob_bytes);
        dn_fetch(dn_mem, blob, P.blob_bytes / 4, tid, nthr);
        for (int i = P.blob_bytes / 4 + tid; i < P.total_floats; i += nthr) dn_mem[i] = 0.f;
        __syncthreads();
        for (int v = 0; v < P.n_nodes; ++v)                  // (biases, like weights, are the host's)
            if (!P.nodes[v].is_input)
                for (int i = tid; i < P.nodes[v].n_bias; i += nthr) dn_mem[P.nodes[v].bias_off + i] = P.nodes[v].bias[i];
    }
    const long long t0 = init.t, run0 = init.run_t;
    if (tid == 0) {
        gave_up = 0;
        conv_done = 0;
        int n = 0;
        n_vectors = 0;
        for (int v = 0; v < P.n_nodes; ++v) {
            const DnNode& nd = P.nodes[v];
            if (!nd.is_input) continue;
            in_src[n] = reinterpret_cast<const T*>(static_cast<const char*>(init.in_base[nd.input_slot]) + run0 * init.in_stride_bytes[nd.input_slot]) + (size_t)b0 * nd.C;
            in_step[n] = init.in_stride_bytes[nd.input_slot] / (long long)sizeof(T);
            in_len[n] = nb * nd.C;                           // input nodes have Cpad == C
            n_vectors += nb * nd.C / 4;
            for (int i = 0; i < 3; ++i) in_buf[n][i] = nd.buf[i];
            ++n;
        }
        n_in = n;
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (tid < 2 * P.n_levels) {
        // one arrival announces the bytes; in the last level every fetching thread arrives when its copies have landed, and
        // every rank that sends no states does once per frame; in a level with convolutions, what this rank computes is complete
        const int l = tid >> 1, n_arrive = 1 + (H->conv_units[l] > 0) + (l == P.n_levels - 1 ? 32 * __popc(H->fetch_mask) + P.n_idle : 0);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(dn_smem(&bars[l][tid & 1])), "r"(n_arrive) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // (their bulk copies go where this thread has stored zeros)
    // The other CTAs may store into this one from here on: its barriers stand, the buffers of frame 1 are zeroed, and those of frame 0,
    // filled below, are stored into again only once this CTA has sent its part of frame 1.
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    // (Weights and tables do not depend on the kernel before this one; states and input frames do.)
    sr_wait_for_predecessor();
    // frame t of every node from the state buffers in global memory (relative frame 0)
    const int par0 = (int)(t0 & 1);
    for (int v = 0; v < P.n_nodes; ++v) {
        const DnNode& nd = P.nodes[v];
        const T* gsrc = static_cast<const T*>(nd.gstate[par0]) + (size_t)b0 * nd.C;
        float* dst = dn_mem + nd.buf[0];
        if (CONV && nd.step != 4)
            for (int i = tid; i < nb * (nd.C / 4); i += nthr) {
                const int b = i / (nd.C / 4), v = i - b * (nd.C / 4);
                dn_load(dst + v * nd.step + b * nd.seq, gsrc + 4 * i, 4, 0, 1);
            }
        else if (nd.Cpad == nd.C) dn_load(dst, gsrc, nb * nd.C, tid, nthr);              // rows are contiguous: four values at a time
        else
            for (int i = tid; i < nb * nd.C; i += nthr) dst[(i / nd.C) * nd.Cpad + (i % nd.C)] = dn_value(gsrc[i]);
    }
    // Input frame k of the run (relative frame k) -> buffer k % 3, by the warps of fetch_mask.
    const int f_nthr = 32 * __popc(H->fetch_mask);
    const int f_tid = (H->fetch_mask >> warp) & 1 ? 32 * __popc(H->fetch_mask & ((1 << warp) - 1)) + lane : -1;
    auto fetch_inputs = [&](int k) {
        if (f_tid < 0) return;
        for (int i = 0; i < n_in; ++i) dn_load(dn_mem + in_buf[i][k % 3], in_src[i] + (k - 1) * in_step[i], in_len[i], f_tid, f_nthr);
    };
    fetch_inputs(1);
    // What a fetching thread takes of input frame k: vectors of four values f_nthr apart, through all inputs, kDnHeld of them from its
    // `first` on.  (Where a vector lies is worked out from the one before, and what exceeds kDnHeld goes in as many at a time.  With a
    // search per vector and the rest one by one these few warps were what the frame waited for: 784-128-128-10 network in bf16, us per
    // frame at 8 / 32 / 64 / 256 sequences 2.60 / 5.24 / 5.24 / 15.2, so 2.01 / 3.65 / 4.53 / 13.1; with 12 or 16 the same.)
    uint2 held[kDnHeld];
    auto each_vector = [&](int first, int k, auto&& take) {
        int i = -1, len = 0, v = f_tid + first * f_nthr;
        const T* src = nullptr;
        float* dst = nullptr;
#pragma unroll
        for (int r = 0; r < kDnHeld; ++r, v += f_nthr) {
            while (v * 4 >= len) {
                v -= len / 4;
                if (++i >= n_in) return;
                len = in_len[i];
                src = in_src[i] + (k - 1) * in_step[i];
                dst = dn_mem + in_buf[i][k % 3];
            }
            take(r, src + v * 4, dst + v * 4);
        }
    };
    auto hold_vectors = [&](int first, int k) { each_vector(first, k, [&](int r, const T* src, float*) { held[r] = *reinterpret_cast<const uint2*>(src); }); };
    auto store_vectors = [&](int first, int k) { each_vector(first, k, [&](int r, const T*, float* dst) { *reinterpret_cast<float4*>(dst) = dn_widen(held[r]); }); };
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

    int f = 0;
    for (; f < n_frames && !*(volatile int*)&gave_up; ++f) {                         // relative frame f -> f + 1
        // the input frame after the next one is on its way during this update; it has landed when the last level's barrier
        // completes
        const int par = (f + 1) & 1;
        const uint32_t phase = (uint32_t)(f >> 1) & 1u;
        if (sizeof(T) == 4) {
            if (f + 1 < n_frames) fetch_inputs(f + 2);
        } else if (f_tid >= 0 && f + 1 < n_frames) {
            hold_vectors(0, f + 2);
        }
        if (sizeof(T) == 4 && f_tid >= 0) asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(dn_smem(&bars[P.n_levels - 1][par])) : "memory");
        for (int l = 1; l <= P.n_levels; ++l) {
            const uint32_t bar = dn_smem(&bars[l - 1][par]);
            if (tid == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(H->level_bytes[l - 1]) : "memory");
            // Nobody runs more than a frame ahead of a rank, because a level needs the states of every rank with a unit in it;
            // a rank without any says so instead.
            if (H->idle && l == P.n_levels && tid < CL)
                asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(dn_map_rank(bar, (uint32_t)tid)) : "memory");
            for (int u = H->level_begin[l - 1] + warp; u < H->level_begin[l]; u += kDnWarps) {
                const DnUnit un = H->units[u];
                if (un.nrows == 0) continue;
                if (CONV && (un.flags & 4)) dn_conv_unit<CL, S < 4 ? 2 : 4, T>(H, un, dn_mem, wsm, init, f, lane, b0, nb, run0, bar, l - 1, rank, &conv_done);
                else if (un.nrows > 2) dn_unit<4, CL, S, T, CONV>(H, un, dn_mem, wsm, init, f, lane, b0, nb, run0, bar);
                else dn_unit<2, CL, S, T, CONV>(H, un, dn_mem, wsm, init, f, lane, b0, nb, run0, bar);
            }
            // The next input frame, loaded ahead of the update, goes into its buffer; what is more than the threads hold follows, as many
            // vectors on their way as they hold.
            if (sizeof(T) == 2 && l == P.n_levels && f_tid >= 0) {
                if (f + 1 < n_frames) {
                    store_vectors(0, f + 2);
                    for (int first = kDnHeld; f_tid + first * f_nthr < n_vectors; first += kDnHeld) {
                        hold_vectors(first, f + 2);
                        store_vectors(first, f + 2);
                    }
                }
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
            }
            if (!dn_wait(bar, phase, &gave_up, P.wait_limit)) break;    // the level is complete in this CTA's copy
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // Whatever the others send to this CTA counts on a barrier that it has waited for, so it may leave: unless it gave up, or another
    // one still copies out of its shared memory (convolutions).
    __syncthreads();
    if (CONV || *(volatile int*)&gave_up) dn_cluster_sync();
    if (*(volatile int*)&gave_up) {
        // Nobody starts a store any more.  What is on its way lands first: all that can be is of the frame in which the wait expired or
        // of the next; what will not come, because its sender gave up too, ends with the limit.
        if (tid == 0) {
            const long long begin = clock64();
            for (int g = max(f - 1, 0); g <= f && g < n_frames; ++g)
                for (int l = 0; l < P.n_levels; ++l)
                    while (!dn_try_wait(dn_smem(&bars[l][(g + 1) & 1]), (uint32_t)(g >> 1) & 1u) && clock64() - begin <= P.wait_limit) {}
        }
        __syncthreads();
    }
    if (tid == 0 && gave_up) atomicExch(P.error, 1);

    // the last frame back to the state buffers in global memory (parity of t + T); every rank holds a full copy and
    // writes its share of it
    {
        const int parT = (int)((t0 + n_frames) & 1);
        const int gtid = (int)rank * nthr + tid, gthr = CL * nthr;
        for (int v = 0; v < P.n_nodes; ++v) {
            const DnNode& nd = P.nodes[v];
            const float* src = dn_mem + (nd.is_input ? nd.buf[n_frames % 3] : nd.buf[n_frames & 1]);
            T* gdst = static_cast<T*>(nd.gstate[parT]) + (size_t)b0 * nd.C;
            if (CONV && nd.step != 4)
                for (int i = gtid; i < nb * (nd.C / 4); i += gthr) {
                    const int b = i / (nd.C / 4), v = i - b * (nd.C / 4);
                    dn_store4(gdst + 4 * i, src + v * nd.step + b * nd.seq);
                }
            else if (nd.Cpad == nd.C)
                for (int i = gtid * 4; i < nb * nd.C; i += gthr * 4) dn_store4(gdst + i, src + i);
            else
                for (int i = gtid; i < nb * nd.C; i += gthr) dn_store(gdst + i, src[(i / nd.C) * nd.Cpad + (i % nd.C)]);
        }
    }
}

// ------------------------------------------------------------------------------------------ host side
struct DnEngine {
    DnParams P{};
    std::vector<int> edge_of_host;                 // host edge -> index in P.edges
    int cluster = 8;                               // CTAs per cluster
    int samples = 8;                               // sequences per cluster
    bool one_wave = false;                         // the device holds all clusters of the batch at once
    std::vector<int> row_lo;                       // [node][rank] first row of the rank's slice, cluster + 1 entries per node
    std::vector<std::vector<int>> w_off;           // [rank][edge]
    std::vector<DnBlobHdr> hdrs;                   // per rank
    SrRegion r_blobs;
    int smem_bytes = 0;
    bool attr_set = false;
    std::vector<cudaEvent_t> ev;
    size_t ev_used = 0;
};

DnEngine* dn_of(const sr_graph* g) { return static_cast<DnEngine*>(g->dn); }

typedef void (*DnKernel)(const DnParams, const SrFrameCtl, int);

// (The limit belongs to the kernel, not to a graph: always the same value, or a small network would lower a larger one's.)
bool dn_prepare(DnKernel kernel, int cluster)
{
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDnSmemMax) != cudaSuccess) return false;
    if (cluster > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    return true;
}

int dn_values(const sr_graph* g, int v) { return g->nodes[v].d.h * g->nodes[v].d.w * g->nodes[v].d.c; }
bool dn_is_conv(const sr_graph* g, int v) { return !g->nodes[v].is_input && !g->nodes[v].dense_target; }

template <typename T, bool CONV>
DnKernel dn_kernel_of(int cluster, int samples)
{
    if (cluster == 16)
        return samples == 8 ? sr_dense_kernel<16, 8, T, CONV> : samples == 4 ? sr_dense_kernel<16, 4, T, CONV> : sr_dense_kernel<16, 2, T, CONV>;
    return samples == 8 ? sr_dense_kernel<8, 8, T, CONV> : samples == 4 ? sr_dense_kernel<8, 4, T, CONV> : sr_dense_kernel<8, 2, T, CONV>;
}
DnKernel dn_kernel_of(const sr_graph* g, int cluster, int samples)
{
    bool conv = false;
    for (size_t v = 0; v < g->nodes.size(); ++v) conv = conv || dn_is_conv(g, (int)v);
    if (g->dtype == SR_DTYPE_BF16) return conv ? dn_kernel_of<__nv_bfloat16, true>(cluster, samples) : dn_kernel_of<__nv_bfloat16, false>(cluster, samples);
    return conv ? dn_kernel_of<float, true>(cluster, samples) : dn_kernel_of<float, false>(cluster, samples);
}

// Clusters of this size and shared-memory footprint that the device holds at once with one CTA per SM (0: none): two CTAs on an SM
// share its shared-memory pipe, so a second one there gains little over a second wave.
int dn_clusters_held(const sr_graph* g, int cluster, int samples, int smem_bytes)
{
    DnKernel kernel = dn_kernel_of(g, cluster, samples);
    if (!dn_prepare(kernel, cluster)) { cudaGetLastError(); return 0; }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)cluster);
    cfg.blockDim = dim3((unsigned)(kDnWarps * 32));
    cfg.dynamicSmemBytes = (size_t)std::max(smem_bytes, kDnMoreThanHalf);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

// Plans the engine for a cluster of CL CTAs: rows of every node split evenly over the ranks.  Null if it does not fit.
DnEngine* dn_build(const sr_graph* g, int CL, int S)
{
    const int n_nodes = (int)g->nodes.size(), n_edges = (int)g->edges.size();
    DnEngine* E = new DnEngine();
    DnParams& P = E->P;
    E->cluster = CL;
    E->samples = S;
    P.n_nodes = n_nodes;
    P.n_edges = n_edges;
    P.n_levels = (int)g->groups.size();
    P.B = g->batch;
    // edges sorted by target
    E->edge_of_host.assign(n_edges, -1);
    int pos = 0;
    const SrHostEdge* host_edge[kDnMaxEdges] = {};
    for (int v = 0; v < n_nodes; ++v) {
        P.first_edge[v] = pos;
        for (int e : g->nodes[v].in_edges) {
            const SrHostEdge& he = g->edges[e];
            const int Kpad = (dn_values(g, he.d.src) + 3) / 4 * 4;
            P.edges[pos] = DnEdge{he.d.src, he.d.tgt, he.R, Kpad};
            host_edge[pos] = &he;
            E->edge_of_host[e] = pos++;
        }
    }
    P.first_edge[n_nodes] = pos;
    // row slices and weight offsets per rank
    E->row_lo.assign((size_t)n_nodes * (CL + 1), 0);
    E->w_off.assign(CL, std::vector<int>(kDnMaxEdges, 0));
    int max_w = 0;
    for (int v = 0; v < n_nodes; ++v)
        for (int r = 0; r <= CL; ++r) E->row_lo[(size_t)v * (CL + 1) + r] = dn_is_conv(g, v) ? 0 : dn_values(g, v) * r / CL;
    for (int r = 0; r < CL; ++r) {
        int w = 0;
        for (bool conv : {true, false})                          // (convolutions first: at the same place in every rank)
            for (int e = 0; e < n_edges; ++e) {
                const int v = P.edges[e].tgt;
                if (dn_is_conv(g, v) != conv) continue;
                const int rows = E->row_lo[(size_t)v * (CL + 1) + r + 1] - E->row_lo[(size_t)v * (CL + 1) + r];
                E->w_off[r][e] = w;
                w += conv ? host_edge[e]->K * g->nodes[v].d.c : rows * P.edges[e].Kpad;
            }
        max_w = std::max(max_w, w);
    }
    // shared-memory layout in floats: header, weights, state buffers
    int off = (int)(sizeof(DnBlobHdr) / 4);
    P.hdr_floats = off;
    off += (max_w + 3) / 4 * 4;
    P.blob_bytes = off * 4;
    for (int v = 0; v < n_nodes; ++v) {
        const SrHostNode& n = g->nodes[v];
        DnNode& d = P.nodes[v];
        d.C = dn_values(g, v);
        d.Cpad = (d.C + 3) / 4 * 4;
        d.n_bias = n.d.c;
        d.act = n.d.act;
        d.is_input = n.is_input ? 1 : 0;
        d.input_slot = n.input_slot;
        d.is_output = v == g->info.output_node ? 1 : 0;
        // (a convolution's sequences lie side by side, vector by vector)
        const bool conv = dn_is_conv(g, v);
        d.step = conv ? 4 * (S + 1) : 4;
        d.seq = conv ? 4 : d.Cpad;
        for (int i = 0; i < (n.is_input ? 3 : 2); ++i) {
            d.buf[i] = off;
            off += conv ? d.C / 4 * d.step : S * d.Cpad;
        }
        d.bias_off = off;
        if (!n.is_input) off += (n.d.c + 3) / 4 * 4;
    }
    P.total_floats = off;
    E->smem_bytes = off * 4;
    if (E->smem_bytes > kDnSmemMax) {
        delete E;
        return nullptr;
    }
    // Per rank: units (up to four rows of a node each) with their terms (one per incoming edge).  The units of a level
    // go longest first onto the warp with the least work so far; warp w's i-th unit of the level is entry
    // level_begin + kDnWarps * i + w (gaps have nrows = 0).
    std::vector<DnBlobHdr>& hdrs = E->hdrs;
    hdrs.assign(CL, DnBlobHdr{});
    for (int r = 0; r < CL; ++r) {
        DnBlobHdr& h = hdrs[r];
        std::memset(&h, 0, sizeof(h));
        int n_units = 0, n_terms = 0, n_slices = 0;
        bool fits = true;
        for (int l = 1; l <= P.n_levels && fits; ++l) {
            std::vector<std::pair<long long, DnUnit>> lv;
            h.first_slice[l - 1] = n_slices;
            for (int v : g->groups[l - 1]) {
                const DnNode& d = P.nodes[v];
                if (!dn_is_conv(g, v)) h.level_bytes[l - 1] += d.C * S * 4;
                long long K = 0;
                for (int e = P.first_edge[v]; e < P.first_edge[v + 1]; ++e) K += P.edges[e].Kpad;
                const int lo = E->row_lo[(size_t)v * (CL + 1) + r], hi = E->row_lo[(size_t)v * (CL + 1) + r + 1];
                // a convolution: a run of its blocks of eight quads
                const int quads = d.C / 4, blocks = dn_is_conv(g, v) ? (quads + 7) / 8 : 0, seqs = std::min(S, 4);
                const int first = blocks * r / CL, end = blocks * (r + 1) / CL;
                if (blocks > 0) {
                    const int q0 = std::min(quads, first * 8), q1 = std::min(quads, end * 8);
                    h.level_bytes[l - 1] += (quads - (q1 - q0)) * d.step * 4;
                    h.conv_units[l - 1] += (end - first) * (S / seqs);
                    if (q1 > q0) h.slices[n_slices++] = DnSlice{{d.buf[0] + q0 * d.step, d.buf[1] + q0 * d.step}, (q1 - q0) * d.step * 4, 0};
                }
                for (int i = 0; i < (end - first) * (S / seqs) && fits; ++i) {
                    const int n_e = P.first_edge[v + 1] - P.first_edge[v];
                    if (n_terms + 2 * n_e > kDnMaxTerms) { fits = false; break; }
                    DnUnit u{};
                    u.row0 = (first + i % (end - first)) * 8;
                    u.nrows = std::min(8, quads - u.row0);
                    u.first = (int16_t)(i / (end - first) * seqs);
                    u.term0 = n_terms;
                    u.n_terms = n_e;
                    u.bias_off = d.bias_off;
                    u.Cpad = d.step;
                    u.C = d.C;
                    u.flags = (d.act == 1 ? 1 : 0) | (d.is_output ? 2 : 0) | 4;
                    u.buf[0] = d.buf[0];
                    u.buf[1] = d.buf[1];
                    u.channels = (int16_t)g->nodes[v].d.c;
                    u.width = (int16_t)g->nodes[v].d.w;
                    long long steps = 0;
                    for (int e = P.first_edge[v]; e < P.first_edge[v + 1]; ++e) {
                        const SrHostEdge& he = *host_edge[e];
                        const DnNode& sn = P.nodes[P.edges[e].src];
                        const sr_node_desc& sd = g->nodes[he.d.src].d;
                        DnTerm& tm = h.terms[n_terms++];
                        tm.w_off = E->w_off[r][e];
                        tm.Kpad = he.k_eff | he.stride_eff << 8 | he.pad_eff << 16;
                        tm.xp = sn.seq;
                        tm.R = P.edges[e].R;
                        tm.n_buf = (sn.is_input ? 3 : 2) | sn.step << 8;
                        for (int q = 0; q < 3; ++q) tm.buf[q] = sn.buf[q < (tm.n_buf & 0xFF) ? q : 0];
                        DnConv cv{};
                        cv.Hs = sd.h; cv.Ws = sd.w; cv.Cs = sd.c;
                        std::memcpy(&h.terms[n_terms++], &cv, sizeof(cv));
                        steps += he.K * (sd.c % 4 == 0 ? 1 : 2);
                    }
                    lv.push_back({steps * 16 + 256, u});
                }
                for (int row = lo; row < hi && fits; row += kDnRows) {
                    const int nr = std::min(kDnRows, hi - row), n_e = P.first_edge[v + 1] - P.first_edge[v];
                    if (n_terms + n_e > kDnMaxTerms) { fits = false; break; }
                    DnUnit u{};
                    u.nrows = nr;
                    u.row0 = row;
                    u.term0 = n_terms;
                    u.n_terms = n_e;
                    u.bias_off = d.bias_off;
                    u.Cpad = d.Cpad;
                    u.C = d.C;
                    u.flags = (d.act == 1 ? 1 : 0) | (d.is_output ? 2 : 0);
                    u.buf[0] = d.buf[0];
                    u.buf[1] = d.buf[1];
                    for (int e = P.first_edge[v]; e < P.first_edge[v + 1]; ++e) {
                        const DnNode& sn = P.nodes[P.edges[e].src];
                        DnTerm& tm = h.terms[n_terms++];
                        tm.w_off = E->w_off[r][e] + (row - lo) * P.edges[e].Kpad;
                        tm.Kpad = P.edges[e].Kpad;
                        tm.xp = sn.seq;
                        tm.R = P.edges[e].R;
                        tm.n_buf = (sn.is_input ? 3 : 2) | sn.step << 8;
                        for (int i = 0; i < 3; ++i) tm.buf[i] = sn.buf[i < (tm.n_buf & 0xFF) ? i : 0];
                    }
                    lv.push_back({K * (4 + (nr > 2 ? 4 : 2)) + 256, u});     // loads per step + reduction and stores
                }
            }
            if (!fits) break;
            std::stable_sort(lv.begin(), lv.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
            std::vector<std::vector<DnUnit>> of_warp(kDnWarps);
            std::vector<long long> load(kDnWarps, 0);
            for (auto& u : lv) {
                // a warp issues through scheduler (warp % 4): the least loaded scheduler first, then its least loaded warp
                long long sched[4] = {0, 0, 0, 0};
                for (int w = 0; w < kDnWarps; ++w) sched[w & 3] += load[w];
                int w = 0;
                for (int c = 1; c < kDnWarps; ++c)
                    if (sched[c & 3] < sched[w & 3] || (sched[c & 3] == sched[w & 3] && load[c] < load[w])) w = c;
                of_warp[w].push_back(u.second);
                load[w] += u.first;
            }
            size_t rounds = 0;
            for (auto& q : of_warp) rounds = std::max(rounds, q.size());
            if (n_units + (int)rounds * kDnWarps > kDnMaxUnits) { fits = false; break; }
            for (size_t i = 0; i < rounds; ++i)
                for (int w = 0; w < kDnWarps; ++w) h.units[n_units++] = i < of_warp[w].size() ? of_warp[w][i] : DnUnit{};
            h.level_begin[l] = n_units;
            if (l == 1) {
                // warps without a unit in the first level fetch the input frames, if there are at least two of them
                int idle_warps = 0;
                for (int w = 0; w < kDnWarps; ++w)
                    if (of_warp[w].empty()) h.fetch_mask |= 1 << w;
                for (int w = 0; w < kDnWarps; ++w) idle_warps += (h.fetch_mask >> w) & 1;
                if (idle_warps < 2) h.fetch_mask = (1 << kDnWarps) - 1;
            }
        }
        for (int l = P.n_levels + 1; l <= kDnMaxLevels; ++l) h.level_begin[l] = n_units;
        for (int l = P.n_levels; l <= kDnMaxLevels; ++l) h.first_slice[l] = n_slices;
        h.n_units = n_units;
        h.idle = 1;
        for (int u = 0; u < n_units; ++u)
            if (h.units[u].nrows > 0) h.idle = 0;
        P.n_idle += h.idle;
        if (!fits) {
            delete E;
            return nullptr;
        }
    }
    return E;
}

}  // namespace

void sr_dn_destroy(sr_graph* g)
{
    if (DnEngine* E = dn_of(g))
        for (cudaEvent_t e : E->ev) cudaEventDestroy(e);
    delete dn_of(g);
    g->dn = nullptr;
}

bool sr_dn_available(const sr_graph* g) { return g->dn != nullptr; }
bool sr_dn_one_wave(const sr_graph* g) { return g->dn != nullptr && dn_of(g)->one_wave; }

void sr_dn_describe(const sr_graph* g, int* cluster_size, int* smem_bytes)
{
    const DnEngine* E = dn_of(g);
    *cluster_size = E ? E->cluster : 0;
    *smem_bytes = E ? E->smem_bytes : 0;
}

// The engine applies to graphs whose edges are dense, or convolutions of a quarter of a million multiply-adds per sample at most, small enough
// for the shared memory of a cluster.  Rows of every dense node are split evenly over the ranks.
sr_status sr_dn_plan(sr_graph* g, size_t& offset)
{
    sr_dn_destroy(g);
    if (!g->opt_resident || g->opt_engine != 0) return SR_OK;
    const int n_nodes = (int)g->nodes.size(), n_edges = (int)g->edges.size();
    if (n_nodes > kDnMaxNodes || n_edges > kDnMaxEdges || (int)g->groups.size() > kDnMaxLevels || g->groups.empty()) return SR_OK;
    if ((int)g->input_nodes.size() > SR_MAX_INPUTS) return SR_OK;
    // (the other resident engine's, where it applies)
    if (sr_rs_available(g)) return SR_OK;
    double work = 0;                                         // of the convolutions
    for (int v = 0; v < n_nodes; ++v) {
        const SrHostNode& n = g->nodes[v];
        if ((double)n.d.h * n.d.w * n.d.c > kDnSmemMax / 4) return SR_OK;
        if (n.is_input && dn_values(g, v) % 4 != 0) return SR_OK;
        if (dn_is_conv(g, v) && (n.d.c % 4 != 0 || n.d.c > 1024 || n.d.w > 1024)) return SR_OK;
    }
    for (const SrHostEdge& e : g->edges) {
        const sr_node_desc &s = g->nodes[e.d.src].d, &t = g->nodes[e.d.tgt].d;
        if (e.d.kind == SR_EDGE_CONV) {
            if (e.k_eff > 32 || e.stride_eff > 255 || e.pad_eff > 255) return SR_OK;
            work += (double)e.K * t.h * t.w * t.c;
        } else if (e.d.kind == SR_EDGE_MEAN_DENSE && s.h * s.w != 1) {
            return SR_OK;
        }
    }
    if (work > kDnConvWork) return SR_OK;
    // With one level per frame (the streaming rollout) a frame is one round of work units and one exchange: sixteen CTAs (a
    // non-portable cluster size) halve the units of each CTA, while with several levels per frame the costlier exchange of the
    // larger cluster outweighs that.  Measured on the 784-128-128-10 network, four clusters of two sequences, per frame: streaming
    // 1.45 us with sixteen, 2.19 with eight; sequential 3.4 and 3.3.  The device holds fewer than half as many of the larger
    // clusters (7 against 15), and a second wave costs more than they win (64 sequences, 64 frames: 342 us against 254), so they
    // are used only where all of a run go out at once.
    DnEngine* E = nullptr;
    if (g->groups.size() == 1) {
        E = dn_build(g, kDnMaxCluster, kDnMaxSamples);
        if (E && (g->batch + kDnMaxSamples - 1) / kDnMaxSamples > dn_clusters_held(g, kDnMaxCluster, kDnMaxSamples, E->smem_bytes)) {
            delete E;
            E = nullptr;
        }
    }
    if (!E) E = dn_build(g, 8, kDnMaxSamples);
    // Fewer sequences per cluster shorten a frame, because the loads of the states shrink with them: per frame of one wave of that
    // network 1.45, 1.87 and 2.50 us with two, four and eight sequences and sixteen CTAs, 2.19, 2.79 and 3.68 with eight CTAs
    // (sequential 3.3, 4.2, 5.4).  The split whose waves end first by these ratios is taken.  (They are that network's.  Networks of
    // 64- and 256-wide layers at 1 to 512 sequences were faster by this rule than with eight sequences per cluster throughout.)
    if (E) {
        const int cl = E->cluster;
        double best = 0.0;
        int best_waves = 0;
        for (int S = kDnMaxSamples; S >= 2; S /= 2) {
            DnEngine* F = S == E->samples ? E : dn_build(g, cl, S);       // (the first is the one there is)
            if (!F) continue;
            const int clusters = (g->batch + S - 1) / S, held = std::max(dn_clusters_held(g, cl, S, F->smem_bytes), 1);
            const int waves = (clusters + held - 1) / held;
            const double cost = waves * (S == 8 ? 1.0 : S == 4 ? 0.76 : 0.6);
            if (best_waves == 0 || cost < best) {
                best = cost;
                best_waves = waves;
                if (F != E) delete E;
                E = F;
            } else {
                delete F;
            }
        }
        E->one_wave = best_waves == 1;
        // A frame of a convolutional network takes the launch path little longer for many sequences than for one, and this engine as much
        // longer as there are waves.  So it is for what goes out at once, in fp32 also for two waves of frames of several levels (launches);
        // in bf16, where the tensor cores do the convolutions, frames of one level only with up to four sequences per cluster.  us per frame
        // launched / resident (MNIST network SR; 14 x 14 x 4 to a recurrent 7 x 7 x 16):
        //   fp32, one level, 100 samples (one wave) 12.1 / 8.1; 9.4 / 6.6 at 64; 128 (two) 13.3 / 15.7; 10.7 / 13.0; 256 (three) 20.1 / 23.5; 14.2 / 19.4
        //   fp32, sequential, 100 19.2 / 9.3; 14.4 / 7.5; 128 19.8 / 18.0; 15.7 / 14.7; 256 25.8 / 27.0; 19.1 / 22.1
        //   bf16, one level, 8 7.1 / 4.2; 64 (eight sequences a cluster) 8.4 / 8.9; sequential, 64 13.0 / 12.7; 12.5 / 11.7; 128 (two) 19.8 / 26.4
        // (Of 48 sizes and networks the former rule, any number of waves in fp32, had 13 up to 49 % slower than launches; this one
        // has a 14 x 14 x 4 to 7 x 7 x 8 at 128 samples launched, 10.8, that the engine would take 8.5 for, and four up to 6 %.)
        const int most_waves = g->dtype == SR_DTYPE_F32 && g->groups.size() > 1 ? 2 : 1;
        if (E && work > 0 && (best_waves > most_waves || (g->dtype == SR_DTYPE_BF16 && g->groups.size() == 1 && E->samples > 4))) {
            delete E;
            E = nullptr;
        }
    }
    // A graph that fits the built-in workspace without this engine keeps fitting (fp32 networks of dense edges only have always had
    // its tables counted).
    if (E && (work > 0 || g->dtype == SR_DTYPE_BF16) && offset - g->r_items.bytes <= (size_t)SR_STATIC_WORKSPACE_BYTES &&
        offset - g->r_items.bytes + (size_t)E->cluster * E->P.blob_bytes + 256 > (size_t)SR_STATIC_WORKSPACE_BYTES) {
        delete E;
        E = nullptr;
    }
    if (!E) return SR_OK;
    const int CL = E->cluster;
    DnParams& P = E->P;
    E->r_blobs.offset = offset;
    E->r_blobs.bytes = (size_t)CL * P.blob_bytes;
    offset = sr_align_up(offset + E->r_blobs.bytes, 256);
    g->dn = E;
    // the per-rank table images; they go to the workspace when one is bound
    g->dn_headers.assign((size_t)CL * sizeof(DnBlobHdr), 0);
    for (int r = 0; r < CL; ++r) std::memcpy(g->dn_headers.data() + (size_t)r * sizeof(DnBlobHdr), &E->hdrs[r], sizeof(DnBlobHdr));
    return SR_OK;
}

sr_status sr_dn_bind(sr_graph* g)
{
    DnEngine* E = dn_of(g);
    if (!E) return SR_OK;
    DnParams& P = E->P;
    const int CL = E->cluster;
    char* ws = g->ws;
    P.blobs = reinterpret_cast<const unsigned char*>(ws + E->r_blobs.offset);
    for (int v = 0; v < P.n_nodes; ++v) {
        const SrHostNode& n = g->nodes[v];
        P.nodes[v].gstate[0] = ws + n.state[0].offset;
        P.nodes[v].gstate[1] = ws + n.state[1].offset;
        P.nodes[v].bias = reinterpret_cast<const float*>(ws + n.bias.offset);
    }
    // the workspace was zeroed by the caller of bind: weights start at zero, headers go in now
    if (cudaMemcpy2D(ws + E->r_blobs.offset, P.blob_bytes, g->dn_headers.data(), sizeof(DnBlobHdr), sizeof(DnBlobHdr), CL, cudaMemcpyHostToDevice) != cudaSuccess)
        return SR_ERR_CUDA;
    return SR_OK;
}

sr_status sr_dn_set_weights(sr_graph* g, int edge, const float* w)
{
    DnEngine* E = dn_of(g);
    if (!E) return SR_OK;
    const DnParams& P = E->P;
    const int CL = E->cluster;
    const int e = E->edge_of_host[edge];
    const SrHostEdge& he = g->edges[edge];
    const int v = he.d.tgt, K = he.K, Kpad = P.edges[e].Kpad;
    if (dn_is_conv(g, v)) {                                  // [C_out][K] -> [K][C_out], the same for every rank
        const int C = g->nodes[v].d.c;
        const size_t n = (size_t)K * C;
        std::vector<float> h(n * CL);
        for (int co = 0; co < C; ++co)
            for (int kk = 0; kk < K; ++kk) h[(size_t)kk * C + co] = w[(size_t)co * K + kk];
        for (int r = 1; r < CL; ++r) std::copy_n(h.begin(), n, h.begin() + n * r);
        // one copy for all ranks where the edge lies at the same place in each
        bool same = true;
        for (int r = 1; r < CL; ++r) same = same && E->w_off[r][e] == E->w_off[0][e];
        for (int r = 0; r < (same ? 1 : CL); ++r) {
            char* dst = g->ws + E->r_blobs.offset + (size_t)r * P.blob_bytes + sizeof(DnBlobHdr) + (size_t)E->w_off[r][e] * 4;
            if (cudaMemcpy2D(dst, P.blob_bytes, h.data(), n * 4, n * 4, same ? CL : 1, cudaMemcpyHostToDevice) != cudaSuccess) return SR_ERR_CUDA;
        }
        return SR_OK;
    }
    const int rows = dn_values(g, v);
    std::vector<float> h((size_t)rows * Kpad, 0.f);
    for (int row = 0; row < rows; ++row) std::memcpy(&h[(size_t)row * Kpad], w + (size_t)row * K, sizeof(float) * K);
    const int* lo = &E->row_lo[(size_t)v * (CL + 1)];
    bool same = true;
    for (int r = 1; r < CL; ++r) same = same && E->w_off[r][e] == E->w_off[0][e] && lo[r + 1] - lo[r] == lo[1] - lo[0];
    for (int r = 0; r < (same ? 1 : CL); ++r) {
        const size_t bytes = (size_t)(lo[r + 1] - lo[r]) * Kpad * sizeof(float);
        if (bytes == 0) continue;
        char* dst = g->ws + E->r_blobs.offset + (size_t)r * P.blob_bytes + sizeof(DnBlobHdr) + (size_t)E->w_off[r][e] * 4;
        if (cudaMemcpy2D(dst, P.blob_bytes, &h[(size_t)lo[r] * Kpad], bytes, bytes, same ? CL : 1, cudaMemcpyHostToDevice) != cudaSuccess) return SR_ERR_CUDA;
    }
    return SR_OK;
}

sr_status sr_dn_launch(sr_graph* g, int T, const SrFrameCtl& init, cudaStream_t s)
{
    DnEngine* E = dn_of(g);
    if (!E) return SR_ERR_STATE;
    const int CL = E->cluster;
    const int S = E->samples;
    auto kernel = dn_kernel_of(g, CL, S);
    if (!E->attr_set) {
        if (!dn_prepare(kernel, CL)) return SR_ERR_CUDA;
        E->attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((g->batch + S - 1) / S * CL));
    cfg.blockDim = dim3((unsigned)(kDnWarps * 32));
    cfg.dynamicSmemBytes = (size_t)E->smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool plain = cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
    bool timed = g->opt_time_tc != 0 && plain;
    cfg.numAttrs = plain && !timed ? 2 : 1;                   // may start early (see SrFollow)
    E->P.error = reinterpret_cast<int32_t*>(g->ws + g->r_flags.offset);
    E->P.wait_limit = (long long)std::max(1, g->opt_wait_ms) * 2000000LL;
    if (timed && E->ev_used + 2 > E->ev.size()) {
        if (E->ev.size() >= 4096) timed = false;
        for (int i = 0; timed && i < 2; ++i) {
            cudaEvent_t e = nullptr;
            if (cudaEventCreate(&e) != cudaSuccess) timed = false;
            else E->ev.push_back(e);
        }
        if (E->ev_used + 2 > E->ev.size()) timed = false;
    }
    if (timed) cudaEventRecord(E->ev[E->ev_used], s);
    if (cudaLaunchKernelEx(&cfg, kernel, E->P, init, T) != cudaSuccess) return SR_ERR_CUDA;
    if (timed) {
        cudaEventRecord(E->ev[E->ev_used + 1], s);
        E->ev_used += 2;
    }
    return SR_OK;
}

sr_status sr_dn_timing(sr_graph* g, double* ms, long long* launches)
{
    DnEngine* E = dn_of(g);
    *ms = 0.0;
    *launches = 0;
    if (!E) return SR_OK;
    for (size_t i = 0; i + 1 < E->ev_used; i += 2) {
        if (cudaEventSynchronize(E->ev[i + 1]) != cudaSuccess) return SR_ERR_CUDA;
        float t = 0.f;
        if (cudaEventElapsedTime(&t, E->ev[i], E->ev[i + 1]) != cudaSuccess) return SR_ERR_CUDA;
        *ms += t;
        *launches += 1;
    }
    E->ev_used = 0;
    return SR_OK;
}
