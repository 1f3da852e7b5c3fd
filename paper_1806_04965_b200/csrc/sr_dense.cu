// Dense resident engine: the frame update  x_v = sigma(b_v + sum_e W_e x_src(e))  (paper Sec. A1.2) of a small network
// whose edges are all dense, in fp32, for all T frames of a run in ONE launch.
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
// The sums run in a fixed order, so results are reproducible bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "sr_dense.h"

namespace {

constexpr int kDnMaxNodes = 16, kDnMaxEdges = 32, kDnMaxLevels = 16, kDnMaxUnits = 128;
constexpr int kDnMaxSamples = 8;       // sequences per cluster, most
constexpr int kDnMoreThanHalf = 120 * 1024;   // of an SM's shared memory, bytes
constexpr int kDnMaxCluster = 16;      // CTAs per cluster: 8, or 16 (a non-portable size) for rollouts with one level per frame
constexpr int kDnWarps = 8;            // 256 threads: a work unit keeps 64 registers of packed accumulators and its operands
constexpr int kDnRows = 4;             // output rows per work unit
constexpr int kDnSmemMax = 220 * 1024;

struct DnNode {
    float* gstate[2];                  // state buffers in global memory, [B][C], by frame parity
    const float* bias;
    int32_t C, Cpad, act, is_input, input_slot, is_output;
    int32_t buf[3];                    // float offsets of the shared-memory state buffers: frame f lives in buf[f % 3] (input
                                       // nodes) or buf[f & 1] (others)
    int32_t bias_off;                  // float offset of the node's bias copy in shared memory
};

struct DnEdge { int32_t src, tgt, R, Kpad; };

// One incoming edge of a work unit, ready to use (32 bytes): where the unit's weight rows start (floats from the
// rank's first weight), the padded reduction length = row pitch of the weights, the row pitch of the source state,
// the frames the edge looks back (Eq. 2), and the source's shared-memory buffers (three for an input node).
struct DnTerm { int32_t w_off, Kpad, xp, R, n_buf, buf[3]; };
static_assert(sizeof(DnTerm) == 32, "read as two 16-byte words");

// Up to four rows of a node with everything a warp needs (48 bytes).  nrows = 0: no unit (a gap in a warp's list).
struct DnUnit {
    int32_t nrows, row0, term0, n_terms;
    int32_t bias_off, Cpad, C, flags;                        // flags: 1 = ReLU, 2 = the output node
    int32_t buf[2], pad_[2];                                 // the node's two shared-memory buffers by frame parity
};
static_assert(sizeof(DnUnit) == 48, "read as three 16-byte words");

constexpr int kDnMaxTerms = 256;

struct DnBlobHdr {                     // head of a rank's blob; the rank's weight slices follow
    int32_t n_units, fetch_mask, idle, pad_;                 // fetch_mask: warps that fetch input frames; idle: the rank has no unit
    int32_t level_begin[kDnMaxLevels + 1];                   // units of level l: [level_begin[l-1], level_begin[l]); warp w
    int32_t pad2_[3];                                        // takes entries w, w + kDnWarps, ... of a level
    DnUnit units[kDnMaxUnits];
    DnTerm terms[kDnMaxTerms];
};
static_assert(sizeof(DnBlobHdr) % 16 == 0, "the weights that follow are read with 16-byte loads");
static_assert(offsetof(DnBlobHdr, units) % 16 == 0 && offsetof(DnBlobHdr, terms) % 16 == 0, "tables are read with 16-byte loads");

struct DnParams {
    int32_t n_nodes, n_edges, n_levels, B;
    int32_t blob_bytes, hdr_floats, total_floats, n_idle;    // n_idle: ranks without a unit
    int32_t level_bytes[kDnMaxLevels];                       // bytes that a level's new states are, in one CTA's copy
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
// Bounded wait for a phase of a barrier that other CTAs' stores complete.
__device__ __forceinline__ bool dn_wait(uint32_t bar, uint32_t parity, volatile int* gave_up, long long limit)
{
    long long t0 = 0;
    for (int i = 0;; ++i) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
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

// One work unit: up to R rows of a node for the S sequences of the cluster, relative frame f -> f + 1.
// The loads of a reduction step are issued ahead of the multiply-adds that use them: the weights and the first four
// sequences of step i + 1 while the last four sequences of step i are still being multiplied.
template <int R, int CL, int S>
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
        const int bi = tm.n_buf == 3 ? sf % 3 : (sf & 1);
        const float* xs = dn_mem + (bi == 0 ? tm.buf[0] : (bi == 1 ? tm.buf[1] : tm.buf[2])) + lane * 4;
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
        for (int k = 0; k < n_k; k += 128) {
            ulonglong2 an[R], xb[G];
            const int kn = k + 128 < n_k ? k + 128 : k;               // the last step re-reads itself (no branch)
            if (S > G) {
#pragma unroll
                for (int b = 0; b < G; ++b) xb[b] = *reinterpret_cast<const ulonglong2*>(xs + (b + G) * xp + k);
                dn_fma<R, S, G>(acc2, a, xa, 0);
#pragma unroll
                for (int r = 0; r < R; ++r) an[r] = *reinterpret_cast<const ulonglong2*>(w0 + ro[r] + kn);
#pragma unroll
                for (int b = 0; b < G; ++b) xa[b] = *reinterpret_cast<const ulonglong2*>(xs + b * xp + kn);
                dn_fma<R, S, G>(acc2, a, xb, S - G);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) an[r] = *reinterpret_cast<const ulonglong2*>(w0 + ro[r] + kn);
#pragma unroll
                for (int b = 0; b < G; ++b) xb[b] = *reinterpret_cast<const ulonglong2*>(xs + b * xp + kn);
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
    const uint32_t cell = dn_smem(dn_mem + (((f + 1) & 1) ? un.buf[1] : un.buf[0]) + b * un.Cpad + un.row0);
    constexpr uint32_t kPerLane = CL > kLanes ? CL / kLanes : 1;      // ranks that each of them serves
    const uint32_t q = (uint32_t)(lane % kLanes) * kPerLane;
    if (q >= CL) {
        // (more lanes than ranks: nothing to send)
    } else if (R == 4 && un.nrows == 4 && (un.row0 & 3) == 0) {
        const float z4[4] = {z[0], z[1], z[2 % R], z[3 % R]};
#pragma unroll
        for (uint32_t i = 0; i < kPerLane; ++i) dn_st_async4(cell, bar, q + i, z4);
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < un.nrows) {
#pragma unroll
                for (uint32_t i = 0; i < kPerLane; ++i) dn_st_async(cell + 4 * r, bar, q + i, z[r]);
            }
    }
    if ((un.flags & 2) && init.out_base && lane % kLanes == 0 && b < nb) {
        float* o = init.out_base + (run0 + f) * init.out_stride + (long long)(b0 + b) * un.C + un.row0;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < un.nrows) o[r] = z[r];
    }
}

template <int CL, int S>
__global__ void __launch_bounds__(kDnWarps * 32, 1)
sr_dense_kernel(const DnParams P, const SrFrameCtl init, int T)
{
    extern __shared__ __align__(16) float dn_mem[];
    // the input nodes as the fetching warps need them: first float of this cluster's sequences in the caller's frame 0
    // of the run, floats from one frame to the next, floats per frame, the three shared-memory buffers
    __shared__ const float* in_src[SR_MAX_INPUTS];
    __shared__ long long in_step[SR_MAX_INPUTS];
    __shared__ int in_len[SR_MAX_INPUTS], in_buf[SR_MAX_INPUTS][3], n_in;
    __shared__ uint64_t bars[kDnMaxLevels][2];               // per level and frame parity: the level's new states have arrived
    __shared__ int gave_up;
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
    }
    const long long t0 = init.t, run0 = init.run_t;
    if (tid == 0) {
        gave_up = 0;
        int n = 0;
        for (int v = 0; v < P.n_nodes; ++v) {
            const DnNode& nd = P.nodes[v];
            if (!nd.is_input) continue;
            in_src[n] = reinterpret_cast<const float*>(static_cast<const char*>(init.in_base[nd.input_slot]) + run0 * init.in_stride_bytes[nd.input_slot]) + (size_t)b0 * nd.C;
            in_step[n] = init.in_stride_bytes[nd.input_slot] / 4;
            in_len[n] = nb * nd.C;                           // input nodes have Cpad == C
            for (int i = 0; i < 3; ++i) in_buf[n][i] = nd.buf[i];
            ++n;
        }
        n_in = n;
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (tid < 2 * P.n_levels) {
        // one arrival announces the bytes; in the last level every fetching thread arrives when its copies have landed, and
        // every rank that sends no states does once per frame
        const int l = tid >> 1, n_arrive = 1 + (l == P.n_levels - 1 ? 32 * __popc(H->fetch_mask) + P.n_idle : 0);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(dn_smem(&bars[l][tid & 1])), "r"(n_arrive) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // (Weights and tables do not depend on the kernel before this one; states and input frames do.)
    sr_wait_for_predecessor();
    // frame t of every node from the state buffers in global memory (relative frame 0)
    const int par0 = (int)(t0 & 1);
    for (int v = 0; v < P.n_nodes; ++v) {
        const DnNode& nd = P.nodes[v];
        const float* gsrc = nd.gstate[par0] + (size_t)b0 * nd.C;
        float* dst = dn_mem + nd.buf[0];
        if (nd.Cpad == nd.C) dn_fetch(dst, gsrc, nb * nd.C, tid, nthr);                  // rows are contiguous: 16-byte copies
        else
            for (int i = tid; i < nb * nd.C; i += nthr) dst[(i / nd.C) * nd.Cpad + (i % nd.C)] = gsrc[i];
        if (!nd.is_input)
            for (int i = tid; i < nd.C; i += nthr) dn_mem[nd.bias_off + i] = nd.bias[i];
    }
    // Input frame k of the run (relative frame k) -> buffer k % 3, by the warps of fetch_mask.
    const int f_nthr = 32 * __popc(H->fetch_mask);
    const int f_tid = (H->fetch_mask >> warp) & 1 ? 32 * __popc(H->fetch_mask & ((1 << warp) - 1)) + lane : -1;
    auto fetch_inputs = [&](int k) {
        if (f_tid < 0) return;
        for (int i = 0; i < n_in; ++i) dn_fetch(dn_mem + in_buf[i][k % 3], in_src[i] + (k - 1) * in_step[i], in_len[i], f_tid, f_nthr);
    };
    fetch_inputs(1);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    dn_cluster_sync();                                       // every CTA of the cluster has its buffers in place before remote writes start

    for (int f = 0; f < T && !*(volatile int*)&gave_up; ++f) {                // relative frame f -> f + 1
        // the input frame after the next one is on its way during this update; it has landed when the last level's barrier
        // completes
        const int par = (f + 1) & 1;
        const uint32_t phase = (uint32_t)(f >> 1) & 1u;
        if (f + 1 < T) fetch_inputs(f + 2);
        if (f_tid >= 0) asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(dn_smem(&bars[P.n_levels - 1][par])) : "memory");
        for (int l = 1; l <= P.n_levels; ++l) {
            const uint32_t bar = dn_smem(&bars[l - 1][par]);
            if (tid == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(P.level_bytes[l - 1]) : "memory");
            // Nobody runs more than a frame ahead of a rank, because a level needs the states of every rank with a unit in it;
            // a rank without any says so instead.
            if (H->idle && l == P.n_levels && tid < CL)
                asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(dn_map_rank(bar, (uint32_t)tid)) : "memory");
            for (int u = H->level_begin[l - 1] + warp; u < H->level_begin[l]; u += kDnWarps) {
                const DnUnit un = H->units[u];
                if (un.nrows == 0) continue;
                if (un.nrows > 2) dn_unit<4, CL, S>(H, un, dn_mem, wsm, init, f, lane, b0, nb, run0, bar);
                else dn_unit<2, CL, S>(H, un, dn_mem, wsm, init, f, lane, b0, nb, run0, bar);
            }
            if (!dn_wait(bar, phase, &gave_up, P.wait_limit)) break;    // the level is complete in this CTA's copy
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (*(volatile int*)&gave_up) __nanosleep(100000);       // stores on their way to this CTA land before it leaves
    __syncwarp();
    dn_cluster_sync();                                       // no CTA leaves while another one may still store into it
    if (tid == 0 && gave_up) atomicExch(P.error, 1);

    // relative frame T back to the state buffers in global memory (parity of t + T); every rank holds a full copy and
    // writes its share of it
    {
        const int parT = (int)((t0 + T) & 1);
        const int gtid = (int)rank * nthr + tid, gthr = CL * nthr;
        for (int v = 0; v < P.n_nodes; ++v) {
            const DnNode& nd = P.nodes[v];
            const float* src = dn_mem + (nd.is_input ? nd.buf[T % 3] : nd.buf[T & 1]);
            float* gdst = nd.gstate[parT] + (size_t)b0 * nd.C;
            if (nd.Cpad == nd.C)
                for (int i = gtid * 4; i < nb * nd.C; i += gthr * 4) *reinterpret_cast<float4*>(gdst + i) = *reinterpret_cast<const float4*>(src + i);
            else
                for (int i = gtid; i < nb * nd.C; i += gthr) gdst[i] = src[(i / nd.C) * nd.Cpad + (i % nd.C)];
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

DnKernel dn_kernel_of(int cluster, int samples)
{
    if (cluster == 16) return samples == 8 ? sr_dense_kernel<16, 8> : samples == 4 ? sr_dense_kernel<16, 4> : sr_dense_kernel<16, 2>;
    return samples == 8 ? sr_dense_kernel<8, 8> : samples == 4 ? sr_dense_kernel<8, 4> : sr_dense_kernel<8, 2>;
}

// Clusters of this size and shared-memory footprint that the device holds at once with one CTA per SM (0: none): two CTAs on an SM
// share its shared-memory pipe, so a second one there gains little over a second wave.
int dn_clusters_held(int cluster, int samples, int smem_bytes)
{
    DnKernel kernel = dn_kernel_of(cluster, samples);
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
    for (int v = 0; v < n_nodes; ++v) {
        P.first_edge[v] = pos;
        for (int e : g->nodes[v].in_edges) {
            const SrHostEdge& he = g->edges[e];
            const int Kpad = (g->nodes[he.d.src].d.c + 3) / 4 * 4;
            P.edges[pos] = DnEdge{he.d.src, he.d.tgt, he.R, Kpad};
            E->edge_of_host[e] = pos++;
        }
    }
    P.first_edge[n_nodes] = pos;
    // row slices and weight offsets per rank
    E->row_lo.assign((size_t)n_nodes * (CL + 1), 0);
    E->w_off.assign(CL, std::vector<int>(kDnMaxEdges, 0));
    int max_w = 0;
    for (int v = 0; v < n_nodes; ++v)
        for (int r = 0; r <= CL; ++r) E->row_lo[(size_t)v * (CL + 1) + r] = g->nodes[v].d.c * r / CL;
    for (int r = 0; r < CL; ++r) {
        int w = 0;
        for (int e = 0; e < n_edges; ++e) {
            const int v = P.edges[e].tgt;
            const int rows = E->row_lo[(size_t)v * (CL + 1) + r + 1] - E->row_lo[(size_t)v * (CL + 1) + r];
            E->w_off[r][e] = w;
            w += rows * P.edges[e].Kpad;
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
        d.C = n.d.c;
        d.Cpad = (n.d.c + 3) / 4 * 4;
        d.act = n.d.act;
        d.is_input = n.is_input ? 1 : 0;
        d.input_slot = n.input_slot;
        d.is_output = v == g->info.output_node ? 1 : 0;
        for (int i = 0; i < (n.is_input ? 3 : 2); ++i) {
            d.buf[i] = off;
            off += S * d.Cpad;
        }
        d.bias_off = off;
        if (!n.is_input) off += d.Cpad;
    }
    P.total_floats = off;
    for (int l = 0; l < P.n_levels; ++l) {
        P.level_bytes[l] = 0;
        for (int v : g->groups[l]) P.level_bytes[l] += g->nodes[v].d.c * S * 4;
    }
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
        int n_units = 0, n_terms = 0;
        bool fits = true;
        for (int l = 1; l <= P.n_levels && fits; ++l) {
            std::vector<std::pair<long long, DnUnit>> lv;
            for (int v : g->groups[l - 1]) {
                const DnNode& d = P.nodes[v];
                long long K = 0;
                for (int e = P.first_edge[v]; e < P.first_edge[v + 1]; ++e) K += P.edges[e].Kpad;
                const int lo = E->row_lo[(size_t)v * (CL + 1) + r], hi = E->row_lo[(size_t)v * (CL + 1) + r + 1];
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
                        tm.xp = sn.Cpad;
                        tm.R = P.edges[e].R;
                        tm.n_buf = sn.is_input ? 3 : 2;
                        for (int i = 0; i < 3; ++i) tm.buf[i] = sn.buf[i < tm.n_buf ? i : 0];
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

// The engine applies to fp32 graphs in which every node is a vector (h = w = 1) and every edge dense, small enough for
// the shared memory of a cluster.  Rows of every node are split evenly over the ranks.
sr_status sr_dn_plan(sr_graph* g, size_t& offset)
{
    sr_dn_destroy(g);
    if (!g->opt_resident || g->opt_engine != 0 || g->dtype != SR_DTYPE_F32) return SR_OK;
    const int n_nodes = (int)g->nodes.size(), n_edges = (int)g->edges.size();
    if (n_nodes > kDnMaxNodes || n_edges > kDnMaxEdges || (int)g->groups.size() > kDnMaxLevels || g->groups.empty()) return SR_OK;
    if ((int)g->input_nodes.size() > SR_MAX_INPUTS) return SR_OK;
    for (const SrHostNode& n : g->nodes) {
        if (n.d.h != 1 || n.d.w != 1) return SR_OK;
        if (n.is_input && n.d.c % 4 != 0) return SR_OK;
    }
    for (const SrHostEdge& e : g->edges)
        if (e.d.kind == SR_EDGE_CONV) return SR_OK;
    // With one level per frame (the streaming rollout) a frame is one round of work units and one exchange: sixteen CTAs (a
    // non-portable cluster size) halve the units of each CTA, while with several levels per frame the costlier exchange of the
    // larger cluster outweighs that.  Measured on the 784-128-128-10 network, four clusters of two sequences, per frame: streaming
    // 1.45 us with sixteen, 2.19 with eight; sequential 3.4 and 3.3.  The device holds fewer than half as many of the larger
    // clusters (7 against 15), and a second wave costs more than they win (64 sequences, 64 frames: 342 us against 254), so they
    // are used only where all of a run go out at once.
    DnEngine* E = nullptr;
    if (g->groups.size() == 1) {
        E = dn_build(g, kDnMaxCluster, kDnMaxSamples);
        if (E && (g->batch + kDnMaxSamples - 1) / kDnMaxSamples > dn_clusters_held(kDnMaxCluster, kDnMaxSamples, E->smem_bytes)) {
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
        int best_s = 0, best_waves = 0;
        for (int S = kDnMaxSamples; S >= 2; S /= 2) {
            DnEngine* F = S == kDnMaxSamples ? E : dn_build(g, cl, S);
            if (!F) continue;
            const int clusters = (g->batch + S - 1) / S, held = std::max(dn_clusters_held(cl, S, F->smem_bytes), 1);
            const int waves = (clusters + held - 1) / held;
            const double cost = waves * (S == 8 ? 1.0 : S == 4 ? 0.76 : 0.6);
            if (F != E) delete F;
            if (best_s == 0 || cost < best) { best = cost; best_s = S; best_waves = waves; }
        }
        if (best_s != E->samples) {
            delete E;
            E = dn_build(g, cl, best_s);
        }
        if (E) E->one_wave = best_waves == 1;
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
        P.nodes[v].gstate[0] = reinterpret_cast<float*>(ws + n.state[0].offset);
        P.nodes[v].gstate[1] = reinterpret_cast<float*>(ws + n.state[1].offset);
        P.nodes[v].bias = reinterpret_cast<const float*>(ws + n.bias.offset);
    }
    // the workspace was zeroed by the caller of bind: weights start at zero, headers go in now
    for (int r = 0; r < CL; ++r)
        if (cudaMemcpy(ws + E->r_blobs.offset + (size_t)r * P.blob_bytes, g->dn_headers.data() + (size_t)r * sizeof(DnBlobHdr),
                       sizeof(DnBlobHdr), cudaMemcpyHostToDevice) != cudaSuccess)
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
    for (int r = 0; r < CL; ++r) {
        const int lo = E->row_lo[(size_t)v * (CL + 1) + r], hi = E->row_lo[(size_t)v * (CL + 1) + r + 1];
        if (hi <= lo) continue;
        std::vector<float> h((size_t)(hi - lo) * Kpad, 0.f);
        for (int row = lo; row < hi; ++row)
            std::memcpy(&h[(size_t)(row - lo) * Kpad], w + (size_t)row * K, sizeof(float) * K);
        char* dst = g->ws + E->r_blobs.offset + (size_t)r * P.blob_bytes + sizeof(DnBlobHdr) + (size_t)E->w_off[r][e] * 4;
        if (cudaMemcpy(dst, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return SR_ERR_CUDA;
    }
    return SR_OK;
}

sr_status sr_dn_launch(sr_graph* g, int T, const SrFrameCtl& init, cudaStream_t s)
{
    DnEngine* E = dn_of(g);
    if (!E) return SR_ERR_STATE;
    const int CL = E->cluster;
    const int S = E->samples;
    auto kernel = dn_kernel_of(CL, S);
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
