// Tensor-core engine: the node update  x_v = sigma(b_v + sum_e f_e(theta_e, x_src(e)))  (paper Sec. A1.2)
// for all convolutional nodes of one launch group as ONE grouped implicit GEMM on tcgen05 / TMEM.
//
// The sum over the incoming edges of a node is one convolution over the concatenated sources (paper
// Sec. A notes the equivalence): the K loop of an output tile simply walks the K-blocks of every
// incoming edge, tap by tap, into one TMEM accumulator.
//
// GEMM shape.  D[c_out][pixel] = sum_k W[c_out][k] * X[pixel][k]: the weights are the M operand
// (128 rows per instruction, one tile per 128 output channels), the output pixels are the N operand.
// Measured on B200 (issued behind elect.sync), one tcgen05.mma of M = 128 costs 128 / 96 / 64 / 48 / 40 cycles at N = 256 /
// 192 / 128 / 64 / 32: N / 2, or (M + N) / 4 where that is more (the operands come out of shared memory at 128 bytes per
// cycle); copies into shared memory at up to 90 bytes per cycle and SM do not slow it down.
//
// Operands.  K-block = one filter tap x up to 64 input channels.  Activation tiles come straight from
// the NHWC state of the source node through 4-D TMA boxes (zero fill outside the image = zero
// padding); a stride-s edge reads one of s*s residue-class views of the source, so every tap is again
// a dense box.  The node's weight matrix [C_out][K] (K-major) keeps its columns in the order the K loop
// walks them, so that consecutive K-blocks of equal width are one 3-D tensor and a weight group (one slot of
// the weight ring) is ONE TMA copy.  Few-channel input edges (C_in = 1 or 3) are staged per frame into an im2col
// tensor with K padded to 16/32/64/128 so that they are ordinary K-blocks.
//
// Pixel tile.  A tile is tb samples x th rows x (8 * nl) columns; its nl "lanes" of 8 columns lie side by side in one
// activation box and in one accumulator of up to 256 TMEM columns, and share every weight block (nl MMAs per K = 16
// step).  Within a lane column n of the GEMM is pixel (b, r, x) with n = (b * (th + sep) + r) * 8 + x: the rows of the
// stacked box (sep = how far the taps that share a box are apart; columns with r >= th are never stored).  A K-major
// swizzled operand may start at any multiple of 128 bytes and its 8-row groups may be any multiple of 128 bytes apart,
// so ALL taps of an edge whose input pixels lie in the same residue class of the stride are windows of ONE box that
// start dy box rows and dx pixels further in: a 3 x 3 stride-1 edge loads one box per 64 channels for nine taps.  A node
// none of whose edges shares a box (1 x 1 filters, strides above the filter size) takes "flat" tiles of any width
// instead, whose pixels are consecutive.
//
// Work items.  An item is one pixel tile of one plan (a node, or up to four narrow nodes fused, see TcNode).  CTAs are
// persistent, one per SM.
//
// Warp roles in a CTA of 384 threads: warp 2 = keeper (finds the items, copies the K-loop tables of their nodes into shared
// memory ahead of time); warp 0 = weight producer (a ring of equal slots); warp 3 = activation producer (a ring of bytes:
// boxes differ in size); warp 1 = MMA issuer (owns TMEM; one host-made record per eight or so MMAs); warps 4..11 = epilogue
// (TMEM lane = output channel; bias, ReLU, bf16, NHWC stores in which a warp writes 32 consecutive channels of one pixel).
// Every wait is bounded; on expiry the kernel sets the graph's error word, waits for its own copies, frees
// TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <tuple>
#include <type_traits>
#include <vector>

#include "sr_tc.h"
#include "sr_tc_lists.h"

namespace {

constexpr int kMaxCols = 256;                         // TMEM columns of an accumulator = pixels of a tile, separators included
constexpr int kThreads = 384;
constexpr int kEpiWarps = 8;                          // warps 4..11
constexpr int kBoxes = 8;                             // activation boxes in flight
constexpr int kMaxW = 12;                             // weight ring depth (one weight group per slot)
constexpr int kItems = 8;                             // work items the keeper may be ahead of the epilogue
constexpr int kTables = 3;                            // node tables in shared memory
// Dynamic shared memory of a CTA.  With the 11 KiB of static shared memory this leaves about 12 KiB of the SM's 228 KiB
// free: the other kernels of a frame (input staging, dense heads: up to 7.4 KiB per block) run beside
// the persistent CTAs, and measured on B200 they queue behind them, frame after frame, once less than about 10 KiB of
// the SM's shared-memory partition is left (a 117 us frame then takes 170 us).
constexpr int kSmemBudget = 204 * 1024;
constexpr int kMaxNodeKb = 128;                       // K-blocks per node
constexpr int kMaxFused = 4;                          // nodes of a plan
// The most columns of a tile that are tried.  160: two 8 x 8 images with the gap between them (144 columns), which took either 256
// columns for three images or 64 for one.  Us per frame without / with it: ten-node network at 8 / 16 samples 18.6 / 17.0, 25.9 / 25.0,
// sequential at 20 / 32 / 128 105.9 / 97.8, 111.2 / 106.1, 197.5 / 186.5, six-node sequential at 256 212 / 203, hybrid at 20 samples 41.4 / 37.0.
constexpr int kTileCols[] = {256, 160, 128, 64};
constexpr int kVariants = sizeof(kTileCols) / sizeof(int);
constexpr int kMaxParts = 8;                          // parts of an item's reduction

// A run of equally wide K-blocks of a node's reduction as the weight producer sees it: n_groups weight groups (one copy
// and one ring slot each) of one or two blocks (see TcNode::pairs).
struct TcRun {
    uint16_t map1, map2;                // tensor maps: dims (channels of a block, output channels, blocks), box of one / two blocks
    uint16_t bytes16;                   // bytes of a block's weights / 16
    uint16_t n_groups;
    uint16_t blk0, pad_;                // the first of them
};
constexpr int kMaxRuns = 3;                           // block widths 64, 32, 16

// One activation box of a node's reduction (16 bytes).
struct TcAct {
    uint16_t x_map0, x_map1;// tensor map of the activation box for source frame parity 0 / 1
    uint16_t x_bytes16;     // (bytes of the activation box) / 16
    int8_t qx, qy;          // box origin relative to the tile origin (columns, rows)
    uint8_t c0_16;          // (first channel of the box) / 16
    uint8_t flags;          // 1: the edge reads frame t (R = 1), else frame t+1
    uint16_t ring_kb;       // KiB the box takes in the activation ring
    uint32_t pad_;
};
static_assert(sizeof(TcAct) == 16, "copied as one 16-byte word");

// One burst of MMAs as the issuer sees it (32 bytes): one or two weight slots ("halves"), each applied in up to two
// segments of K = 32 (two MMAs per lane; K = 16, one MMA, where a K-block has 16 channels) to a window of one activation
// box.  The tensor pipe takes an MMA only when the one before has all but started, so whatever the issuing thread does
// between two MMAs beyond about 128 cycles leaves the pipe idle, and everything around a burst costs it about 550 cycles
// (measured on B200 with clock reads between the parts: decode and waits 150, election and branch 75, commits and the rest
// of the loop 230).  So everything that can be worked out on the host is, and the issuer spreads the rest of the work for
// the next burst between this burst's MMAs.
struct TcBurst {
    uint16_t x_off16[4];    // per segment (0, 1: first half, 2, 3: second): (byte offset of the operand window in its box) / 16
    uint32_t x_hi[2];       // per half: upper word of the activation descriptor (swizzle, SBO = one image row of the box)
    uint32_t w_hi;          // upper word of the weight descriptor
    uint32_t flags;         // bits 0-3: segments present; kBu...
    uint16_t l1_off16;      // (distance of a lane's window from the one before) / 16
    uint16_t w1_off16;      // (distance of a half's second segment of weights from its first) / 16
    uint8_t size[2];        // KiB the halves' fresh boxes take in the activation ring
    uint16_t pad_;
};
static_assert(sizeof(TcBurst) == 32, "copied as two 16-byte words");
constexpr uint32_t kBuNew0 = 1u << 8, kBuNew1 = 1u << 9;      // the first / second half opens a fresh activation box
constexpr uint32_t kBuLast0 = 1u << 10, kBuLast1 = 1u << 11;  // the first / second half is the last reader of its box
constexpr uint32_t kBuTwo = 1u << 12;                         // the burst has a second half
constexpr uint32_t kBuK16 = 1u << 13;                         // segments of one MMA
constexpr uint32_t kBuFirst0 = 1u << 14, kBuFirst1 = 1u << 15;   // the first MMA of the half (per lane of the tile) overwrites
constexpr int kBuOff = 16, kBuMix = 24;                       // from these bits on, four for each half: quarters of the TMEM lanes that the half leaves
                                                              // alone (nodes of the plan that do not read its source); that it writes first, where
                                                              // others that it writes have sums already

// A plan can cover SEVERAL nodes of 32 or 64 channels that have the same shape: an M = 128 instruction on a 64-channel node is half
// empty, on a 32-channel node three quarters, so the weights of up to two or four nodes take the rows one after the other, and
// every K-block of a source that several of them read (same filter geometry, same frame) serves them all.  TMEM lanes
// rows * q .. belong to the plan's node q.  Nodes are joined if they share a source, or if one of them has next to no reduction of
// its own; of all joins the one that saves most K-blocks comes first.  (Deepest CIFAR10 network: 29 K-blocks for the four nodes of
// its first block, where two plans of two had 11 and 27, and 72 for those of the second instead of 81.)  The MMAs of a K-block leave the
// lanes of a node that does not read its source alone (an output-lane mask): rows of zero weights there would turn an infinity in that
// source into a NaN.  Without / with the masks, us per pass: deepest CIFAR10 network 1139 / 1143, six-node at 256 samples 3216 / 3226,
// ten-node 8297 / 8339; launches of fewer items lose more: 1 to 5 % in most, six-node with
// 16 x 16 images at 33 / 130 samples 236 / 252, 510 / 548, 36 x 36 at 33 674 / 727, ten-node with 16 x 16 at 33 347 / 365.  (It is the kernel
// compiled with masks rather than the masked MMAs: constant masks and an order of the K-blocks that leaves a tenth of them masked
// took as long; where the copies of a burst lie does matter, see the issuer.)
struct alignas(16) TcNode {
    void* state[kMaxFused][2];
    const float* bias[kMaxFused];
    int32_t relu, rows, n_nodes, C; // relu: a bit per node; rows: rows of the weight matrix per node (0: the plan has one node)
    int32_t H, W;
    int32_t tw, th, tb, sep;        // geometry of the tile (see the file comment): tw = columns of a lane
    int32_t nl, lane_cols;          // lanes, TMEM columns of each (N of the MMA)
    int32_t n_runs, n_act, n_bu;    // lengths of the node's tables
    uint32_t part_lanes;            // bit 4 * p + q: part p of a split item has K-blocks for quarter q of the TMEM lanes
    uint32_t pairs[4];              // bit i: weight group i of the node has two blocks
    TcRun runs[kMaxRuns];
    int32_t part, n_parts, part_chunks;     // of a split item (see the kernel); part_chunks: 16-column chunks per part
};
static_assert(sizeof(TcNode) % 16 == 0, "copied as 16-byte words");

struct TcParams {
    const CUtensorMap* maps;
    const uint4* tables;
    const TcTile* tiles;
    SrFrameArgs fr;
    int* error;                     // device-side error code
    int* sched;                     // counters of the shared list, or null
    long long wait_limit;
    int n_tiles, n_own;             // items in all; those of the matrix
    int B, follow;
    int table_bytes;                // shared memory of one node table
    int n_w, w_slot;                // weight ring: slots and their size
    int ring_kb;                    // activation ring in KiB
    int exch_off;                   // (SPLIT) where what other parts send lies: bytes from the start of the weight ring
};

// ------------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// PEERS: what completes the barrier was written by other CTAs of the cluster.
template <bool PEERS = false>
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if (PEERS)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Non-blocking probe.
__device__ __forceinline__ uint32_t mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// True in one lane of the (converged) warp.  The tcgen05 and TMA instructions take their operands from uniform registers:
// behind `if (lane == 0)` the compiler has to assume that several lanes with different operands may arrive, behind
// elect.sync it knows that it is one.  Measured on B200 (four MMAs of N = 256, one barrier wait, one table read and one
// commit per K-block, cycles per MMA): 158 behind lane == 0, 128 (the tensor pipe's own rate) behind elect.sync.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p)::"memory");
    return p != 0;
}
// Bounded wait.  Returns false if the limit expired or another role already gave up.  A launch may start early, while a run of many
// frames before it is still on; the limit must not count that time, so every role waits for the predecessor ahead of its first
// bounded wait that depends, through whatever other role, on the predecessor.
template <bool PEERS>
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long limit)
{
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait<PEERS>(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
    }
}
template <bool PEERS = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long limit)
{
    if (mbar_try_wait<PEERS>(bar, parity)) return true;
    return mbar_wait_slow<PEERS>(bar, parity, abort_flag, limit);
}
// Wait for a copy this thread started itself, before the CTA gives up its shared memory.  It has its own limit and
// does not look at the abort flag: after another role gave up, the copies in flight still have to land.
__device__ __noinline__ void mbar_wait_drain(uint32_t bar, uint32_t parity, long long limit)
{
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit) return;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* map, uint32_t bar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// Ask for a box to be brought into L2 (no shared memory, no barrier: fire and forget).
__device__ __forceinline__ void tma_prefetch_4d(const void* map, int c0, int c1, int c2, int c3)
{
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];"
                 ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* map, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The descriptors are given as (address word, shared upper word).
__device__ __forceinline__ void tc_mma_bf16_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                                 uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// Words of ones: TMEM lanes that an MMA does not write (four words of 32 lanes).
struct TcLanes { uint32_t w[4]; };
__device__ __forceinline__ TcLanes tc_lanes(uint32_t quarters)
{
    return TcLanes{{0u - (quarters & 1u), 0u - ((quarters >> 1) & 1u), 0u - ((quarters >> 2) & 1u), 0u - ((quarters >> 3) & 1u)}};
}
__device__ __forceinline__ void tc_mma_bf16_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                                 uint32_t accumulate, const TcLanes& off)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, {%7, %8, %9, %10}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(off.w[0]), "r"(off.w[1]), "r"(off.w[2]), "r"(off.w[3])
        : "memory");
}
__device__ __forceinline__ void tc_commit_if(uint32_t bar, uint32_t cond)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t"
                 "@p tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(cond) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 TMEM lanes x 16 columns: thread T gets columns 2 * (T % 4), + 1 (and those + 8: r[4..7]) of lanes T / 4 (r[0, 1]) and T / 4 + 8
// (r[2, 3]), i.e. the fragments that stmatrix takes.
__device__ __forceinline__ void tc_ld_16x16(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t local, uint32_t rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
// A store into another CTA's shared memory that counts its bytes on a barrier there.
__device__ __forceinline__ void st_async_v4(uint32_t remote, uint32_t remote_bar, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(remote), "r"(a), "r"(b), "r"(c), "r"(d), "r"(remote_bar) : "memory");
}

// ------------------------------------------------------------------------------------------ the kernel
// Work items.  CTA c walks column c of a matrix of items made on the host (longest first onto the least loaded CTA).  The
// kernel ends when its slowest CTA ends, and the cost of an item is only an estimate: measured on B200 such lists left
// that CTA 2-8 % above the mean.  So (sched != nullptr) the matrix holds only the larger items, and the smallest ones, a
// fifth of the work, form ONE shared list behind it from which every CTA takes, by a device-wide counter, when its own
// column is done.  The keeper warp looks the items up ahead of everybody else and hands them on through a ring in shared
// memory, together with the K-loop tables of their nodes (kTables of them stay in shared memory): no other role reads
// a table from global memory, which cost each of them two to three dependent round trips per item (6-8 % of the kernel).
// An item of the shared list is asked for at most kAhead items ahead of the epilogue, so that a slow CTA does not hoard them.
constexpr int kAhead = 3;

// Split reductions (SPLIT: a launch in clusters).  Where a launch has fewer items than SMs, its time is that of the longest
// reduction.  Such an item is cut along K into 2, 4 or 8 parts, one per CTA of a cluster: each part walks its K-blocks like an item
// of its own (a TcNode of its own), with the weights and boxes of these blocks only.  The accumulators are summed through
// distributed shared memory, every part for its share of the columns: a part sends the fp32 fragments of the others' columns to
// them (st.async, 16 bytes per thread) and finishes its own: bias, activation, store.  The order of the sums is fixed.  A CTA has one
// split item at most, the last of its list, so the room for what others send is used once, and one barrier, on which those bytes
// count, is all there is between the CTAs.  Where that room would cost the weight ring its depth, it lies in the rings, which are
// idle by then, and the parts tell each other first that they are (half a microsecond more).  Everything that others write into a
// CTA it has waited for when it leaves.  Measured on B200, us per pass of 16 frames without / with it: six-node network at one
// sample 246 / 143 (sequential 862 / 567), ten-node at 1 / 8 / 20 samples 387 / 166, 403 / 276, 581 / 413 (sequential at 1 / 8 1601 / 940, 1680 / 1178),
// stress graph at 1 / 4 samples 547 / 284, 757 / 671, deepest CIFAR10 network at 1 / 16 352 / 162, 463 / 277.
// Alternatives that lost: a cluster barrier at the end and the sums always in the rings (8.8 -> 10.5 with both); two threads that
// start weight copies in turn (deepest CIFAR10 network at 16 samples 18.8 -> 22.5, at 128 73.8 -> 77.6); two issuing threads with an
// accumulator each for tiles of up to 128 columns (8.8 -> 9.6); launches of half an SM's shared memory, so that the next one
// sets up beside them (14.9 -> 22 before the split: the ring is too shallow).
// MASKED: some K-block of the launch leaves lanes alone (see TcNode).  A kernel of its own, because a launch of an item or two per CTA
// fetches its code from L2: with the masks in every launch the ten-node network, sequential at 16 samples, took 1421 us per pass, so 1379.
// Registers: 80 at most, so that an SM has room for a block of the heads (128 registers x 256 threads) or three of the frame input
// beside a CTA.  (SPLIT is bound to them; unbound, with the sums of all parts in flight, it took 114, and the deepest CIFAR10 network at
// 16 samples, whose heads then waited for the launch to end, 18.6 us per frame, so 17.0.  Without SPLIT the compiler needs 77, and
// being held to 80 costs the ten-node network 2 %.)
template <bool SPLIT, bool MASKED>
__global__ void __launch_bounds__(kThreads, SPLIT ? 2 : 1) sr_tc_group_kernel(const __grid_constant__ TcParams P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * kBoxes + 2 * kMaxW + 4 + kItems + 2];
    __shared__ uint4 clear_words[SPLIT ? kMaxParts : 1];   // what the other parts of a split item say `clear` with
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ TcTile items[kItems];                       // the item ring; node -1 = end of the list
    __shared__ uint32_t box_start[kBoxes];                 // the activation producer's own: `head` at the start of each box
    __shared__ volatile int epi_done;                      // items the epilogue has finished
    __shared__ __align__(16) uint16_t epi_buf[kEpiWarps][16 * 32];   // per epilogue warp: 16 pixels x 32 channels, bf16
    __shared__ int pix_off[2][kMaxCols];                   // number of every pixel of an item in its node's state, -1 = not stored

    if (!(P.follow & 2)) sr_let_successor_start();
    const long long wait_limit = P.wait_limit;
    // A wait limit of zero (a host-side test hook) means "every wait has already expired": report it and return
    // before any barrier, tensor memory, copy or MMA is touched.
    if (wait_limit <= 0) {
        sr_wait_for_predecessor();
        if (threadIdx.x == 0) atomicExch(P.error, 1);
        return;
    }
    // weight ring first: an M = 128 instruction on a node with fewer than 128 output channels reads
    // rows past its weight box, which then still lie inside this allocation
    const uint32_t w_ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_ring = w_ring + (uint32_t)(P.n_w * P.w_slot);
    const uint32_t tab_off = a_ring + (uint32_t)P.ring_kb * 1024u - smem_u32(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar_afull = smem_u32(&bars[0]), bar_aempty = smem_u32(&bars[kBoxes]);
    const uint32_t bar_wfull = smem_u32(&bars[2 * kBoxes]), bar_wempty = smem_u32(&bars[2 * kBoxes + kMaxW]);
    const uint32_t bar_tfull = smem_u32(&bars[2 * kBoxes + 2 * kMaxW]), bar_tempty = bar_tfull + 16, bar_item = bar_tempty + 16;
    const uint32_t bar_sums = bar_item + 8 * kItems, bar_clear = bar_sums + 8;      // (SPLIT) what the other parts send has arrived; they may

    if (threadIdx.x == 0) {
        abort_flag = 0;
        epi_done = 0;
        for (int s = 0; s < kBoxes; ++s) {
            mbar_init(bar_afull + 8 * s, 1);
            mbar_init(bar_aempty + 8 * s, 1);
        }
        for (int s = 0; s < P.n_w; ++s) {
            mbar_init(bar_wfull + 8 * s, 1);
            mbar_init(bar_wempty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull + 8 * a, 1);
            mbar_init(bar_tempty + 8 * a, kEpiWarps);
        }
        for (int s = 0; s < kItems; ++s) mbar_init(bar_item + 8 * s, 1);
        if (SPLIT) {
            mbar_init(bar_sums, 1);
            mbar_init(bar_clear, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // (the keeper's first item is on its way meanwhile)
    TcTile first;
    first.node = -1;
    if (warp == 2 && (int)blockIdx.x < P.n_own) first = P.tiles[blockIdx.x];
    tc_fence_before();
    if (SPLIT) cluster_sync();                             // (the other CTAs' barriers stand, too)
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    volatile int* abortp = &abort_flag;

    const SrFrame F = sr_frame(P.fr);
    const int prev = (int)(F.t & 1), cur = prev ^ 1;
    auto table_of = [&](const TcTile& it) { return reinterpret_cast<const TcNode*>(smem_raw + tab_off + (uint32_t)(it.slot * P.table_bytes)); };

    if (warp == 2) {
        // ---------------------------------------------------------------- keeper
        // (It does not wait for the predecessor to look at tables; the shared list's counter is the predecessor's too.)
        bool waited = false;
        int slot_node = -1, slot_gen = -1;                 // lane s < kTables: the node whose table slot s holds, the last item that uses it
        int slot = -1, cached = -1;
        bool own = true, ok = true;
        for (int it = 0; ok; ++it) {
            TcTile tl;
            tl.node = -1;
            if (own) {
                const long long idx = (long long)blockIdx.x + (long long)it * gridDim.x;
                if (it == 0) tl = first;
                else if (idx < P.n_own) tl = P.tiles[idx];
                own = tl.node >= 0;                        // the rest of this CTA's column is padding
            }
            // room in the item ring (and, for an item of the shared list, not too far ahead)
            const int ahead = own ? kItems : kAhead;
            if (it - epi_done >= ahead) {
                if (!waited) sr_wait_for_predecessor();    // (the epilogue does; see mbar_wait_slow)
                waited = true;
                const long long t0 = clock64();
                while (ok && it - epi_done >= ahead) {
                    if (*abortp || clock64() - t0 > wait_limit) ok = false;
                    __nanosleep(40);
                }
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) { *abortp = 1; break; }
            }
            if (!own && P.sched && P.n_own < P.n_tiles) {
                int v = 0;
                if (!waited) sr_wait_for_predecessor();
                waited = true;
                if (lane == 0) v = P.n_own + atomicAdd(P.sched, 1);
                v = __shfl_sync(0xffffffffu, v, 0);
                if (v < P.n_tiles) tl = P.tiles[v];
            }
            if (tl.node >= 0 && tl.node != cached) {
                // another node: is its table still here?  Else it replaces the one whose last use is longest ago, once the
                // epilogue has finished the items that use that one
                const uint32_t hit = __ballot_sync(0xffffffffu, lane < kTables && slot_node == tl.node);
                if (hit) {
                    slot = __ffs(hit) - 1;
                } else {
                    slot = 0;
                    int oldest = __shfl_sync(0xffffffffu, slot_gen, 0);
                    for (int q = 1; q < kTables; ++q) {
                        const int gq = __shfl_sync(0xffffffffu, slot_gen, q);
                        if (gq < oldest) { oldest = gq; slot = q; }
                    }
                    if (epi_done <= oldest && !waited) {
                        sr_wait_for_predecessor();
                        waited = true;
                    }
                    const long long t0 = clock64();
                    while (ok && epi_done <= oldest) {
                        if (*abortp || clock64() - t0 > wait_limit) ok = false;
                        __nanosleep(40);
                    }
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) { *abortp = 1; break; }
                    uint4* dst = reinterpret_cast<uint4*>(smem_raw + tab_off + slot * P.table_bytes);
                    const uint4* src = P.tables + tl.node;
                    for (int i = lane; i < tl.words; i += 32) dst[i] = src[i];
                    if (lane == slot) slot_node = tl.node;
                }
                cached = tl.node;
            }
            if (lane == slot) slot_gen = it;
            tl.slot = slot;
            __syncwarp();
            if (lane == 0) {
                items[it & (kItems - 1)] = tl;
                mbar_arrive(bar_item + 8 * (it & (kItems - 1)));
            }
            if (tl.node < 0) break;
        }
    } else if (warp == 0) {
        // ---------------------------------------------------------------- weight producer
        // (One elected thread per producer, no warp-wide votes: what a ring slot costs between its release and its next copy is
        // the latency of this loop.)
        if (elect_one()) {
            uint32_t n = 0, s = 0, ph = 1;                        // copies started; next slot, parity of its release
            const uint32_t n_w = (uint32_t)P.n_w, w_slot = (uint32_t)P.w_slot;
            bool ok = true, waited = false;
            for (int it = 0; ok; ++it) {
                // (the first item and the first n_w slots come without the predecessor, the rest is up to the issuer and the epilogue)
                if (it > 0 && !waited && !mbar_test_wait(bar_item + 8 * (it & (kItems - 1)), (it / kItems) & 1)) {
                    sr_wait_for_predecessor();
                    waited = true;
                }
                ok = mbar_wait(bar_item + 8 * (it & (kItems - 1)), (it / kItems) & 1, abortp, wait_limit);
                if (!ok) break;
                const TcTile& tl = items[it & (kItems - 1)];
                if (tl.node < 0) break;
                const TcNode* nd = table_of(tl);
                const int n_runs = nd->n_runs, m0 = tl.m0;
                int gi = 0;                                       // weight group of the node
                for (int r = 0; r < n_runs && ok; ++r) {
                    const TcRun R = nd->runs[r];
                    const CUtensorMap* map1 = &P.maps[R.map1];
                    const CUtensorMap* map2 = &P.maps[R.map2];
                    const uint32_t bytes = (uint32_t)R.bytes16 << 4;
                    const int end = gi + R.n_groups;
                    int blk = R.blk0;
                    for (; gi < end; ++gi) {
                        const uint32_t two = R.map1 == R.map2 ? 0u : (nd->pairs[gi >> 5] >> (gi & 31)) & 1u;
                        if (n == n_w && !waited) {
                            sr_wait_for_predecessor();
                            waited = true;
                        }
                        ok = mbar_wait(bar_wempty + 8 * s, ph, abortp, wait_limit);
                        if (!ok) break;
                        mbar_expect_tx(bar_wfull + 8 * s, bytes << two);
                        tma_load_3d(w_ring + s * w_slot, two ? map2 : map1, bar_wfull + 8 * s, 0, m0, blk);
                        blk += 1 + (int)two;
                        ++n;
                        if (++s == n_w) { s = 0; ph ^= 1; }
                    }
                }
            }
            // every copy this thread started must have landed before the CTA may exit
            for (uint32_t v = 0; v < n_w && v < n; ++v) mbar_wait_drain(bar_wfull + 8 * v, ((n - 1 - v) / n_w) & 1, wait_limit);
        }
    } else if (warp == 3) {
        // ---------------------------------------------------------------- activation producer
        // Box j uses barrier pair j % kBoxes and the bytes [pos, pos + size) of the ring; it wraps as a whole.  `head` counts KiB
        // from the start of the launch, skipped ones included: head minus the start of the oldest box is what is in use.
        // (The weights do not depend on the predecessor, so their producer does not wait for it; the activations do.)
        // Everything up to the first request is done ahead of that wait: tables read, tensor map and instructions fetched (from the
        // end of the wait to the request 0.4-0.6 us without that, 0.05-0.2 so).
        if (elect_one()) {
            bool waited = false;
            uint32_t n = 0, n_free = 0;                           // boxes started; boxes known to be released
            uint32_t pos = 0, head = 0;
            const uint32_t ring = (uint32_t)P.ring_kb;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                ok = mbar_wait(bar_item + 8 * (it & (kItems - 1)), (it / kItems) & 1, abortp, wait_limit);
                if (!ok) break;
                const TcTile& tl = items[it & (kItems - 1)];
                const int node = tl.node, w0 = tl.w0, h0 = tl.h0, b0 = tl.b0;
                if (node < 0) break;
                const TcNode* nd = table_of(tl);
                const int n_act = nd->n_act;
                const uint4* tab = reinterpret_cast<const uint4*>(nd + 1) + 2 * nd->n_bu;
                auto box_of = [&](int i) { const uint4 q = tab[i]; TcAct k; std::memcpy(&k, &q, sizeof(k)); return k; };
                int next = 0;                                     // 0: not looked up, 1: of the same node, 2: not
                for (int i = 0; i < n_act; ++i) {
                    const TcAct k = box_of(i);
                    const uint32_t size = k.ring_kb, s = n & (kBoxes - 1);
                    if (pos + size > ring) { head += ring - pos; pos = 0; }
                    while (n != n_free && (n - n_free == kBoxes || head + size - box_start[n_free & (kBoxes - 1)] > ring)) {
                        ok = mbar_wait(bar_aempty + 8 * (n_free & (kBoxes - 1)), (n_free / kBoxes) & 1, abortp, wait_limit);
                        if (!ok) break;
                        ++n_free;
                    }
                    if (!ok) break;
                    const int par = (k.flags & 1) ? prev : cur;
                    const CUtensorMap* map = &P.maps[par ? k.x_map1 : k.x_map0];
                    if (!waited) {
                        asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
                        sr_wait_for_predecessor();
                        if (P.follow & 2) sr_let_successor_start();
                        waited = true;
                    }
                    mbar_expect_tx(bar_afull + 8 * s, (uint32_t)k.x_bytes16 << 4);
                    tma_load_4d(a_ring + pos * 1024u, map, bar_afull + 8 * s, (int)k.c0_16 << 4, w0 + k.qx, h0 + k.qy, b0);
                    box_start[s] = head;
                    head += size;
                    pos += size;
                    ++n;
                    // A box that comes from DRAM takes longer than the ring covers, so every request is followed by an L2 prefetch
                    // of the box two further on (of the next work item when this one ends, if it is there and of the same node).
                    const bool here = i + 2 < n_act;
                    const int j = here ? i + 2 : i + 2 - n_act;
                    int pw = w0, ph = h0, pb = b0;
                    if (!here) {
                        const TcTile& nx = items[(it + 1) & (kItems - 1)];
                        if (next == 0) next = mbar_test_wait(bar_item + 8 * ((it + 1) & (kItems - 1)), ((it + 1) / kItems) & 1) && nx.node == node ? 1 : 2;
                        if (next == 1) { pw = nx.w0; ph = nx.h0; pb = nx.b0; }
                    }
                    if ((here || next == 1) && j < n_act) {
                        const TcAct p = box_of(j);
                        const int pp = (p.flags & 1) ? prev : cur;
                        tma_prefetch_4d(&P.maps[pp ? p.x_map1 : p.x_map0], (int)p.c0_16 << 4, pw + p.qx, ph + p.qy, pb);
                    }
                }
            }
            if (!waited) {
                sr_wait_for_predecessor();
                if (P.follow & 2) sr_let_successor_start();
            }
            for (uint32_t v = 0; v < kBoxes && v < n; ++v) mbar_wait_drain(bar_afull + 8 * v, ((n - 1 - v) / kBoxes) & 1, wait_limit);
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // One elected thread does everything (see TcBurst): while it issues the MMAs of a burst it works out the next one's
        // addresses and probes (without blocking) whether its operands are there; the commits of a half follow the first
        // MMA of the next one.  A burst that is not ready, or not of the common kind, takes the plain path: half by half, a
        // wait, its MMAs, its commits.
        if (elect_one()) {
            uint32_t a_n = 0xFFFFFFFFu, a_base = 0, a_end = 0;    // number of the activation box in use; its start and the end of
                                                                  // the latest box in the ring, KiB
            uint32_t w_cur = 0, w_ph = 0;                         // next weight slot and its phase
            const uint32_t a_base0 = (a_ring >> 4) | 0x10000u, w_base0 = (w_ring >> 4) | 0x10000u;   // lower descriptor words
            const uint32_t w_step = (uint32_t)P.w_slot >> 4, ring = (uint32_t)P.ring_kb, n_w = (uint32_t)P.n_w;
            struct Burst {
                uint32_t fl, xh0, xh1, wh, l1, x0, x1, x2, x3, v0, v1, v2, v3;
                uint32_t bw0, pw0, bw1, pw1, ba0, pa0, ba1, pa1;  // full barriers and phases of the weight slots and boxes
            };
            // Slots, phases and addresses of the burst recorded in (o, r).  A half that does not open a box reads the one in
            // use (it was waited for before, waiting for its phase again costs nothing); a missing half repeats the first.
            auto decode = [&](const uint4 o, const uint4 r, Burst& b) {
                const uint32_t fl = r.y;
                b.fl = fl; b.xh0 = o.z; b.xh1 = o.w; b.wh = r.x; b.l1 = r.z & 0xFFFFu;
                const uint32_t w1 = r.z >> 16, size0 = r.w & 0xFFu, size1 = (r.w >> 8) & 0xFFu;
                if (fl & kBuNew0) {
                    a_base = a_end + size0 > ring ? 0u : a_end;
                    a_end = a_base + size0;
                    ++a_n;
                }
                b.ba0 = bar_afull + 8 * (a_n & (kBoxes - 1)); b.pa0 = (a_n / kBoxes) & 1u;
                const uint32_t xb0 = a_base0 + a_base * 64u;
                if (fl & kBuNew1) {
                    a_base = a_end + size1 > ring ? 0u : a_end;
                    a_end = a_base + size1;
                    ++a_n;
                }
                b.ba1 = bar_afull + 8 * (a_n & (kBoxes - 1)); b.pa1 = (a_n / kBoxes) & 1u;
                const uint32_t xb1 = a_base0 + a_base * 64u;
                b.bw0 = bar_wfull + 8 * w_cur; b.pw0 = w_ph;
                b.v0 = w_base0 + w_cur * w_step;
                if (++w_cur == n_w) { w_cur = 0; w_ph ^= 1; }
                b.bw1 = b.bw0; b.pw1 = b.pw0; b.v2 = b.v0;
                if (fl & kBuTwo) {
                    b.bw1 = bar_wfull + 8 * w_cur; b.pw1 = w_ph;
                    b.v2 = w_base0 + w_cur * w_step;
                    if (++w_cur == n_w) { w_cur = 0; w_ph ^= 1; }
                }
                b.v1 = b.v0 + w1; b.v3 = b.v2 + w1;
                b.x0 = xb0 + (o.x & 0xFFFFu); b.x1 = xb0 + (o.x >> 16); b.x2 = xb1 + (o.y & 0xFFFFu); b.x3 = xb1 + (o.y >> 16);
            };
            bool ok = true;
            for (int it = 0; ok; ++it) {
                ok = mbar_wait(bar_item + 8 * (it & (kItems - 1)), (it / kItems) & 1, abortp, wait_limit);
                if (!ok) break;
                const TcTile& tl = items[it & (kItems - 1)];
                if (tl.node < 0) break;
                const TcNode* nd = table_of(tl);
                const uint4* tab = reinterpret_cast<const uint4*>(nd + 1);
                const int n_bu = nd->n_bu;
                const uint32_t nl = (uint32_t)nd->nl, lane_cols = (uint32_t)nd->lane_cols;
                // instruction descriptor: D = f32, A = B = bf16, both K-major, M = 128 output channels, N = pixels of a lane
                const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((lane_cols >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
                const uint32_t acc = (uint32_t)it & 1u, d0 = tmem_base + acc * kMaxCols, d1 = d0 + lane_cols;
                Burst c;
                decode(tab[0], tab[1], c);
                if (it == 0) sr_wait_for_predecessor();
                ok = mbar_wait(bar_tempty + 8 * acc, (((uint32_t)it >> 1) & 1u) ^ 1u, abortp, wait_limit);
                if (!ok) break;
                tc_fence_after();                                     // the accumulator was just handed back
                uint32_t ready = mbar_test_wait(c.bw0, c.pw0) & mbar_test_wait(c.bw1, c.pw1) & mbar_test_wait(c.ba0, c.pa0) & mbar_test_wait(c.ba1, c.pa1);
                uint32_t p_fl = 0, p_w1 = 0, p_a1 = 0;                // commits owed for the second half of the burst before
                auto pay = [&](uint32_t cond) {
                    tc_commit_if(p_w1, cond);
                    tc_commit_if(p_a1, cond ? p_fl & kBuLast1 : 0u);
                };
                uint32_t owed = 0;
                for (int bu = 0; bu < n_bu; ++bu) {
                    const int nx = bu + 1 < n_bu ? bu + 1 : bu;
                    const uint4 o = tab[2 * nx], r = tab[2 * nx + 1];
                    Burst n = c;
                    if (!ready) ready = mbar_test_wait(c.bw0, c.pw0) & mbar_test_wait(c.bw1, c.pw1) & mbar_test_wait(c.ba0, c.pa0) & mbar_test_wait(c.ba1, c.pa1);
                    // The common kind; `masked`: with lanes that it leaves alone.
                    auto common = [&](auto masked) {
                        const TcLanes off0 = tc_lanes(c.fl >> kBuOff), off1 = tc_lanes(c.fl >> (kBuOff + 4));
                        const uint32_t sum0 = c.fl & kBuFirst0 ? 0u : 1u, sum1 = decltype(masked)::value && (c.fl & kBuFirst1) ? 0u : 1u;
                        auto mma0 = [&](uint32_t d, uint32_t w, uint32_t x, uint32_t sum) {
                            if constexpr (decltype(masked)::value) tc_mma_bf16_lohi(d, w, c.wh, x, c.xh0, idesc, sum, off0);
                            else tc_mma_bf16_lohi(d, w, c.wh, x, c.xh0, idesc, sum);
                        };
                        auto mma1 = [&](uint32_t d, uint32_t w, uint32_t x, uint32_t sum) {
                            if constexpr (decltype(masked)::value) tc_mma_bf16_lohi(d, w, c.wh, x, c.xh1, idesc, sum, off1);
                            else tc_mma_bf16_lohi(d, w, c.wh, x, c.xh1, idesc, sum);
                        };
                        // a K = 16 step moves both operands 32 bytes along K: +2 in the descriptors' address field
                        mma0(d0, c.v0, c.x0, sum0);
                        pay(owed);
                        mma0(d0, c.v0 + 2, c.x0 + 2, 1u);
                        if (bu + 1 < n_bu) decode(o, r, n);
                        mma0(d0, c.v1, c.x1, 1u);
                        mma0(d0, c.v1 + 2, c.x1 + 2, 1u);
                        if (nl == 2) {
                            mma0(d1, c.v0, c.x0 + c.l1, sum0);
                            mma0(d1, c.v0 + 2, c.x0 + c.l1 + 2, 1u);
                            mma0(d1, c.v1, c.x1 + c.l1, 1u);
                            mma0(d1, c.v1 + 2, c.x1 + c.l1 + 2, 1u);
                        }
                        mma1(d0, c.v2, c.x2, sum1);
                        tc_commit(c.bw0 + 8 * kMaxW);
                        tc_commit_if(c.ba0 + 8 * kBoxes, c.fl & kBuLast0);
                        mma1(d0, c.v2 + 2, c.x2 + 2, 1u);
                        ready = mbar_test_wait(n.bw0, n.pw0) & mbar_test_wait(n.ba0, n.pa0);
                        mma1(d0, c.v3, c.x3, 1u);
                        ready &= mbar_test_wait(n.bw1, n.pw1) & mbar_test_wait(n.ba1, n.pa1);
                        mma1(d0, c.v3 + 2, c.x3 + 2, 1u);
                        if (nl == 2) {
                            mma1(d1, c.v2, c.x2 + c.l1, sum1);
                            mma1(d1, c.v2 + 2, c.x2 + c.l1 + 2, 1u);
                            mma1(d1, c.v3, c.x3 + c.l1, 1u);
                            mma1(d1, c.v3 + 2, c.x3 + c.l1 + 2, 1u);
                        }
                        p_fl = c.fl; p_w1 = c.bw1 + 8 * kMaxW; p_a1 = c.ba1 + 8 * kBoxes;
                        owed = 1;
                    };
                    // A burst whose operands are not there, or of another kind: half by half.
                    auto plain = [&](auto masked) {
                        pay(owed);
                        owed = 0;
#pragma unroll
                        for (uint32_t h = 0; h < 2; ++h) {
                            if (h == 1 && !(c.fl & kBuTwo)) break;
                            ok = mbar_wait(h ? c.bw1 : c.bw0, h ? c.pw1 : c.pw0, abortp, wait_limit) && mbar_wait(h ? c.ba1 : c.ba0, h ? c.pa1 : c.pa0, abortp, wait_limit);
                            if (!ok) break;
                            const uint32_t off = (c.fl >> (kBuOff + 4 * h)) & 15u, mix = (c.fl >> (kBuMix + 4 * h)) & 15u;
                            const uint32_t sum = c.fl & (h ? kBuFirst1 : kBuFirst0) ? 0u : 1u;
                            for (uint32_t l = 0; l < nl; ++l) {
                                const uint32_t d = d0 + l * lane_cols, xl = l * c.l1, xh = h ? c.xh1 : c.xh0;
                                const uint32_t xa = (h ? c.x2 : c.x0) + xl, xb = (h ? c.x3 : c.x1) + xl, va = h ? c.v2 : c.v0, vb = h ? c.v3 : c.v1;
                                auto mma = [&](uint32_t w, uint32_t x, uint32_t sum, uint32_t off) {
                                    if constexpr (decltype(masked)::value) tc_mma_bf16_lohi(d, w, c.wh, x, xh, idesc, sum, tc_lanes(off));
                                    else tc_mma_bf16_lohi(d, w, c.wh, x, xh, idesc, sum);
                                };
                                if (decltype(masked)::value && mix) mma(va, xa, 0u, ~mix);
                                mma(va, xa, sum, off | mix);
                                if (!(c.fl & kBuK16)) mma(va + 2, xa + 2, 1u, off);
                                if (c.fl & (h ? 8u : 2u)) {
                                    mma(vb, xb, 1u, off);
                                    if (!(c.fl & kBuK16)) mma(vb + 2, xb + 2, 1u, off);
                                }
                            }
                            tc_commit((h ? c.bw1 : c.bw0) + 8 * kMaxW);
                            tc_commit_if((h ? c.ba1 : c.ba0) + 8 * kBoxes, c.fl & (h ? kBuLast1 : kBuLast0));
                        }
                        if (ok && bu + 1 < n_bu) {
                            decode(o, r, n);
                            ready = mbar_test_wait(n.bw0, n.pw0) & mbar_test_wait(n.bw1, n.pw1) & mbar_test_wait(n.ba0, n.pa0) & mbar_test_wait(n.ba1, n.pa1);
                        }
                    };
                    // Where the copies for bursts with masks lie matters as much as what they do.  A launch of cut items, which fetches its
                    // code from L2, has copies of both kinds for bursts without masks and both for those with, out of the way (six-node
                    // network at 20 samples 316 us per pass with one copy of the plain kind, so 297; ten-node at 8 280 / 272).  One of many
                    // items has the masked copy of the common kind out of the way and one of the plain kind (with two the deepest
                    // CIFAR10 network took 1150 us instead of 1080, the six-node at 48 samples 571 instead of 562).
                    if constexpr (MASKED && SPLIT) {
                        const bool usual = ready && (c.fl & (15u | kBuK16)) == 15u && nl <= 2 && (c.fl >> kBuMix) == 0;
                        if (__builtin_expect((c.fl >> kBuOff) == 0, 1)) {
                            if (usual) common(std::false_type());
                            else plain(std::false_type());
                        } else {
                            if (usual) common(std::true_type());
                            else plain(std::true_type());
                        }
                        if (!ok) break;
                    } else if (ready && (c.fl & (15u | kBuK16)) == 15u && nl <= 2 && (!MASKED || (c.fl >> kBuMix) == 0)) {
                        if (!MASKED || __builtin_expect((c.fl >> kBuOff) == 0, 1)) common(std::false_type());
                        else common(std::bool_constant<MASKED>());
                    } else {
                        plain(std::bool_constant<MASKED>());
                        if (!ok) break;
                    }
                    c = n;
                }
                if (!ok) break;
                pay(owed);
                tc_commit(bar_tfull + 8 * acc);
            }
        }
    } else if (warp >= 4) {
        // ---------------------------------------------------------------- epilogue (warps 4..11)
        // TMEM lane = output channel, TMEM column = pixel.  Two warps share each quarter of the 128 lanes and take
        // alternate 16-column chunks.  A warp turns 32 channels x 16 pixels into NHWC order through a 1 KiB shared-memory buffer:
        // bias, ReLU and bf16 on fragments of 8 x 8 that stmatrix stores transposed, then every thread reads back 8 consecutive
        // channels of one pixel and stores them as one 16-byte word, so a pixel's 32 channels leave the warp as one 64-byte
        // run.  (With one 2-byte store per value the deepest CIFAR10 network took 74.6 us per frame, so 72.5.)  The number of
        // every pixel of the work item in the state (or -1 for separator rows and pixels outside the image) is tabulated
        // once per item, in one of two tables, so that one barrier per item is enough; that barrier also makes giving up a
        // joint decision.
        sr_wait_for_predecessor();
        const int ew = warp - 4, quarter = ew & 3, half = ew >> 2;      // TMEM lanes 32*quarter .. +31 belong to this warp
        const int et = threadIdx.x - 128;                               // 0..255 among the epilogue threads
        uint16_t* tbuf = &epi_buf[ew][0];
        // the buffer holds 64 bytes per pixel; its four 16-byte chunks (8 channels each) are stored at chunk ^ (pixel / 2 % 4), which
        // keeps both the matrix stores (rows = pixels) and the reads (8 pixels x 4 chunks) free of bank conflicts
        const int st_px = lane & 7, ld_px = lane >> 2;
        const uint32_t st_addr = smem_u32(tbuf) + st_px * 64 + (((lane >> 3) ^ ((st_px >> 1) & 3)) * 16);
        const uint32_t ld_off = (uint32_t)(ld_px * 64 + (((lane & 3) ^ ((ld_px >> 1) & 3)) * 16));
        bool ok = true, owed_sums = false;                              // the other parts of a split item may still send
        for (int it = 0;; ++it) {
            ok = ok && mbar_wait(bar_item + 8 * (it & (kItems - 1)), (it / kItems) & 1, abortp, wait_limit);
            const TcTile tl = items[it & (kItems - 1)];
            const bool work = ok && tl.node >= 0;
            const TcNode* nd = work ? table_of(tl) : nullptr;
            int* poff = pix_off[it & 1];
            int n_cols = 0;
            if (work) {
                const int tw = nd->tw, th = nd->th, rows = th + nd->sep, lane_cols = nd->lane_cols, nl = nd->nl;
                n_cols = nl * lane_cols;
                const int l = et / lane_cols, nn = et - l * lane_cols, x = nn % tw, q = nn / tw, r = q % rows, bi = q / rows;
                const int b = tl.b0 + bi, y = tl.h0 + r, xx = tl.w0 + l * tw + x;
                const bool in = l < nl && r < th && bi < nd->tb && b < P.B && y < nd->H && xx < nd->W;
                poff[et] = in ? (b * nd->H + y) * nd->W + xx : -1;
            }
            uint32_t stop;
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                         : "=r"(stop) : "r"(work ? 0u : 1u) : "memory");
            if (et == 0) epi_done = it;                              // every warp has finished the items before this one
            if (stop) {
                if (!ok) *abortp = 1;
                if (SPLIT && owed_sums) mbar_wait_drain(bar_sums, 0, wait_limit);
                break;
            }
            const uint32_t acc = (uint32_t)it & 1u;
            const int rows = nd->rows, C = nd->C;
            const int which = rows == 32 ? quarter : rows == 64 ? quarter >> 1 : 0;       // the plan's node that this warp's TMEM lanes belong to
            const bool there = which < nd->n_nodes;
            __nv_bfloat16* out = static_cast<__nv_bfloat16*>(nd->state[which][cur]);
            const int co_w = rows ? (quarter * 32) & (rows - 1) : tl.m0 + quarter * 32;   // first channel of this warp
            float bias[4];                                          // of channels co_w + lane / 4 + 0, 8, 16, 24
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int co = co_w + (lane >> 2) + 8 * q;
                bias[q] = there && co < C ? __ldg(nd->bias[which] + co) : 0.f;
            }
            const bool relu = (nd->relu >> which) & 1;
            const bool gvalid = there && co_w + (lane & 3) * 8 < C;          // this thread's group of 8 channels exists
            ok = mbar_wait(bar_tfull + 8 * acc, ((uint32_t)it >> 1) & 1u, abortp, wait_limit);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) continue;                                      // to the joint decision at the next barrier
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * kMaxCols;
            uint32_t lo[8], hi[8];                                  // TMEM lanes 0..15 and 16..31 of the quarter
            const int c_first = half * 16;
            auto fetch = [&](int c0) {
                tc_ld_16x16(taddr + c0, lo);
                tc_ld_16x16(taddr + (16u << 16) + c0, hi);
            };
            // the 32 channels x 16 pixels in lo, hi; `fetch_next` is called when their registers are free
            auto finish = [&](int c0, auto fetch_next) {
                uint32_t h[2][4];                                   // [8 pixels][8 channels]: two pixels of one channel per word
#pragma unroll
                for (int pb = 0; pb < 2; ++pb)
#pragma unroll
                    for (int cb = 0; cb < 4; ++cb) {
                        const uint32_t* r = (cb < 2 ? lo : hi) + pb * 4 + (cb & 1) * 2;
                        __nv_bfloat162 z = __floats2bfloat162_rn(__uint_as_float(r[0]) + bias[cb], __uint_as_float(r[1]) + bias[cb]);
                        if (relu) z = __hmax2(z, __floats2bfloat162_rn(0.f, 0.f));
                        h[pb][cb] = *reinterpret_cast<const uint32_t*>(&z);
                    }
                fetch_next();
                stmatrix_x4_trans(st_addr, h[0][0], h[0][1], h[0][2], h[0][3]);
                stmatrix_x4_trans(st_addr + 512, h[1][0], h[1][1], h[1][2], h[1][3]);
                __syncwarp();
#pragma unroll
                for (int pass = 0; pass < 2; ++pass) {
                    const int o = poff[c0 + pass * 8 + (lane >> 2)];
                    if (o >= 0 && gvalid) {
                        const uint4 w = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>(tbuf) + pass * 512 + ld_off);
                        *reinterpret_cast<uint4*>(out + (size_t)o * C + co_w + (lane & 3) * 8) = w;
                    }
                }
                __syncwarp();
            };
            if (SPLIT && nd->n_parts > 1) {
                const int n_parts = nd->n_parts, me = nd->part, per = nd->part_chunks, n_chunks = n_cols / 16;
                const int own0 = min(me * per, n_chunks), own1 = min(own0 + per, n_chunks);
                // fragments of chunk c from part p: 8 KiB at ((p less one beyond me) * per + c - own0) * 8 KiB, of which this warp
                // writes and reads the same 2 KiB, a thread the same 64 bytes
                const uint32_t mine = w_ring + (uint32_t)(P.exch_off + quarter * 2048 + lane * 16);
                owed_sums = true;
                if (et == 0) mbar_expect_tx(bar_sums, (uint32_t)((n_parts - 1) * (own1 - own0)) * 8192u);
                if (P.exch_off == 0) {
                    // (into the rings, which are idle when all parts have come this far)
                    if (et == 0) {
                        mbar_expect_tx(bar_clear, 16u * (uint32_t)(n_parts - 1));
                        for (int p = 0; p < n_parts; ++p)
                            if (p != me) st_async_v4(map_rank(smem_u32(&clear_words[me]), tl.rank0 + p), map_rank(bar_clear, tl.rank0 + p), 1u, 1u, 1u, 1u);
                    }
                    ok = mbar_wait<true>(bar_clear, 0, abortp, wait_limit);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) continue;
                }
                for (int c = half; c < n_chunks; c += 2) {
                    const int to = c / per;
                    if (to == me) continue;
                    fetch(c * 16);
                    const uint32_t dst = map_rank(mine + (uint32_t)((me < to ? me : me - 1) * per + c - to * per) * 8192u, tl.rank0 + to);
                    const uint32_t bar = map_rank(bar_sums, tl.rank0 + to);
                    tc_wait_ld();
                    st_async_v4(dst, bar, lo[0], lo[1], lo[2], lo[3]);
                    st_async_v4(dst + 512, bar, lo[4], lo[5], lo[6], lo[7]);
                    st_async_v4(dst + 1024, bar, hi[0], hi[1], hi[2], hi[3]);
                    st_async_v4(dst + 1536, bar, hi[4], hi[5], hi[6], hi[7]);
                }
                ok = mbar_wait<true>(bar_sums, 0, abortp, wait_limit);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) continue;
                owed_sums = false;
                // (a part without K-blocks for these lanes has no sums for them)
                const uint32_t have = nd->part_lanes >> quarter;
                for (int c = own0 + ((own0 ^ half) & 1); c < own1; c += 2) {
                    fetch(c * 16);
                    tc_wait_ld();
                    if (MASKED && !((have >> (4 * me)) & 1u)) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) lo[i] = hi[i] = 0u;
                    }
#pragma unroll 1
                    for (int p = 0; p + 1 < n_parts; ++p) {
                        const bool has = !MASKED || ((have >> (4 * (p < me ? p : p + 1))) & 1u);
                        const uint4* x = reinterpret_cast<const uint4*>(smem_raw + (mine - smem_u32(smem_raw)) + (size_t)(p * per + c - own0) * 8192u);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint4 v = has ? x[q * 32] : make_uint4(0u, 0u, 0u, 0u);
                            uint32_t* r = (q < 2 ? lo : hi) + (q & 1) * 4;
                            r[0] = __float_as_uint(__uint_as_float(r[0]) + __uint_as_float(v.x));
                            r[1] = __float_as_uint(__uint_as_float(r[1]) + __uint_as_float(v.y));
                            r[2] = __float_as_uint(__uint_as_float(r[2]) + __uint_as_float(v.z));
                            r[3] = __float_as_uint(__uint_as_float(r[3]) + __uint_as_float(v.w));
                        }
                    }
                    finish(c * 16, [] {});
                }
            } else {
                if (c_first < n_cols) fetch(c_first);
                for (int c0 = c_first; c0 < n_cols; c0 += 32) {
                    tc_wait_ld();
                    finish(c0, [&] {
                        if (c0 + 32 < n_cols) fetch(c0 + 32);       // the next chunk, on its way during the stores
                    });
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty + 8 * acc);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    // Given up: those that have not left may still write to this CTA.  (What they have sent has landed when they arrive here: a part that
    // sends then waits, or drains, for a sum from this CTA that does not come, as long as a wait may last.)
    if (SPLIT && abort_flag) cluster_sync();
    if (threadIdx.x == 0 && abort_flag) atomicExch(P.error, 1);
    if (threadIdx.x == 0 && P.sched && P.n_own < P.n_tiles) {
        // the CTA that leaves last (none takes an item any more) puts the counters back for the next launch
        __threadfence();
        if (atomicAdd(P.sched + 1, 1) == (int)gridDim.x - 1) {
            P.sched[0] = 0;
            P.sched[1] = 0;
            __threadfence();
        }
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ------------------------------------------------------------------------------------------ host side
struct KbHost {
    int edge;
    bool stem;
    int stem_index;
    int ky, kx, c0, bk;
    int k_off;
    bool x_load;       // opens a fresh activation box (else: reads the box opened by an earlier tap of its class)
    int x_shift;       // pixels by which this tap's window is shifted inside the box
    int x_width;       // pixels per image row of the box
    int x_rows;        // image rows of the box, per sample
    bool x_release;
    int box_qy = 0, box_qx = 0, box_ry = 0, box_rx = 0;   // origin and residue class of the box (loading block)
    int src_col = 0;   // first column of this block in the edge's own weight matrix [C_out][k * k * C_in]
    int run = 0;       // run of equally wide K-blocks this block belongs to, and its index inside the run
    int blk = 0;
    int w_off = 0;     // byte offset of this block's weights inside the group's slot
    int ring_kb = 0;   // KiB the box takes in the activation ring
    std::vector<std::pair<int, int>> users;   // the edges that this block serves (of different nodes of the plan, the first is `edge`), and
                                              // the first row of their weights in the plan's weight matrix
};

// Consecutive K-blocks of equal channel-block width: one 3-D view (channels of a block, output channels, blocks) of
// the node's weight matrix, whose columns are stored in the order the K loop walks them.
struct WRun { int bk, first_col, n_blocks; };
struct WGroup { int run, blk, n, first_kb; };

struct NodePlan {
    int node;
    std::vector<int> nodes;         // the nodes of the plan, `node` first
    int rows_total(const sr_graph* g) const { return (int)nodes.size() * g->nodes[node].d.c; }   // rows of the weight matrix
    std::vector<int> in_edges(const sr_graph* g) const
    {
        std::vector<int> all;
        for (int v : nodes) all.insert(all.end(), g->nodes[v].in_edges.begin(), g->nodes[v].in_edges.end());
        return all;
    }
    int sep, span;                  // rows / columns the taps that share one activation box are apart at most
    int tw, th, tb, nl, lane_cols;  // tile geometry (see the file comment)
    bool flat;
    int k_total;                    // columns of the concatenated weight matrix
    // Quarters of the TMEM lanes whose nodes a K-block serves (those that no node has are served by all).
    uint32_t quarters_of(const sr_graph* g, const KbHost& kb) const
    {
        if (nodes.size() == 1) return 15u;
        const int per = g->nodes[node].d.c / 32;
        uint32_t used = (15u << per * nodes.size()) & 15u;
        for (const auto& u : kb.users) used |= ((1u << per) - 1u) << u.second / 32;
        return used;
    }
    std::vector<KbHost> kbs;
    std::vector<WRun> runs;
    int n_parts = 1;                // parts of an item's reduction
    struct Part { std::vector<KbHost> kbs; std::vector<WGroup> wgroups; int table_off, table_words; };   // (its table: see TcTile)
    std::vector<Part> parts;
    SrRegion wcat;
};

struct StemPlan {
    int edge;
    int Kp;
    SrRegion buf[2];
};

struct TcEngine {
    std::vector<NodePlan> nodes;                 // tensor-core nodes
    std::vector<int> node_of;                    // graph node -> index in nodes, or -1
    std::vector<StemPlan> stems;
    std::vector<int> stem_of_edge;
    std::vector<std::vector<TcTile>> group_tiles;
    // per launch group: its items' place in the list of all, those of the matrix; grid and cluster (0: none); shared memory
    struct Launch {
        int first_tile = 0, n_own = 0, grid = 0, cluster = 0;
        int n_w = 2, w_slot = 1024, ring_kb = 0, table_bytes = 0, exch = 0;      // exch: bytes for what the other parts of an item send
        bool fits = false, masked = false;                                       // masked: some K-block of a plan does not serve all of its lanes
        int rings() const { return n_w * w_slot + ring_kb * 1024 + kTables * table_bytes; }
        int exch_off() const { return exch ? rings() : 0; }                      // 0: in the rings
        size_t smem() const { return (size_t)rings() + exch + 1024; }
    };
    std::vector<Launch> launches;
    SrRegion r_maps, r_tables, r_tiles;
    int n_maps = 0, n_tiles = 0;
    // optional timing of the group launches with CUDA events on the launching stream
    std::vector<cudaEvent_t> ev;             // pairs: start, stop
    size_t ev_used = 0;
    double timed_ms = 0.0;
    long long timed_launches = 0;
};

TcEngine* eng(const sr_graph* g) { return static_cast<TcEngine*>(g->tc); }

int block_k(int cs) { return cs % 64 == 0 ? 64 : (cs % 32 == 0 ? 32 : 16); }
int stem_kp(int K) { return K <= 16 ? 16 : (K <= 32 ? 32 : (K <= 64 ? 64 : 128)); }
bool is_stem(const sr_graph* g, const SrHostEdge& e)
{
    const SrHostNode& s = g->nodes[e.d.src];
    return s.is_input && (s.d.c % 16) != 0 && e.K <= 128;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

CUtensorMapSwizzle swizzle_of(int bk)
{
    return bk == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (bk == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

uint32_t desc_hi_of(int bk)
{
    const uint32_t sbo = (uint32_t)(8 * bk * 2) >> 4;                    // 8 rows of bk bf16
    const uint32_t layout = bk == 64 ? 2u : (bk == 32 ? 4u : 6u);        // 128B / 64B / 32B swizzle
    return sbo | (1u << 14) | (layout << 29);
}

// A launch on more than half of the SMs cannot set up its CTAs while the one before it runs: about as many cycles later.  One in
// clusters starts up later than one without.
constexpr long long kLateStart = 4000, kClusterStart = 1000;

// Cycles of one MMA (M = 128, K = 16) of n columns, measured on B200 (see the file comment).
double mma_cycles(int n) { return std::max(n / 2.0, (128 + n) / 4.0); }

// Pick the pixel tile of a node among those of at most max_cols columns: the one that computes the image in the least time,
// where a K-block of 64 channels takes the time of its MMAs or of its copies (at 60 bytes per cycle and SM), whichever is
// longer.  per_box: K-blocks that share one activation box on average.
void choose_tile(int H, int W, int B, int max_cols, int forced_tw, double per_box, NodePlan& P)
{
    double best = 1e30;
    auto offer = [&](bool flat, int tw, int th, int tb, int nl, int n) {
        const int lane_cols = (n + 15) / 16 * 16;
        if (nl * lane_cols > max_cols || th < 1) return;
        const double tiles = (double)((W + tw * nl - 1) / (tw * nl)) * ((H + th - 1) / th) * ((B + tb - 1) / tb);
        const double box_px = flat ? (double)tw * th * tb : (double)(8 * nl + P.span) * (th + P.sep) * tb;
        const double feed = (16384.0 + box_px * 128.0 / per_box) / 60.0;
        const double cost = tiles * (std::max(4.0 * nl * mma_cycles(lane_cols), feed) + 20.0 + 1e-3 * nl);
        if (cost < best) {
            best = cost;
            P.flat = flat; P.tw = tw; P.th = th; P.tb = tb; P.nl = nl; P.lane_cols = lane_cols;
        }
    };
    if (P.sep == 0 && P.span == 0 && W <= max_cols && forced_tw == 0) {
        const int rows = max_cols / W;
        if (rows >= H) {
            const int tb = std::max(1, std::min(B, max_cols / (H * W)));
            offer(true, W, H, tb, 1, tb * H * W);
        } else {
            const int parts = (H + rows - 1) / rows, th = (H + parts - 1) / parts;
            offer(true, W, th, 1, 1, th * W);
        }
    }
    for (int nl = 1; nl <= 8; nl *= 2) {
        if (nl > 1 && 8 * (nl / 2) >= W) break;
        if (forced_tw > 0 && nl != forced_tw / 8 && !(8 * nl >= W && forced_tw > 8 * nl)) continue;
        const int lane_max = max_cols / nl / 16 * 16, rows = lane_max / 8;       // (whole steps of an instruction's N)
        if (rows < 1) break;
        if (rows >= H) {
            const int tb = std::max(1, std::min(B, (lane_max + P.sep * 8) / ((H + P.sep) * 8)));
            offer(false, 8, H, tb, nl, tb * (H + P.sep) * 8 - P.sep * 8);
        } else {
            const int parts = (H + rows - 1) / rows, th = (H + parts - 1) / parts;
            offer(false, 8, th, 1, nl, th * 8);
        }
    }
}

void tap_q(int tap, int pad, int st, int& q, int& r)
{
    const int a = tap - pad;
    q = (a >= 0) ? a / st : -((-a + st - 1) / st);
    r = a - q * st;
}

// Do two edges read the same source through the same filter geometry in the same frame?  (Staged edges are not shared.)
bool same_source(const sr_graph* g, int e1, int e2)
{
    const SrHostEdge& a = g->edges[e1];
    const SrHostEdge& b = g->edges[e2];
    return a.d.src == b.d.src && a.d.kind == SR_EDGE_CONV && b.d.kind == SR_EDGE_CONV && a.k_eff == b.k_eff &&
           a.stride_eff == b.stride_eff && a.pad_eff == b.pad_eff && a.d.pool == b.d.pool && a.K == b.K && a.R == b.R &&
           !is_stem(g, a) && !is_stem(g, b);
}

// The incoming edges of a plan's nodes: an edge of a further node that reads the same source through the same filter geometry in
// the same frame shares the K-blocks of an earlier node's.  edges: (edge, place of its node in the plan).
struct SharedEdge { std::vector<std::pair<int, int>> edges; };
std::vector<SharedEdge> shared_edges(const sr_graph* g, const std::vector<int>& nodes)
{
    std::vector<SharedEdge> out;
    for (int q = 0; q < (int)nodes.size(); ++q)
        for (int e : g->nodes[nodes[q]].in_edges) {
            SharedEdge* with = nullptr;
            for (SharedEdge& s : out)
                if (!with && s.edges.back().second < q && same_source(g, s.edges[0].first, e)) with = &s;
            if (with) with->edges.push_back({e, q});
            else out.push_back(SharedEdge{{{e, q}}});
        }
    return out;
}
int edge_blocks(const sr_graph* g, int e)
{
    const SrHostEdge& he = g->edges[e];
    const int cs = g->nodes[he.d.src].d.c;
    return is_stem(g, he) ? 2 : he.k_eff * he.k_eff * (cs / block_k(cs));
}
int plan_blocks(const sr_graph* g, const std::vector<int>& nodes)
{
    int n = 0;
    for (const SharedEdge& s : shared_edges(g, nodes)) n += edge_blocks(g, s.edges[0].first);
    return n;
}

// The plans of a launch group's nodes, of up to `most` nodes each (see TcNode).
std::vector<std::vector<int>> join_nodes(const sr_graph* g, const std::vector<int>& group, size_t most)
{
    std::vector<std::vector<int>> of;
    for (int v : group)
        if (g->nodes[v].use_tc) of.push_back({v});
    for (bool more = most > 1; more;) {
        int a = -1, b = -1, best = -1;
        for (size_t i = 0; i < of.size(); ++i)
            for (size_t j = i + 1; j < of.size(); ++j) {
                const sr_node_desc &x = g->nodes[of[i][0]].d, &y = g->nodes[of[j][0]].d;
                const size_t n_nodes = of[i].size() + of[j].size();
                if ((x.c != 32 && x.c != 64) || y.c != x.c || y.h != x.h || y.w != x.w || n_nodes * x.c > 128 || n_nodes > most) continue;
                std::vector<int> both = of[i];
                both.insert(both.end(), of[j].begin(), of[j].end());
                std::sort(both.begin(), both.end());
                const int bi = plan_blocks(g, of[i]), bj = plan_blocks(g, of[j]), n = plan_blocks(g, both);
                // without a shared source the joint plan issues as many MMAs as the two; it still pays when one of them has next
                // to no reduction (a node fed by a staged edge only): its tiles are all epilogue, which then runs beside the
                // other's MMAs
                const int saved = bi + bj - n;
                if ((saved > 0 || std::min(bi, bj) <= 2) && n <= kMaxNodeKb && saved > best) {
                    a = (int)i;
                    b = (int)j;
                    best = saved;
                }
            }
        more = a >= 0;
        if (!more) break;
        of[a].insert(of[a].end(), of[b].begin(), of[b].end());
        std::sort(of[a].begin(), of[a].end());
        of.erase(of.begin() + b);
    }
    return of;
}

// The K-blocks of a plan for its tile geometry (the stems' staging buffers exist already).
void build_kblocks(const sr_graph* g, const TcEngine* E, NodePlan& P)
{
    const SrHostNode& n = g->nodes[P.node];
    P.kbs.clear();
    struct Ent { int e; std::vector<std::pair<int, int>> users; };
    std::vector<Ent> ents;
    for (const SharedEdge& sh : shared_edges(g, P.nodes)) {
        Ent en{sh.edges[0].first, {}};
        for (const auto& u : sh.edges) en.users.push_back({u.first, u.second * n.d.c});
        ents.push_back(en);
    }
    // The order of the reduction is free (a sum): edges with wider channel blocks come first, so that K-blocks of
    // equal width form one run each and a run's weights are one 3-D tensor.
    auto width_of = [&](int e) {
        const SrHostEdge& he = g->edges[e];
        return is_stem(g, he) ? std::min(64, E->stems[E->stem_of_edge[e]].Kp) : block_k(g->nodes[he.d.src].d.c);
    };
    std::stable_sort(ents.begin(), ents.end(), [&](const Ent& a, const Ent& b) { return width_of(a.e) > width_of(b.e); });
    const int cols = P.nl * P.tw;                                     // image columns of the tile
    // KiB a box takes in the ring: its pixels, or what the windows of its last tap reach to (columns beyond the tile's
    // pixels are computed on whatever lies there and never stored)
    auto ring_kb = [&](const KbHost& kb, int max_shift) {
        const int sbo_px = P.flat ? 8 : kb.x_width;
        const size_t box = (size_t)kb.x_width * kb.x_rows * P.tb, reach = (size_t)max_shift + (P.nl - 1) * 8 + (size_t)(P.lane_cols / 8 - 1) * sbo_px + 8;
        return (int)((std::max(box, reach) * kb.bk * 2 + 1023) / 1024);
    };
    for (const Ent& en : ents) {
        const int e = en.e;
        const SrHostEdge& he = g->edges[e];
        const SrHostNode& s = g->nodes[he.d.src];
        if (is_stem(g, he)) {
            // a staged edge: its im2col rows are one K-block of 16 / 32 / 64 columns, or two of 64
            const int si = E->stem_of_edge[e], Kp = E->stems[si].Kp, bk = std::min(64, Kp);
            for (int c0 = 0; c0 < Kp; c0 += bk) {
                KbHost kb{e, true, si, 0, 0, c0, bk, 0, true, 0, cols, P.th + (P.tb > 1 ? P.sep : 0), true};
                kb.src_col = c0;
                kb.users = en.users;
                kb.ring_kb = ring_kb(kb, 0);
                P.kbs.push_back(kb);
            }
        } else {
            // Taps whose input pixels fall into the same residue class of the stride read the same view of the source,
            // shifted by whole pixels: they share ONE activation box and differ only in where their window starts inside it.
            const int bk = block_k(s.d.c), k = he.k_eff, st = he.stride_eff;
            struct Tap { int ky, kx, qy, qx; };
            std::map<std::pair<int, int>, std::vector<Tap>> classes;            // (ry, rx) -> taps
            for (int ky = 0; ky < k; ++ky)
                for (int kx = 0; kx < k; ++kx) {
                    int qy, ry, qx, rx;
                    tap_q(ky, he.pad_eff, st, qy, ry);
                    tap_q(kx, he.pad_eff, st, qx, rx);
                    classes[std::make_pair(ry, rx)].push_back(Tap{ky, kx, qy, qx});
                }
            for (int c0 = 0; c0 < s.d.c; c0 += bk)
                for (auto& cl : classes) {
                    const std::vector<Tap>& taps = cl.second;
                    int qy0 = 1 << 20, qx0 = 1 << 20, qy1 = -(1 << 20), qx1 = -(1 << 20);
                    for (const Tap& t : taps) {
                        qy0 = std::min(qy0, t.qy); qx0 = std::min(qx0, t.qx);
                        qy1 = std::max(qy1, t.qy); qx1 = std::max(qx1, t.qx);
                    }
                    // samples are stacked th + sep rows apart; a single sample's box is as high as its taps need
                    const int bw = cols + (qx1 - qx0), bh = P.th + (P.tb > 1 ? P.sep : qy1 - qy0);
                    const size_t first = P.kbs.size();
                    int max_shift = 0;
                    for (size_t i = 0; i < taps.size(); ++i) {
                        const Tap& t = taps[i];
                        // the first tap of the class carries the box origin (qy0, qx0)
                        KbHost kb{e, false, -1, t.ky, t.kx, c0, bk, 0,
                                  i == 0, (t.qy - qy0) * bw + (t.qx - qx0), bw, bh, i + 1 == taps.size()};
                        max_shift = std::max(max_shift, kb.x_shift);
                        kb.src_col = (t.ky * k + t.kx) * s.d.c + c0;
                        kb.users = en.users;
                        kb.box_qy = qy0;
                        kb.box_qx = qx0;
                        kb.box_ry = cl.first.first;
                        kb.box_rx = cl.first.second;
                        P.kbs.push_back(kb);
                    }
                    const int kb = ring_kb(P.kbs[first], max_shift);
                    for (size_t i = first; i < P.kbs.size(); ++i) P.kbs[i].ring_kb = kb;
                }
        }
    }
}

// Cycles of a K-block: those of its MMAs or of its copies (at 60 bytes per cycle), whichever are more; in a launch of few items
// (ring_cycles > 0, see below) also at least its share of the time in which a slot of the weight ring comes round, and of the
// issuing thread's work (720 cycles for two weight slots).
double kb_cycles(const sr_graph* g, const NodePlan& P, const KbHost& kb, double ring_cycles)
{
    const double w_bytes = std::min(P.rows_total(g), 128) * 2.0;
    const double c = std::max((kb.bk / 16) * P.nl * mma_cycles(P.lane_cols), (w_bytes * kb.bk + (kb.x_load ? kb.ring_kb * 1024.0 : 0.0)) / 60.0);
    return ring_cycles > 0 ? std::max(c, (kb.bk == 64 ? 1.0 : 0.5) * std::max(330.0, ring_cycles)) : c;
}
// From the release of a slot to the arrival of the next weights, over the slots: 1 us, or 1.5 us where all SMs have several items.
double ring_cycles(int n_w, bool crowded) { return (crowded ? 3000.0 : 2000.0) / n_w; }

// Weight groups (one copy and one slot of the weight ring each): one K-block of 64 channels, or two narrower ones.
// (Groups of twice the size make a ring of three slots out of one of six: with one of them in use two thirds are in
// flight instead of five sixths.)  A group reads one activation box.  The plan's n_parts parts take about the same time each; a
// box whose taps fall into two parts is loaded by both.
void build_groups(const sr_graph* g, NodePlan& P)
{
    P.runs.clear();
    P.parts.assign(P.n_parts, NodePlan::Part());
    int k_off = 0;
    double total = 0, done = 0;
    for (const KbHost& kb : P.kbs) total += kb_cycles(g, P, kb, ring_cycles(kMaxW, false));
    size_t part = 0;
    for (size_t i = 0; i < P.kbs.size(); ++i) {
        KbHost& kb = P.kbs[i];
        kb.k_off = k_off;
        k_off += kb.bk;
        if (P.runs.empty() || P.runs.back().bk != kb.bk) P.runs.push_back(WRun{kb.bk, kb.k_off, 0});
        kb.run = (int)P.runs.size() - 1;
        kb.blk = P.runs.back().n_blocks++;
        // the next part begins here if this block's middle lies beyond this part's share, or if as many blocks are left as parts
        const double cost = kb_cycles(g, P, kb, ring_cycles(kMaxW, false));
        if (!P.parts[part].kbs.empty() && part + 1 < P.parts.size() &&
            ((done + 0.5 * cost) * P.n_parts > total * (part + 1) || P.kbs.size() - i < P.parts.size() - part))
            ++part;
        done += cost;
        NodePlan::Part& q = P.parts[part];
        q.kbs.push_back(kb);
        if (q.kbs.size() == 1 && !kb.x_load) {
            q.kbs[0].x_load = true;
            P.parts[part - 1].kbs.back().x_release = true;
        }
        if (q.kbs.back().x_load || q.wgroups.back().run != kb.run || q.wgroups.back().n >= (kb.bk == 64 ? 1 : 2))
            q.wgroups.push_back(WGroup{kb.run, kb.blk, 0, (int)q.kbs.size() - 1});
        q.wgroups.back().n += 1;
    }
    P.k_total = k_off;
}

// Two consecutive weight groups are one burst if their K-blocks are equally wide.
bool one_burst(const NodePlan::Part& P, size_t gi)
{
    return gi + 1 < P.wgroups.size() && P.kbs[P.wgroups[gi + 1].first_kb].bk == P.kbs[P.wgroups[gi].first_kb].bk;
}
int count_bursts(const NodePlan::Part& P)
{
    int n = 0;
    for (size_t gi = 0; gi < P.wgroups.size(); ++n) gi += one_burst(P, gi) ? 2 : 1;
    return n;
}

std::vector<TcTile> node_tiles(const sr_graph* g, const NodePlan& P, int node_index)
{
    const SrHostNode& n = g->nodes[P.node];
    std::vector<TcTile> out;
    for (int b0 = 0; b0 < g->batch; b0 += P.tb)
        for (int h0 = 0; h0 < n.d.h; h0 += P.th)
            for (int w0 = 0; w0 < n.d.w; w0 += P.tw * P.nl)
                for (int m0 = 0; m0 < P.rows_total(g); m0 += 128) out.push_back(TcTile{node_index, b0, h0, w0, m0, 0, 0, 0});
    return out;
}

// Estimated cycles of one item of the plan: its K-blocks, start-up and the share of the epilogue that is not hidden.
long long item_cycles(const sr_graph* g, const NodePlan& P, double ring_cycles)
{
    double c = 1500.0;
    for (const KbHost& kb : P.kbs) c += kb_cycles(g, P, kb, ring_cycles);
    return (long long)c;
}

// 16-column chunks of the accumulator that one of an item's parts sums.
int part_chunks(const NodePlan& P, int parts) { return (P.nl * P.lane_cols / 16 + parts - 1) / parts; }

// Estimated cycles of one of the parts of an item of `cycles`: K-blocks and start, and what it sends to the others (8 KiB a chunk).
// Sums that have no room of their own go where the rings were, each part's once these have run dry there: 1200 cycles a part (by a
// constant instead, ten-node sequential at 16 samples 88.9 -> 93.1 us per frame, six-node at 4 samples 10.3 -> 11.4).
long long part_cycles(const NodePlan& P, long long cycles, int parts, bool in_rings)
{
    if (parts <= 1) return cycles;
    return 1500 + (cycles - 1500) / parts + 1200 + (in_rings ? 1200 * (parts - 1) : 0) + 320 * (P.nl * P.lane_cols / 16 - part_chunks(P, parts));
}

cudaLaunchConfig_t cluster_config(int grid, int cluster, size_t smem, cudaStream_t stream, bool early, cudaLaunchAttribute (&at)[2])
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 2 : 1;
    return cfg;
}

// Clusters of a launch that the device holds at once, one CTA to an SM.
int clusters_held(const sr_graph* g, int cluster)
{
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t cfg = cluster_config(cluster, cluster, kSmemBudget, nullptr, false, at);
    int held = 0;
    if (cudaFuncSetAttribute(sr_tc_group_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&held, sr_tc_group_kernel<true, true>, &cfg) == cudaSuccess && held > 0)
        return std::min(held, g->sm_count / cluster);
    cudaGetLastError();
    return std::max(1, g->sm_count / cluster);
}

}  // namespace

// A node goes to the tensor cores if it sums convolutions only, has at least 16 output channels in
// multiples of 8, and every incoming edge either has C_in % 16 == 0 or is a few-channel input edge.  Its pixels (and the
// 16-byte chunks of a staged edge, see sr_input.cuh) are counted in 32 bits.
void sr_tc_select_nodes(sr_graph* g)
{
    for (size_t v = 0; v < g->nodes.size(); ++v) {
        SrHostNode& n = g->nodes[v];
        n.use_tc = false;
        if (n.is_input || n.dense_target || (int)v == g->info.output_node) continue;
        if (n.d.c % 8 != 0 || n.d.c < 16 || n.d.c > 1024) continue;
        const long long pixels = (long long)g->batch * n.d.h * n.d.w;
        bool ok = pixels < 1LL << 31;
        int n_blocks = 0;
        for (int e : n.in_edges) {
            const SrHostEdge& he = g->edges[e];
            const SrHostNode& s = g->nodes[he.d.src];
            if (he.d.kind != SR_EDGE_CONV) ok = false;
            else if (is_stem(g, he) && pixels * ((he.K + 7) / 8) >= (1LL << 32) - (1LL << 24)) ok = false;
            else if (s.d.c % 16 != 0 && !is_stem(g, he)) ok = false;
            else if (he.k_eff > 8) ok = false;
            else n_blocks += is_stem(g, he) ? 2 : he.k_eff * he.k_eff * (s.d.c / block_k(s.d.c));
        }
        if (ok && n_blocks >= 1 && n_blocks <= kMaxNodeKb) n.use_tc = true;
    }
}

sr_status sr_tc_plan(sr_graph* g, size_t& off)
{
    sr_tc_destroy(g);
    bool any = false;
    for (const SrHostNode& n : g->nodes) any |= n.use_tc;
    if (!any) return SR_OK;
    TcEngine* E = new TcEngine();
    g->tc = E;
    E->node_of.assign(g->nodes.size(), -1);
    E->stem_of_edge.assign(g->edges.size(), -1);
    auto take = [&](size_t bytes) {
        SrRegion r;
        r.offset = off;
        r.bytes = bytes;
        off = sr_align_up(off + bytes, 1024);
        return r;
    };
    // staging buffers
    for (size_t e = 0; e < g->edges.size(); ++e) {
        const SrHostNode& t = g->nodes[g->edges[e].d.tgt];
        if (!t.use_tc || !is_stem(g, g->edges[e])) continue;
        StemPlan S;
        S.edge = (int)e;
        S.Kp = stem_kp(g->edges[e].K);
        const size_t bytes = (size_t)g->batch * t.d.h * t.d.w * S.Kp * 2;
        S.buf[0] = take(bytes);
        S.buf[1] = take(bytes);
        E->stem_of_edge[e] = (int)E->stems.size();
        E->stems.push_back(S);
    }
    auto plan_of = [&](const std::vector<int>& nodes) {
        NodePlan P{};
        P.nodes = nodes;
        P.node = nodes[0];
        // sep / span: how many image rows / columns the taps that share one activation box are apart at most
        P.sep = 0;
        P.span = 0;
        for (int e : P.in_edges(g)) {
            const SrHostEdge& he = g->edges[e];
            if (is_stem(g, he)) continue;
            for (int r0 = 0; r0 < he.stride_eff; ++r0) {
                int lo = 1 << 20, hi = -(1 << 20);
                for (int t = 0; t < he.k_eff; ++t) {
                    int q, r;
                    tap_q(t, he.pad_eff, he.stride_eff, q, r);
                    if (r == r0) { lo = std::min(lo, q); hi = std::max(hi, q); }
                }
                if (hi >= lo) P.sep = P.span = std::max(P.sep, hi - lo);
            }
        }
        return P;
    };
    std::map<int, int> held;
    held[1] = g->sm_count;
    for (int cluster = 2; cluster <= kMaxParts; cluster *= 2) held[cluster] = clusters_held(g, cluster);
    // per launch group: tile sizes, K-blocks, ring geometry, work lists
    E->group_tiles.assign(g->groups.size(), {});
    int n_tiles = 0;
    for (size_t gi = 0; gi < g->groups.size(); ++gi) {
        const size_t first_plan = E->nodes.size();
        std::vector<int> members;
        // What can be chosen per plan: the most columns of its tiles (variants, as in kTileCols), and the parts of its items.
        struct Variant { NodePlan P; std::vector<TcTile> tiles; int box_kb = 1, w_slot = 1024, words = 0; long long plain = 0; mutable long long cycles[2][kMaxW + 1] = {}; };   // of an item; by crowded, slots (when they are asked for)
        struct Choice { int v, parts; };
        std::vector<std::vector<Variant>> variants;
        auto variant_of = [&](size_t m, int max_cols) {
            Variant V;
            V.P = E->nodes[members[m]];
            const SrHostNode& n = g->nodes[V.P.node];
            double blocks = 0, boxes = 0;
            for (int e : V.P.in_edges(g)) {
                const SrHostEdge& he = g->edges[e];
                const double cb = is_stem(g, he) ? 1.0 : (double)(g->nodes[he.d.src].d.c / block_k(g->nodes[he.d.src].d.c));
                const int kk = is_stem(g, he) ? 1 : he.k_eff, sd = is_stem(g, he) ? 1 : std::min(he.k_eff, he.stride_eff);
                blocks += cb * kk * kk;
                boxes += cb * sd * sd;
            }
            choose_tile(n.d.h, n.d.w, g->batch, max_cols, g->opt_tile_w, blocks / std::max(1.0, boxes), V.P);
            build_kblocks(g, E, V.P);
            V.tiles = node_tiles(g, V.P, members[m]);
            int bk_max = 16;
            for (const KbHost& kb : V.P.kbs) {
                V.box_kb = std::max(V.box_kb, kb.ring_kb);
                bk_max = std::max(bk_max, kb.bk);
                V.words += 2 * kb.x_load + 1;
            }
            V.w_slot = (int)sr_align_up((size_t)std::min(V.P.rows_total(g), 128) * std::max(64, bk_max) * 2, 1024);
            V.plain = item_cycles(g, V.P, 0.0);
            return V;
        };
        // Shared memory: what the parts of items exchange, the node tables, weight slots, and the rest for activation boxes, of which
        // two of the largest should fit.  A launch with several items per CTA is better off with room for a third box (a box read by
        // one tap only lasts 512 cycles of MMAs, and the one after it has to be on its way before that), one with an item or two per
        // CTA with a deeper weight ring.  Measured on B200, us per frame with six / five / four slots: six-node network at 256 samples
        // 146.3 / 143.0 / 147.8, ten-node at 128 115.1 / 112.7 / 117.9, stress graph at 32 253.9 / 246.2 / 250.7, deep window
        // 100.8 / 100.4 / 103.3; six-node hybrid at 37 samples (one item per CTA) 57.3 / 59.1 / 64.0.
        auto rings = [&](const std::vector<Choice>& ch, int table_words) {
            TcEngine::Launch L;
            int box_kb = 1, words = 0;
            size_t items = 0;
            bool widest = true;
            for (size_t m = 0; m < members.size(); ++m) {
                const Variant& V = variants[m][ch[m].v];
                box_kb = std::max(box_kb, V.box_kb);
                L.w_slot = std::max(L.w_slot, V.w_slot);
                words = std::max(words, V.words / ch[m].parts + 16);
                if (ch[m].parts > 1) L.exch = std::max(L.exch, (ch[m].parts - 1) * part_chunks(V.P, ch[m].parts) * 8192);
                items += V.tiles.size();
                widest = widest && ch[m].v <= 1;
            }
            L.table_bytes = (int)sizeof(TcNode) + (table_words ? table_words : words) * 16;
            const int sums = L.exch;
            for (;;) {
                const int avail = kSmemBudget - 1024 - kTables * L.table_bytes - L.exch;
                L.n_w = g->opt_b_units > 0 ? std::min(kMaxW, std::max(2, g->opt_b_units)) : widest && items > 2 * (size_t)g->sm_count ? 5 : kMaxW;
                while (g->opt_b_units == 0 && L.n_w > 6 && (avail - L.n_w * L.w_slot) / 1024 < 3 * box_kb) --L.n_w;
                while (L.n_w > 3 && (avail - L.n_w * L.w_slot) / 1024 < 2 * box_kb) --L.n_w;
                while (L.n_w > 2 && (avail - L.n_w * L.w_slot) / 1024 < box_kb) --L.n_w;
                L.ring_kb = (avail - L.n_w * L.w_slot) / 1024;
                L.fits = avail > 0 && L.ring_kb >= box_kb && box_kb <= 255;
                if (L.exch == 0 || (L.fits && L.n_w >= 6)) break;
                L.exch = 0;                                        // no room of its own: in the rings
            }
            if (sums > 0 && L.exch == 0 && sums > L.n_w * L.w_slot + L.ring_kb * 1024) L.fits = false;
            return L;
        };
        // cycles and lists of a choice; tail: the epilogue of the widest tile, which no other item hides (13 cycles a column)
        struct Bound { long long longest = 0, total = 0, tail = 0; size_t parts = 0, at = 0; };
        // A launch with more parts than CTAs is crowded; one of half the SMs has fewer of them (counted as if it had all, six-node
        // hybrid at 10 samples 32.8 -> 35.5 us per frame).
        int ctas_now = g->sm_count;
        auto crowded_by = [&](const std::vector<Choice>& ch) {
            size_t parts = 0;
            for (size_t m = 0; m < members.size(); ++m) parts += variants[m][ch[m].v].tiles.size() * ch[m].parts;
            return parts > (size_t)ctas_now;
        };
        auto cycles_of = [&](const Variant& V, int parts, const TcEngine::Launch& L, bool few, bool crowded) {
            if (!few) return V.plain;
            long long& cycles = V.cycles[crowded][L.n_w];
            if (cycles == 0) cycles = item_cycles(g, V.P, ring_cycles(L.n_w, crowded));
            return part_cycles(V.P, cycles, parts, L.exch == 0);
        };
        auto bound_of = [&](const std::vector<Choice>& ch, const TcEngine::Launch& L, bool few) {
            const bool crowded = crowded_by(ch);
            Bound b;
            for (size_t m = 0; m < members.size(); ++m) {
                const Variant& V = variants[m][ch[m].v];
                const long long c = cycles_of(V, ch[m].parts, L, few, crowded);
                b.total += c * ch[m].parts * (long long)V.tiles.size();
                b.parts += V.tiles.size() * ch[m].parts;
                b.tail = std::max(b.tail, 13ll * V.P.nl * V.P.lane_cols / ch[m].parts);
                if (c > b.longest) { b.longest = c; b.at = m; }
            }
            return b;
        };
        auto work_of = [&](const std::vector<Choice>& ch, const TcEngine::Launch& L, bool few, bool tiles) {
            const bool crowded = crowded_by(ch);
            // longest first; all items of a plan are as long
            std::vector<std::pair<long long, size_t>> order;
            size_t n = 0;
            for (size_t m = 0; m < members.size(); ++m) {
                const Variant& V = variants[m][ch[m].v];
                order.push_back({-cycles_of(V, ch[m].parts, L, few, crowded), m});
                n += V.tiles.size();
            }
            std::sort(order.begin(), order.end());
            std::vector<TcWork> work;
            work.reserve(n);
            for (const auto& [c, m] : order)
                for (const TcTile& t : variants[m][ch[m].v].tiles) work.push_back(TcWork{-c, ch[m].parts, tiles ? t : TcTile{}});
            return work;
        };
        // A launch with many items per SM takes the widest tiles (fewest copies per MMA).  For one with few, the split that ends first
        // by the estimate is sought: from the same columns for every plan, the plan whose items take longest gets narrower
        // tiles (of the next or the second next width) or has its items cut into twice as many parts, whichever leaves the shortest
        // bound, again and again.  The line lies at four items of the widest tiles per SM.  At three of them launches of joined nodes had
        // items too long to share out: networks of the CIFAR10 kind with six / four added layers, us per pass of 16 frames with the line at
        // three / four / five, at 40 samples 605 / 447 / 448, at 64 721 / 659 / 755 (in twos 658), at 96 857 / 857 / 906; at 48 542 / 479 / 480, at 72
        // 637 / 605 / 631; stress graph at 6 1012 / 891 / 895; two added layers at 80 485 / 498 / 498; six-node at 48 to 80, ten-node at 40 to 64 samples
        // equal.
        std::vector<Choice> best;
        int best_cluster = 1, best_grid = 0;
        long long best_cost = -1;
        bool few = false;
        auto search = [&](const std::vector<std::vector<int>>& plans) {
            E->nodes.resize(first_plan);
            members.clear();
            for (const std::vector<int>& nodes : plans) {
                members.push_back((int)E->nodes.size());
                E->nodes.push_back(plan_of(nodes));
            }
            variants.assign(members.size(), std::vector<Variant>(kVariants));
            best_cost = -1;
            // (the widths that are looked at)
            auto make = [&](int v) {
                for (size_t m = 0; m < members.size(); ++m) variants[m][v] = variant_of(m, kTileCols[v]);
            };
            make(0);
            size_t widest_items = 0;
            for (size_t m = 0; m < members.size(); ++m) widest_items += variants[m][0].tiles.size();
            few = g->opt_b_units == 0 && g->opt_tile_w == 0 && g->compact == 0 && widest_items <= 4 * (size_t)g->sm_count;
            for (int v = 1; v < kVariants && few; ++v) make(v);
            for (int start = 0; start < kVariants && !members.empty(); ++start) {
                if (start == 1 && !few) continue;              // (ten-node windows of 8 frames, 128 samples: 1842 -> 1905 us per pass with them)
                if (start > 0 && !few) make(start);
                size_t items = 0;
                for (size_t m = 0; m < members.size(); ++m) items += variants[m][start].tiles.size();
                for (int cluster = 1; cluster <= (few ? kMaxParts : 1); cluster *= 2)
                    // all SMs, or half of them: then the next launch starts up on the others
                    for (int half = 0; half < (few ? 2 : 1); ++half) {
                        const int ctas = (half ? std::min(held[cluster], g->sm_count / 2 / cluster) : held[cluster]) * cluster;
                        ctas_now = half ? ctas : g->sm_count;
                        std::vector<Choice> ch(members.size(), Choice{start, 1});
                        for (;;) {
                            const TcEngine::Launch L = rings(ch, 0);
                            const Bound b = bound_of(ch, L, few);
                            const int grid = (int)std::min<size_t>((b.parts + cluster - 1) / cluster * cluster, ctas);
                            const long long fixed = (few ? b.tail : 0) + (grid > g->sm_count / 2 ? kLateStart : 0) + (cluster > 1 ? kClusterStart : 0);
                            if (L.fits && (best_cost < 0 || std::max(b.longest, b.total / grid) + fixed < best_cost)) {
                                const std::vector<TcWork> work = work_of(ch, L, few, false);
                                const long long limit = best_cost < 0 ? kAnyLoad : best_cost - fixed;
                                const long long span = cluster > 1 ? spread_split(work, grid, cluster, nullptr, limit) : spread_items(work, work.size(), grid, nullptr, limit);
                                if (span >= 0 && (best_cost < 0 || span + fixed < best_cost)) {
                                    best_cost = span + fixed;
                                    best = ch;
                                    best_cluster = cluster;
                                    best_grid = grid;
                                }
                            }
                            if (!few) break;
                            const Choice now = ch[b.at];
                            const std::vector<Variant>& of = variants[b.at];
                            Choice ways[3] = {Choice{now.v, now.parts * 2}, Choice{now.v + 1, now.parts}, Choice{now.v + 2, now.parts}};
                            while (ways[1].v < kVariants - 1 && of[ways[1].v].tiles.size() == of[now.v].tiles.size()) ++ways[1].v;
                            ways[2].v = ways[1].v + 1;
                            int way = -1;
                            long long shortest = 0;
                            for (int w = 0; w < 3; ++w) {
                                if (w == 0 && (ways[0].parts > cluster || (int)of[now.v].P.kbs.size() < 2 * ways[0].parts)) continue;
                                if (w > 0 && (ways[w].v >= kVariants || of[ways[w].v].tiles.size() == of[now.v].tiles.size())) continue;
                                ch[b.at] = ways[w];
                                const Bound c = bound_of(ch, rings(ch, 0), few);
                                const long long t = std::max(c.longest, c.total / ctas) + c.tail;
                                if (way < 0 || t < shortest) { way = w; shortest = t; }
                            }
                            if (way < 0) break;
                            ch[b.at] = ways[way];
                        }
                    }
                if (items > 8 * (size_t)g->sm_count) break;            // plenty of items: smaller tiles only cost copies
            }
        };
        // Joined as far as they go, or in twos: the launch that ends first by the estimate (with few tiles, more and shorter items may; joined
        // where it is 3 % ahead).  Networks of the CIFAR10 kind with six added layers, us per pass of 16 frames in twos / joined: at 4
        // samples 181 / 216, 8 248 / 233, 16 277 / 384, 32 528 / 431, 64 658 / 719, 96 940 / 857, 128 1271 / 1120, 256 2506 / 2204; with four: 1 120 / 133,
        // 8 347 / 214, 24 348 / 321, 64 578 / 542, 128 967 / 856.
        const int most = !g->opt_tc_fuse || g->compact > 1 ? 1 : g->compact > 0 ? 2 : kMaxFused;
        const auto joined = join_nodes(g, g->groups[gi], most), twos = join_nodes(g, g->groups[gi], std::min(most, 2));
        search(joined);
        if (joined != twos) {
            const std::vector<NodePlan> plans(E->nodes.begin() + first_plan, E->nodes.end());
            auto kept = std::make_tuple(std::move(members), std::move(variants), best, best_cluster, best_grid, best_cost, few);
            search(twos);
            const long long cost = std::get<5>(kept);
            if (best_cost < 0 || (cost >= 0 && cost * 103 <= best_cost * 100)) {
                E->nodes.resize(first_plan);
                E->nodes.insert(E->nodes.end(), plans.begin(), plans.end());
                std::tie(members, variants, best, best_cluster, best_grid, best_cost, few) = std::move(kept);
            }
        }
        for (int ni : members)
            for (int v : E->nodes[ni].nodes) E->node_of[v] = ni;
        TcEngine::Launch L;
        if (!members.empty()) {
            if (best_cost < 0) return SR_ERR_UNSUPPORTED;
            int words = 1;
            for (size_t m = 0; m < members.size(); ++m) {
                NodePlan& P = E->nodes[members[m]];
                P = variants[m][best[m].v].P;
                P.n_parts = best[m].parts;
                build_groups(g, P);
                for (const NodePlan::Part& q : P.parts) {
                    int n_act = 0;
                    for (const KbHost& kb : q.kbs) n_act += kb.x_load;
                    words = std::max(words, 2 * count_bursts(q) + n_act);
                }
            }
            L = rings(best, words);
            if (!L.fits) return SR_ERR_UNSUPPORTED;
            // Work lists: the items go, longest first, to the CTA with the least work so far; CTA c walks column c of a
            // matrix with one row per round (entries of node -1 pad the shorter columns).  Unless the lists are asked to be
            // static, the smallest items - a fifth of the work, if the launch has more than two items per CTA - stay out of
            // the matrix and follow it as one shared list (see the kernel).
            ctas_now = best_grid > g->sm_count / 2 ? g->sm_count : best_grid;
            const std::vector<TcWork> work = work_of(best, L, few, true);
            std::vector<std::vector<TcTile>> lists;
            size_t n_matrix = work.size(), n_rows = 0;
            if (best_cluster > 1) {
                if (!place_split(work, best_grid, best_cluster, lists)) return SR_ERR_UNSUPPORTED;
                while (std::all_of(lists.end() - best_cluster, lists.end(), [](const auto& l) { return l.empty(); })) lists.resize(lists.size() - best_cluster);
                L.cluster = best_cluster;
            } else {
                if (g->opt_tc_lists == 0 && work.size() > 2 * (size_t)best_grid) {
                    long long total = 0, tail = 0;
                    for (auto& it : work) total += it.cycles;
                    while (n_matrix > (size_t)best_grid && (tail + work[n_matrix - 1].cycles) * 5 <= total) tail += work[--n_matrix].cycles;
                }
                spread_items(work, n_matrix, best_grid, &lists);
            }
            for (auto& l : lists) n_rows = std::max(n_rows, l.size());
            for (size_t r = 0; r < n_rows; ++r)
                for (auto& l : lists) E->group_tiles[gi].push_back(r < l.size() ? l[r] : TcTile{-1, 0, 0, 0, 0, 0, 0, 0});
            L.grid = (int)lists.size();
            for (int ni : members)
                for (const KbHost& kb : E->nodes[ni].kbs) L.masked = L.masked || E->nodes[ni].quarters_of(g, kb) != 15u;
            L.n_own = (int)E->group_tiles[gi].size();
            for (size_t i = n_matrix; i < work.size(); ++i) E->group_tiles[gi].push_back(work[i].tile);
        }
        L.first_tile = n_tiles;
        n_tiles += (int)E->group_tiles[gi].size();
        E->launches.push_back(L);
    }
    for (NodePlan& P : E->nodes) P.wcat = take((size_t)P.rows_total(g) * P.k_total * 2);
    E->n_tiles = n_tiles;
    // tensor maps, as many as there can be: two parities per activation box, two widths per run of weights
    size_t n_maps = 1, n_words = 0;
    for (const NodePlan& P : E->nodes) {
        n_maps += 2 * P.runs.size();
        for (const NodePlan::Part& q : P.parts) {
            const size_t boxes = std::count_if(q.kbs.begin(), q.kbs.end(), [](const KbHost& kb) { return kb.x_load; });
            n_maps += 2 * boxes;
            n_words += sizeof(TcNode) / 16 + 2 * count_bursts(q) + boxes;
        }
    }
    E->r_maps = take(sizeof(CUtensorMap) * n_maps);
    E->r_tables = take(16 * n_words);
    E->r_tiles = take(sizeof(TcTile) * (size_t)std::max(1, n_tiles));
    return SR_OK;
}

sr_status sr_tc_bind(sr_graph* g)
{
    TcEngine* E = eng(g);
    if (!E) return SR_OK;
    EncodeTiledFn encode = encode_fn();
    if (!encode) return SR_ERR_CUDA;
    // Always the largest shared-memory partition: otherwise the SM is configured with the smallest partition that holds
    // this kernel's CTA, which can leave a few hundred bytes, and the frame's other kernels cannot run beside it.
    for (auto kernel : {sr_tc_group_kernel<false, false>, sr_tc_group_kernel<false, true>, sr_tc_group_kernel<true, false>, sr_tc_group_kernel<true, true>})
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            return SR_ERR_CUDA;
    char* ws = g->ws;
    std::vector<CUtensorMap> maps;
    std::map<std::tuple<uintptr_t, int, int, int, int, int, int, int, int>, int> cache;
    // 4-D activation view: dims (C, W', H', B), box (bk, tw, rows, tb)
    auto act_map = [&](char* base, int C, int Wv, int Hv, size_t stride_w, size_t stride_h, size_t stride_b, int bk,
                       int tw, int rows, int tb) -> int {
        auto key = std::make_tuple((uintptr_t)base, C, Wv, Hv, (int)stride_w, bk, tw, rows, tb);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
        if (tw > 256 || rows > 256 || tb > 256) return -1;
        CUtensorMap m;
        cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)Wv, (cuuint64_t)Hv, (cuuint64_t)g->batch};
        cuuint64_t strides[3] = {(cuuint64_t)stride_w, (cuuint64_t)stride_h, (cuuint64_t)stride_b};
        cuuint32_t box[4] = {(cuuint32_t)bk, (cuuint32_t)tw, (cuuint32_t)rows, (cuuint32_t)tb};
        cuuint32_t es[4] = {1, 1, 1, 1};
        if (encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   swizzle_of(bk), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return -1;
        maps.push_back(m);
        cache[key] = (int)maps.size() - 1;
        return (int)maps.size() - 1;
    };
    std::vector<uint4> dt;                             // per node: TcNode, bursts (two words each), activation boxes
    for (NodePlan& P : E->nodes) {
        const SrHostNode& n = g->nodes[P.node];
        TcNode d{};
        d.H = n.d.h; d.W = n.d.w; d.C = n.d.c;
        d.n_nodes = (int)P.nodes.size();
        d.rows = d.n_nodes > 1 ? n.d.c : 0;
        for (int q = 0; q < d.n_nodes; ++q) {
            const SrHostNode& nq = g->nodes[P.nodes[q]];
            for (int par = 0; par < 2; ++par) d.state[q][par] = ws + nq.state[par].offset;
            d.bias[q] = reinterpret_cast<const float*>(ws + nq.bias.offset);
            if (nq.d.act == 1) d.relu |= 1 << q;
        }
        d.tw = P.tw; d.th = P.th; d.tb = P.tb; d.sep = P.sep;
        d.nl = P.nl;
        d.lane_cols = P.lane_cols;
        d.n_parts = P.n_parts;
        d.part_chunks = part_chunks(P, P.n_parts);
        const int rows128 = std::min(P.rows_total(g), 128);
        if (P.k_total > 65535 || (int)P.runs.size() > kMaxRuns) return SR_ERR_UNSUPPORTED;
        // one 3-D view per run: (channels of a block, output channels, blocks of the run); a box of two blocks lands in
        // shared memory block after block, each an ordinary K-major swizzled tile
        std::vector<TcRun> runs;
        for (size_t r = 0; r < P.runs.size(); ++r) {
            const WRun& R = P.runs[r];
            int map_of[2] = {0, -1};
            for (int nb = 1; nb <= (R.bk == 64 ? 1 : 2); ++nb) {
                CUtensorMap m;
                cuuint64_t dims[3] = {(cuuint64_t)R.bk, (cuuint64_t)P.rows_total(g), (cuuint64_t)R.n_blocks};
                cuuint64_t strides[2] = {(cuuint64_t)P.k_total * 2, (cuuint64_t)R.bk * 2};
                cuuint32_t box[3] = {(cuuint32_t)R.bk, (cuuint32_t)rows128, (cuuint32_t)nb};
                cuuint32_t es[3] = {1, 1, 1};
                if (nb > R.n_blocks) break;
                if (encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, ws + P.wcat.offset + (size_t)R.first_col * 2, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(R.bk), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                    return SR_ERR_CUDA;
                maps.push_back(m);
                map_of[nb - 1] = (int)maps.size() - 1;
            }
            if (maps.size() > 65535) return SR_ERR_UNSUPPORTED;
            TcRun t{};
            t.map1 = (uint16_t)map_of[0];
            t.map2 = (uint16_t)(map_of[1] < 0 ? map_of[0] : map_of[1]);   // equal: no group of two blocks
            t.bytes16 = (uint16_t)((size_t)rows128 * R.bk * 2 >> 4);
            runs.push_back(t);
        }
        for (NodePlan::Part& q : P.parts) {
            TcNode e = d;
            e.part = (int)(&q - P.parts.data());
            if (q.wgroups.size() > 32 * sizeof(e.pairs) / sizeof(e.pairs[0])) return SR_ERR_UNSUPPORTED;
            int run = -1;
            for (size_t gi = 0; gi < q.wgroups.size(); ++gi) {
                const WGroup& wg = q.wgroups[gi];
                if (wg.run != run) {
                    run = wg.run;
                    e.runs[e.n_runs] = runs[run];
                    e.runs[e.n_runs++].blk0 = (uint16_t)wg.blk;
                }
                e.runs[e.n_runs - 1].n_groups += 1;
                if (wg.n == 2) e.pairs[gi / 32] |= 1u << (gi % 32);
            }
            std::vector<TcAct> da;
            struct KbIssue { uint32_t x_off16, x_hi, w_hi; };
            std::vector<KbIssue> dm;                      // per K-block: what its MMAs need
            for (const KbHost& kb : q.kbs) {
                const SrHostEdge& he = g->edges[kb.edge];
                const SrHostNode& s = g->nodes[he.d.src];
                TcAct kl{};
                KbIssue km{};
                int map0 = -1, map1 = -1, qxv = 0, qyv = 0;
                kl.flags = (uint8_t)(he.R ? 1 : 0);
                km.w_hi = desc_hi_of(kb.bk);
                const size_t x_bytes = (size_t)kb.bk * 2 * kb.x_width * kb.x_rows * P.tb;
                const size_t sbo_bytes = (size_t)(P.flat ? 8 : kb.x_width) * kb.bk * 2;
                if ((x_bytes >> 4) > 65535 || (sbo_bytes >> 4) > 0x3FFF) return SR_ERR_UNSUPPORTED;
                kl.x_bytes16 = (uint16_t)(x_bytes >> 4);
                kl.ring_kb = (uint16_t)kb.ring_kb;
                km.x_hi = (km.w_hi & ~0x3FFFu) | (uint32_t)(sbo_bytes >> 4);
                km.x_off16 = (uint32_t)(((size_t)kb.x_shift * kb.bk * 2) >> 4);
                if (km.x_off16 + 4 > 65535) return SR_ERR_UNSUPPORTED;
                dm.push_back(km);
                if (!kb.x_load) continue;                // reads the box the first tap of its class loads
                if (kb.stem) {
                    const StemPlan& S = E->stems[kb.stem_index];
                    for (int par = 0; par < 2; ++par)
                        (par ? map1 : map0) = act_map(ws + S.buf[par].offset, S.Kp, n.d.w, n.d.h, (size_t)S.Kp * 2,
                                                      (size_t)n.d.w * S.Kp * 2, (size_t)n.d.h * n.d.w * S.Kp * 2, kb.bk, kb.x_width, kb.x_rows, P.tb);
                } else {
                    // input pixel = stride * (output pixel + q) + r, q = floor((tap - pad) / stride), r the residue:
                    // the residue-class view of the source makes the tap a dense box starting at (w0 + qx, h0 + qy)
                    const int st = he.stride_eff;
                    const int ry = kb.box_ry, rx = kb.box_rx;
                    const int Hv = (s.d.h - ry + st - 1) / st, Wv = (s.d.w - rx + st - 1) / st;
                    if (Hv <= 0 || Wv <= 0) return SR_ERR_UNSUPPORTED;
                    for (int par = 0; par < 2; ++par) {
                        char* base = ws + s.state[par].offset + ((size_t)ry * s.d.w + rx) * s.d.c * 2;
                        (par ? map1 : map0) = act_map(base, s.d.c, Wv, Hv, (size_t)st * s.d.c * 2, (size_t)st * s.d.w * s.d.c * 2,
                                                      (size_t)s.d.h * s.d.w * s.d.c * 2, kb.bk, kb.x_width, kb.x_rows, P.tb);
                    }
                    qxv = kb.box_qx; qyv = kb.box_qy;
                }
                if (map0 < 0 || map1 < 0) return SR_ERR_CUDA;
                if (map0 > 65535 || map1 > 65535 || qxv < -128 || qxv > 127 || qyv < -128 || qyv > 127 || kb.c0 / 16 > 255) return SR_ERR_UNSUPPORTED;
                kl.x_map0 = (uint16_t)map0; kl.x_map1 = (uint16_t)map1;
                kl.qx = (int8_t)qxv; kl.qy = (int8_t)qyv;
                kl.c0_16 = (uint8_t)(kb.c0 / 16);
                da.push_back(kl);
            }
            // Bursts: two consecutive weight groups if their K-blocks are equally wide, else one.
            std::vector<TcBurst> db;
            uint32_t begun = 0;                           // quarters of the lanes that an earlier K-block of the part writes
            for (size_t gi = 0; gi < q.wgroups.size();) {
                const int i0 = q.wgroups[gi].first_kb, bk = q.kbs[i0].bk;
                const bool two = one_burst(q, gi);
                TcBurst b{};
                b.w_hi = dm[i0].w_hi;
                b.l1_off16 = (uint16_t)(8 * bk * 2 >> 4);                          // a lane's window lies 8 pixels after the one before
                b.w1_off16 = (uint16_t)(bk == 64 ? 4 : rows128 * bk * 2 >> 4);     // a block of 64 channels is two segments, a narrower one is one
                b.flags = (two ? kBuTwo : 0) | (bk == 16 ? kBuK16 : 0);
                for (int half = 0; half < (two ? 2 : 1); ++half) {
                    const WGroup& wg = q.wgroups[gi + half];
                    const KbHost& kb0 = q.kbs[wg.first_kb];
                    b.x_hi[half] = dm[wg.first_kb].x_hi;
                    if (kb0.x_load) {
                        b.flags |= half ? kBuNew1 : kBuNew0;
                        b.size[half] = (uint8_t)kb0.ring_kb;
                    }
                    if (q.kbs[wg.first_kb + wg.n - 1].x_release) b.flags |= half ? kBuLast1 : kBuLast0;
                    const uint32_t used = P.quarters_of(g, kb0), first = used & ~begun;
                    b.flags |= (~used & 15u) << (kBuOff + 4 * half);
                    if (first == used) b.flags |= half ? kBuFirst1 : kBuFirst0;
                    else b.flags |= first << (kBuMix + 4 * half);
                    begun |= used;
                    for (int sg = 0; sg < (bk == 64 ? 2 : wg.n); ++sg) {
                        b.x_off16[half * 2 + sg] = (uint16_t)(bk == 64 ? dm[wg.first_kb].x_off16 + 4 * sg : dm[wg.first_kb + sg].x_off16);
                        b.flags |= 1u << (half * 2 + sg);
                    }
                }
                db.push_back(b);
                gi += two ? 2 : 1;
            }
            e.n_bu = (int)db.size();
            e.n_act = (int)da.size();
            for (const NodePlan::Part& other : P.parts)
                for (const KbHost& kb : other.kbs) e.part_lanes |= P.quarters_of(g, kb) << 4 * (&other - P.parts.data());
            const size_t at = dt.size(), words = sizeof(TcNode) / 16;
            q.table_off = (int)at;
            q.table_words = (int)(words + 2 * db.size() + da.size());
            dt.resize(at + q.table_words);
            std::memcpy(dt.data() + at, &e, sizeof(e));
            std::memcpy(dt.data() + at + words, db.data(), db.size() * sizeof(TcBurst));
            std::memcpy(dt.data() + at + words + 2 * db.size(), da.data(), da.size() * sizeof(TcAct));
        }
    }
    if (maps.size() * sizeof(CUtensorMap) > E->r_maps.bytes || dt.size() * sizeof(uint4) > E->r_tables.bytes) return SR_ERR_UNSUPPORTED;
    E->n_maps = (int)maps.size();
    std::vector<TcTile> tiles;
    for (auto& v : E->group_tiles) tiles.insert(tiles.end(), v.begin(), v.end());
    for (TcTile& t : tiles)
        if (t.node >= 0) {
            const NodePlan::Part& q = E->nodes[t.node].parts[t.words];
            t.node = q.table_off;
            t.words = q.table_words;
        }
    g->stems.clear();
    for (const StemPlan& S : E->stems) {
        const SrHostEdge& he = g->edges[S.edge];
        const SrHostNode& s = g->nodes[he.d.src];
        const SrHostNode& t = g->nodes[he.d.tgt];
        SrStem d{};
        d.dst[0] = ws + S.buf[0].offset;
        d.dst[1] = ws + S.buf[1].offset;
        d.slot = s.input_slot;
        d.R = he.R;
        d.Hs = s.d.h; d.Ws = s.d.w; d.Cs = s.d.c; d.Ho = t.d.h; d.Wo = t.d.w;
        d.k = he.k_eff; d.stride = he.stride_eff; d.pad = he.pad_eff; d.Kp = S.Kp; d.K = he.K;
        g->stems.push_back(d);
    }
    auto up = [&](const SrRegion& r, const void* p, size_t bytes) {
        return bytes == 0 || cudaMemcpy(ws + r.offset, p, bytes, cudaMemcpyHostToDevice) == cudaSuccess;
    };
    if (!up(E->r_maps, maps.data(), maps.size() * sizeof(CUtensorMap)) ||
        !up(E->r_tables, dt.data(), dt.size() * sizeof(uint4)) ||
        !up(E->r_tiles, tiles.data(), tiles.size() * sizeof(TcTile)))
        return SR_ERR_CUDA;
    return SR_OK;
}

sr_status sr_tc_set_weights(sr_graph* g, int edge, const float* w_eff)
{
    TcEngine* E = eng(g);
    if (!E) return SR_ERR_STATE;
    const SrHostEdge& he = g->edges[edge];
    const int ni = E->node_of[he.d.tgt];
    if (ni < 0) return SR_ERR_STATE;
    const NodePlan& P = E->nodes[ni];
    const SrHostNode& t = g->nodes[he.d.tgt];
    // the node's weight matrix keeps its columns in the order the K loop walks them: every K-block of this edge
    // takes its slice [C_out][block width] of the edge's own matrix (a staged edge: all of it, zero-padded)
    // (K-blocks of an edge that follow one another go in one copy)
    bool any = false;
    std::vector<uint16_t> h;
    auto row_of = [&](const KbHost& kb) {
        for (const auto& u : kb.users)
            if (u.first == edge) return u.second;
        return -1;
    };
    for (size_t i = 0; i < P.kbs.size();) {
        const int row_off = row_of(P.kbs[i]);
        if (row_off < 0) { ++i; continue; }
        size_t end = i;
        int width = 0;
        while (end < P.kbs.size() && row_of(P.kbs[end]) == row_off) width += P.kbs[end++].bk;
        h.assign((size_t)t.d.c * width, 0);
        int col = 0;
        for (size_t j = i; j < end; ++j) {
            const KbHost& kb = P.kbs[j];
            const int n_src = kb.stem ? std::max(0, std::min(kb.bk, he.K - kb.src_col)) : kb.bk;
            for (int co = 0; co < t.d.c; ++co) {
                const float* src = w_eff + (size_t)co * he.K + kb.src_col;
                uint16_t* dst = &h[(size_t)co * width + col];
                for (int k = 0; k < n_src; ++k) {                 // to the nearest bfloat16, ties to even; NaN stays NaN
                    uint32_t u;
                    std::memcpy(&u, &src[k], 4);
                    const uint32_t r = (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
                    dst[k] = (uint16_t)((u & 0x7FFFFFFFu) > 0x7F800000u ? 0x7FFFu : r);
                }
            }
            col += kb.bk;
        }
        char* dst = g->ws + P.wcat.offset + ((size_t)row_off * P.k_total + P.kbs[i].k_off) * 2;
        if (cudaMemcpy2D(dst, (size_t)P.k_total * 2, h.data(), (size_t)width * 2, (size_t)width * 2, t.d.c, cudaMemcpyHostToDevice) != cudaSuccess)
            return SR_ERR_CUDA;
        any = true;
        i = end;
    }
    if (!any) return SR_ERR_STATE;
    return SR_OK;
}

bool sr_tc_stages(const sr_graph* g, int edge)
{
    return g->nodes[g->edges[edge].d.tgt].use_tc && is_stem(g, g->edges[edge]);
}

int sr_tc_launch_group(sr_graph* g, int group, SrFollow how, cudaStream_t s)
{
    TcEngine* E = eng(g);
    if (!E || E->group_tiles[group].empty()) return 0;
    const TcEngine::Launch& L = E->launches[group];
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    bool timed = g->opt_time_tc != 0 && cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
    if (timed) {
        if (E->ev_used + 2 > E->ev.size()) {
            if (E->ev.size() >= 4096) timed = false;
            else
                for (int i = 0; i < 2; ++i) {
                    cudaEvent_t e = nullptr;
                    if (cudaEventCreate(&e) != cudaSuccess) { timed = false; break; }
                    E->ev.push_back(e);
                }
        }
        if (timed && E->ev_used + 2 <= E->ev.size()) cudaEventRecord(E->ev[E->ev_used], s);
        else timed = false;
    }
    TcParams P{};
    P.maps = reinterpret_cast<const CUtensorMap*>(g->ws + E->r_maps.offset);
    P.tables = reinterpret_cast<const uint4*>(g->ws + E->r_tables.offset);
    P.tiles = reinterpret_cast<const TcTile*>(g->ws + E->r_tiles.offset) + L.first_tile;
    P.fr = g->frame;
    P.error = reinterpret_cast<int*>(g->ws + g->r_flags.offset);
    P.sched = g->opt_tc_lists == 0 ? P.error + 16 : nullptr;
    P.wait_limit = (long long)g->opt_wait_ms * 2000000LL;
    P.n_tiles = (int)E->group_tiles[group].size();
    P.n_own = L.n_own;
    P.B = g->batch;
    P.table_bytes = L.table_bytes;
    P.n_w = L.n_w;
    P.w_slot = L.w_slot;
    P.ring_kb = L.ring_kb;
    P.exch_off = L.exch_off();
    P.follow = how.flags();
    if (L.cluster) {
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = cluster_config(L.grid, L.cluster, L.smem(), s, how.early && !timed, at);
        cudaLaunchKernelEx(&cfg, L.masked ? sr_tc_group_kernel<true, true> : sr_tc_group_kernel<true, false>, P);
    } else {
        sr_launch(L.masked ? sr_tc_group_kernel<false, true> : sr_tc_group_kernel<false, false>, L.grid, kThreads, L.smem(), s, how.early && !timed, P);
    }
    if (timed) {
        cudaEventRecord(E->ev[E->ev_used + 1], s);
        E->ev_used += 2;
    }
    return 1;
}

void sr_tc_describe(const sr_graph* g, int group, sr_launch_plan* out)
{
    *out = sr_launch_plan{};
    const TcEngine* E = eng(g);
    if (!E || E->group_tiles[group].empty()) return;
    const TcEngine::Launch& L = E->launches[group];
    for (const TcTile& t : E->group_tiles[group]) {
        if (t.node < 0) continue;
        const NodePlan& P = E->nodes[t.node];
        out->items += t.words == 0;
        out->parts = std::max(out->parts, P.n_parts);
        out->columns = std::max(out->columns, P.nl * P.lane_cols);
        out->joined = std::max(out->joined, (int)P.nodes.size());
    }
    out->ctas = L.grid;
    out->cluster = std::max(1, L.cluster);
    out->sums_in_rings = out->parts > 1 && L.exch == 0;
    out->masked = L.masked;
}

// Sum of the event-timed durations of the tensor-core group launches since the last call (synchronises).
sr_status sr_tc_timing(sr_graph* g, double* ms, long long* launches)
{
    TcEngine* E = eng(g);
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

bool sr_tc_group_has_work(const sr_graph* g, int group)
{
    TcEngine* E = eng(g);
    return E && !E->group_tiles[group].empty();
}

void sr_tc_destroy(sr_graph* g)
{
    if (g && g->tc) {
        for (cudaEvent_t e : eng(g)->ev) cudaEventDestroy(e);
        delete eng(g);
        g->tc = nullptr;
    }
}
