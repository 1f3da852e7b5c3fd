// Internal structures of the streaming-rollout library: host-side graph, device-side tables.
#pragma once
#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/sr_rollout.h"

#define SR_MAX_INPUTS 4

// ------------------------------------------------------------------ tables read by the kernels
// One incoming edge of a node, as the CUDA-core ("direct") kernels see it.  A pooled edge
// (conv k, stride s, then 2x2 average) is stored as the single convolution it equals:
// kernel k+s, stride 2s, same padding, box-filtered weights.
struct SrDevEdge {
    const void* src[2];     // source state, frame parity 0 / 1
    const float* w;         // conv: [k*k*Cs][C_out] (K-major rows, channels contiguous); dense: [C_out][K]
    int32_t Hs, Ws, Cs;     // source shape
    int32_t kind, k, stride, pad;
    int32_t R;              // 1: read frame t, 0: read frame t+1 (Eq. 2)
    int32_t K;              // reduction length of this edge
    int32_t src_is_input;
};

struct SrDevNode {
    void* state[2];
    const float* bias;
    int32_t H, W, C, act;
    int32_t first_edge, n_edges;     // range in the SrDevEdge table
    int32_t is_output;
    int32_t untiled;                 // conv nodes: 0: conv_tile takes them; 1: conv_item; 2 (bf16), 4 (fp32): conv_item on
                                     // conv_tile's items, in the kernel for weights that are not finite
};

// One block's work in a grouped direct launch.
struct SrDirectItem {
    int32_t node;        // index into the SrDevNode table
    int32_t b0;          // first sample (dense nodes: sample chunk); its complement: four pixels per thread (conv_tile)
    int32_t p0;          // first pixel (conv nodes) or first output channel (dense nodes)
    int32_t pad_;        // conv nodes on conv_tile: first channel | log2(channel quads per block) << 24 | 1 << 30 (slices of the reduction)
};

// Dense / mean-dense nodes as the head kernels see them: passed as kernel parameters.
#define SR_HEAD_EDGES 6
#define SR_HEAD_NODES 6
struct SrHeadEdge {
    const void* src[2];
    const float* w;              // [C_out][K]
    int32_t HW, Cs, kind, R, K, slot;        // slot: the source's place among the input nodes, or -1
};
struct SrHeadNode {
    void* state[2];
    const float* bias;
    int32_t C, act, is_output, n_edges;
    int32_t has_mean, mean_q, pad_[2];       // mean_q: outputs per warp (nodes with a mean-dense edge)
    SrHeadEdge edges[SR_HEAD_EDGES];
};

// The nodes of sr_wide_head_kernel: their edges lie in one list.
#define SR_WIDE_EDGES 48
#define SR_WIDE_NODES 8
struct SrWideNode {
    void* state[2];
    const float* bias;
    int32_t C, act, is_output, n_edges;
    int32_t first_edge, q;                   // q: outputs per warp
};

// What a launch needs to know about its frame.  Plain launches carry it by value; launches recorded in a CUDA graph read it
// from a control block in device memory, which lets the recorded sequence be replayed for later frames.
struct SrFrameCtl {
    int64_t t;                            // frame updates completed since reset
    int64_t run_t;                        // frame updates completed inside the current step / run call
    const void* in_base[SR_MAX_INPUTS];   // frame used by update run_t is in_base + run_t * in_stride_bytes
    int64_t in_stride_bytes[SR_MAX_INPUTS];
    float* out_base;                      // output of update run_t goes to out_base + run_t * out_stride (floats); may be null
    int64_t out_stride;
};

struct SrFrameArgs {
    const SrFrameCtl* ctl;                // null: the values are in v
    int64_t off;                          // frames to add to t and run_t
    SrFrameCtl v;
};

// How the launches of a rollout follow one another in ONE stream (programmatic dependent launch): a kernel launched with
// `early` may be scheduled as soon as every block of the kernel before it has let its successor start, and
// sr_wait_for_predecessor returns when that kernel has completed and its writes are visible.
//   main     waits before it touches anything an earlier kernel reads or writes;
//   beside   does not depend on the main kernel of its group and runs beside it: the main kernel (`late`) lets its successor
//            start only after its own wait, so everything before the group is complete when a beside kernel starts; it does its
//            work at once and ONE of its blocks waits for its predecessor at the end, so that it completes after the main kernel
//            and whoever waits for it has waited for both.
// What the blocks of a beside kernel that never wait rely on: the programming model promises visibility to whoever executes
// griddepcontrol.wait, and none of them does.  They read what kernels ahead of the main one wrote.  Those had completed, with
// their writes performed for the whole device, when the main kernel's wait returned; every block of the main kernel signals
// after that wait, and a beside kernel starts only once all of them have.  So the values stand in L2 when it starts, and what is
// left is a line that its SM's L1 may hold from an earlier frame.  What a beside kernel reads once it reads past L1
// (sr_load_past_l1); one that reads a value many times (staging, convolutions) begins with a fence, an acquire at device scope,
// which drops those lines (and takes 0.5 us, or 1 us beside a running main kernel).  Nothing is read through the non-coherent path
// but weights, which only the host writes.
// (Before, a second stream joined by events carried the beside kernels; measured on B200 the fork and join cost 1-3 us per frame
// on the GPU and four calls on the host.)
struct SrFollow {
    bool early = false, beside = false, late = false;
    int flags() const { return (beside ? 1 : 0) | (late ? 2 : 0); }
};
#ifdef __CUDACC__
__device__ __forceinline__ void sr_wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void sr_let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void sr_begin(int follow_flags)
{
    if (!(follow_flags & 2)) sr_let_successor_start();
    if (!(follow_flags & 1)) sr_wait_for_predecessor();
    if (follow_flags & 2) sr_let_successor_start();
}
__device__ __forceinline__ void sr_drop_old_lines(int follow_flags)
{
    if (follow_flags & 1) __threadfence();
}
// (Not volatile: a beside kernel may load as early as it likes.)
__device__ __forceinline__ float4 sr_load_past_l1(const float4* p)
{
    float4 v;
    asm("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 sr_load_past_l1(const uint4* p)
{
    uint4 v;
    asm("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 sr_load_past_l1(const uint2* p)
{
    uint2 v;
    asm("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float sr_load_past_l1(const float* p)
{
    float v;
    asm("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short sr_load_past_l1(const unsigned short* p)
{
    unsigned short v;
    asm("ld.global.cg.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void sr_end(int follow_flags)
{
    if ((follow_flags & 1) && blockIdx.x == 0) sr_wait_for_predecessor();
}

template <typename Params>
inline cudaError_t sr_launch(void (*kernel)(const Params), int blocks, int threads, size_t smem, cudaStream_t stream, bool early, const Params& p)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

struct SrFrame { long long t, run_t; };   // this launch computes frame t+1 from frame t
__device__ __forceinline__ SrFrame sr_frame(const SrFrameArgs& a)
{
    SrFrame f;
    f.t = (a.ctl ? a.ctl->t : a.v.t) + a.off;
    f.run_t = (a.ctl ? a.ctl->run_t : a.v.run_t) + a.off;
    return f;
}
__device__ __forceinline__ const char* sr_frame_input(const SrFrameArgs& a, const SrFrame& f, int slot)
{
    const char* base = static_cast<const char*>(a.ctl ? a.ctl->in_base[slot] : a.v.in_base[slot]);
    return base + f.run_t * (a.ctl ? a.ctl->in_stride_bytes[slot] : a.v.in_stride_bytes[slot]);
}
// The caller's output buffer for this frame, or null.
__device__ __forceinline__ float* sr_frame_output(const SrFrameArgs& a, const SrFrame& f)
{
    float* base = a.ctl ? a.ctl->out_base : a.v.out_base;
    return base ? base + f.run_t * (a.ctl ? a.ctl->out_stride : a.v.out_stride) : nullptr;
}
#endif

// ------------------------------------------------------------------ host-side graph
struct SrRegion { size_t offset = 0, bytes = 0; };

struct SrHostNode {
    sr_node_desc d;
    bool is_input = false;
    int level = 0;
    int input_slot = -1;
    std::vector<int> in_edges;
    bool dense_target = false;     // all incoming edges are dense / mean-dense
    bool use_tc = false;
    bool w_finite = true;          // every weight of the incoming edges is finite (nodes of the CUDA-core kernels)
    SrRegion state[2], bias;
    bool bias_set = false;
};

struct SrHostEdge {
    sr_edge_desc d;
    int R = 1;
    // the convolution actually executed (pooled edges are rewritten)
    int k_eff = 0, stride_eff = 0, pad_eff = 0, K = 0;
    SrRegion w_direct;
    bool w_set = false, w_finite = true;
};

// A few-channel input edge staged as im2col rows (see sr_input.cu).
struct SrStem {
    void* dst[2];                  // by frame parity
    int slot, R;                   // input node (index among the inputs); the edge's R
    int Hs, Ws, Cs, Ho, Wo, k, stride, pad, Kp, K;
};

struct sr_graph {
    std::vector<SrHostNode> nodes;
    std::vector<SrHostEdge> edges;
    int batch = 0, dtype = 0, elem = 4;
    sr_info info{};
    std::vector<int> input_nodes;
    std::vector<std::vector<int>> groups;          // groups[l-1] = nodes of level l
    // options
    int opt_engine = 0, opt_graph_frames = 0, opt_b_units = 0, opt_tile_w = 0, opt_overlap = 1, opt_time_tc = 0;
    int opt_tc_fuse = 1;                           // nodes of at most 64 channels that share a source run as one 128-row plan
    int opt_tc_lists = 0;                          // tensor-core work items: 1 = a list per CTA made on the host, 0 = the same plus a shared list of the smallest items
    int opt_wait_ms = 1000;                        // limit of every device-side wait; 0 = expire at once (test hook)
    int opt_resident = 1, opt_rs_cluster = 0, opt_rs_warps = 0, opt_rs_split = 0;   // 16-channel work units: 0 never, 1 always, 2 by cost
    // workspace
    size_t ws_bytes = 0;
    bool planned = false;                          // the workspace layout stands for the current options
    int compact = 0;                               // 0: launches planned for speed; 1, 2: for small tables, for small weights too (see plan)
    char* ws = nullptr;
    SrRegion r_nodes, r_edges, r_ctl, r_items;
    SrRegion r_clear;                              // what a reset zeroes: the flags, then the non-input nodes' parity-0 states
    SrRegion r_flags;                              // int 0: device-side error code (0 = none); ints 16, 17: the shared work list's counters
    int sm_count = 148;                            // of the device that is current when the graph is planned
    std::vector<SrStem> stems;                     // filled when a workspace is bound
    std::vector<const SrStem*> stems_of[4];        // those that a mask of R names (see sr_stems): nothing is allocated on a launch
    unsigned input_read = 0;                       // bit i: some edge reads input node i's state itself (not a staged copy)
    std::vector<int> group_item_count;             // per group
    std::vector<SrDirectItem> items;
    std::vector<int> group_item_offset;
    std::vector<char> group_sliced;                // per group: some item's reduction is cut into slices
    std::vector<std::vector<int>> group_head_nodes;       // per group: nodes of the head kernels
    std::vector<std::vector<SrHeadNode>> group_heads;     // and what they need to know about them (filled when a workspace is bound)
    std::vector<std::vector<SrWideNode>> group_wide;
    std::vector<std::vector<SrHeadEdge>> group_wide_edges;
    // dynamic state
    SrFrameArgs frame{};                           // of the launches being queued
    int64_t t = 0;
    int64_t launches = 0;
    void* tc = nullptr;                            // tensor-core engine state (opaque here)
    void* rs = nullptr;                            // resident engine state (opaque here)
    void* dn = nullptr;                            // dense resident engine state (opaque here)
    std::vector<unsigned char> dn_headers;         // its per-rank table images, uploaded when a workspace is bound
    void* graphs = nullptr;                        // CUDA-graph cache (opaque here)
    bool input_feeds_same_frame = false;           // some edge that leaves an input node has R = 0
    // deep-window mode: a second graph of the same network whose batch holds the W frames of a window side by side
    sr_graph* window = nullptr;
    bool is_window = false;                        // of another graph: never in the built-in workspace
    int window_frames = 0;
    std::vector<char> in_window;                   // per node: its current state is the last frame of the window's states
    std::vector<std::vector<float>> kept_weights;  // the parameters as the caller set them (host copies), for that graph
    std::vector<std::vector<float>> kept_bias;
    int static_device = -1;                        // >= 0: bound to the built-in workspace of that device
    bool stage_dirty = false;                      // the resident kernel ran: staged copies of the input state are stale
};

// sr_compile.cpp
sr_status sr_compile(sr_graph* g, const sr_node_desc* nodes, int n_nodes, const sr_edge_desc* edges, int n_edges,
                     const uint8_t* R);

void sr_window_tableau(const sr_graph* g, int W, int32_t* T /* [W + 1][n_nodes] */);

inline size_t sr_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
