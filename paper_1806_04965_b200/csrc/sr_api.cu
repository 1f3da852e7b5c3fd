// C ABI of the streaming-rollout library: graph objects, workspace layout, parameter upload and the
// per-frame launch sequence (frame input, one launch group per tableau level, buffer flip).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "sr_internal.h"
#include "sr_kernels.h"
#include "sr_dense.h"
#include "sr_resident.h"
#include "sr_tc.h"

// Built-in workspace for callers that may not allocate device memory.  In host code the array's name
// is only a handle: its device address is looked up once per device and that pointer is what the
// kernels get (through the ordinary bind path).  The work lists of the CUDA-core kernels have room beyond the size that callers know: 16
// bytes per 512 values or so (see sr_direct_conv_items; more where images are tiny).
constexpr size_t kStaticBytes = SR_STATIC_WORKSPACE_BYTES + SR_STATIC_WORKSPACE_BYTES / 256;
static __device__ __align__(256) unsigned char sr_static_workspace[kStaticBytes];

namespace {

// One owner per device: the graph that bound the array last.  Binding takes the array away from the previous owner,
// which becomes unbound (its calls then fail with SR_ERR_STATE on the host instead of running kernels on tables the
// new owner has overwritten).
struct StaticSlot {
    void* address = nullptr;
    sr_graph* owner = nullptr;
};
std::mutex static_mutex;
StaticSlot static_slot[64];

void unbind(sr_graph* g)
{
    g->ws = nullptr;
    g->static_device = -1;
    for (SrHostEdge& e : g->edges) e.w_set = false;
    for (SrHostNode& n : g->nodes) n.bias_set = false;
}

void sr_release_static_workspace(sr_graph* g)
{
    std::lock_guard<std::mutex> lock(static_mutex);
    if (g->static_device >= 0 && g->static_device < 64 && static_slot[g->static_device].owner == g)
        static_slot[g->static_device].owner = nullptr;
    g->static_device = -1;
}

struct GraphCache {
    cudaStream_t capture_stream = nullptr;
    cudaGraphExec_t exec = nullptr;
    int frames = 0;
    int kernels = 0;
};

// Launches recorded in a CUDA graph are recorded anew by the next run.
void forget_recorded(sr_graph* g)
{
    GraphCache* c = static_cast<GraphCache*>(g->graphs);
    if (c && c->exec) cudaGraphExecDestroy(c->exec);
    if (c) c->exec = nullptr;
}

float round_bf16_host(float f)
{
    uint32_t u;
    std::memcpy(&u, &f, 4);
    if ((u & 0x7F800000u) == 0x7F800000u) return f;
    u += 0x7FFFu + ((u >> 16) & 1u);
    u &= 0xFFFF0000u;
    std::memcpy(&f, &u, 4);
    return f;
}

size_t node_elems(const sr_graph* g, int v)
{
    const sr_node_desc& d = g->nodes[v].d;
    return (size_t)g->batch * d.h * d.w * d.c;
}

SrRegion take(size_t& off, size_t bytes)
{
    SrRegion r;
    r.offset = off;
    r.bytes = bytes;
    off = sr_align_up(off + bytes, 256);
    return r;
}

// Whether the built-in workspace takes a graph of this size.
bool fits_built_in(const sr_graph* g, size_t need) { return need - g->r_items.bytes <= (size_t)SR_STATIC_WORKSPACE_BYTES && need <= kStaticBytes; }

// Decide the engine of every node, lay out the workspace and build the block work lists.  Sets *least: bytes that the graph needs
// however it is planned.
sr_status lay_out(sr_graph* g, size_t* least)
{
    const int n_nodes = (int)g->nodes.size(), n_edges = (int)g->edges.size();
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0) g->sm_count = sms;
    for (int v = 0; v < n_nodes; ++v) {
        SrHostNode& n = g->nodes[v];
        n.dense_target = false;
        if (n.is_input) continue;
        int n_conv = 0, n_dense = 0;
        for (int e : n.in_edges) (g->edges[e].d.kind == SR_EDGE_CONV ? n_conv : n_dense)++;
        if (n_conv && n_dense) return SR_ERR_UNSUPPORTED;        // a node sums either convolutions or dense maps
        n.dense_target = n_dense > 0;
        n.use_tc = false;
    }
    if ((int)g->input_nodes.size() > SR_MAX_INPUTS) return SR_ERR_UNSUPPORTED;
    if (g->opt_engine == 0 && g->dtype == SR_DTYPE_BF16) sr_tc_select_nodes(g);
    size_t off = 0;
    // what a reset zeroes comes first, in one piece
    g->r_clear.offset = off;
    g->r_flags = take(off, 256);
    for (int v = 0; v < n_nodes; ++v)
        if (!g->nodes[v].is_input) g->nodes[v].state[0] = take(off, node_elems(g, v) * g->elem);
    g->r_clear.bytes = off - g->r_clear.offset;
    for (int v = 0; v < n_nodes; ++v) {
        SrHostNode& n = g->nodes[v];
        if (n.is_input) n.state[0] = take(off, node_elems(g, v) * g->elem);
        n.state[1] = take(off, node_elems(g, v) * g->elem);
        n.bias = take(off, (size_t)n.d.c * sizeof(float));
    }
    g->input_read = 0;
    for (int e = 0; e < n_edges; ++e)
        if (g->nodes[g->edges[e].d.src].is_input && !sr_tc_stages(g, e)) g->input_read |= 1u << g->nodes[g->edges[e].d.src].input_slot;
    for (int e = 0; e < n_edges; ++e) {
        SrHostEdge& he = g->edges[e];
        const SrHostNode& t = g->nodes[he.d.tgt];
        he.w_direct = SrRegion();
        if (!t.use_tc) he.w_direct = take(off, (size_t)he.K * t.d.c * sizeof(float));
    }
    *least = off;
    for (const SrHostEdge& he : g->edges)
        if (g->nodes[he.d.tgt].use_tc) *least += (size_t)he.K * g->nodes[he.d.tgt].d.c * g->elem;
    g->r_nodes = take(off, sizeof(SrDevNode) * n_nodes);
    g->r_edges = take(off, sizeof(SrDevEdge) * n_edges);
    g->r_ctl = take(off, sizeof(SrFrameCtl));
    // work lists of the direct kernels, one contiguous range per group
    g->items.clear();
    g->group_item_offset.clear();
    g->group_item_count.clear();
    g->group_sliced.clear();
    g->group_head_nodes.assign(g->groups.size(), {});
    const int dco = sr_direct_dense_outputs_per_block(),
              dsb = sr_direct_dense_samples_per_block();
    for (size_t gi = 0; gi < g->groups.size(); ++gi) {
        g->group_item_offset.push_back((int)g->items.size());
        for (int v : g->groups[gi]) {
            const SrHostNode& n = g->nodes[v];
            if (n.use_tc) continue;
            if (n.dense_target) {
                if (sr_head_class(g, v) != 0) {
                    g->group_head_nodes[gi].push_back(v);
                } else {
                    for (int b0 = 0; b0 < g->batch; b0 += dsb)
                        for (int c0 = 0; c0 < n.d.c; c0 += dco) g->items.push_back(SrDirectItem{v, b0, c0, 0});
                }
            } else {
                sr_direct_conv_items(g, v, g->items);
            }
        }
        // the items with the longest reductions first: a launch ends when its last block ends
        auto work = [&](const SrDirectItem& it) {
            long long k = 0;
            for (int e : g->nodes[it.node].in_edges) k += g->edges[e].K;
            return k * (it.b0 < 0 ? 4 : 1);
        };
        std::stable_sort(g->items.begin() + g->group_item_offset.back(), g->items.end(),
                         [&](const SrDirectItem& a, const SrDirectItem& b) { return work(a) > work(b); });
        g->group_item_count.push_back((int)g->items.size() - g->group_item_offset.back());
        g->group_sliced.push_back(0);
        for (size_t i = g->group_item_offset.back(); i < g->items.size(); ++i)
            if (!g->nodes[g->items[i].node].dense_target && sr_direct_sliced(g->items[i])) g->group_sliced.back() = 1;
    }
    g->r_items = take(off, sizeof(SrDirectItem) * std::max<size_t>(1, g->items.size()));
    sr_status st = sr_tc_plan(g, off);
    if (st != SR_OK) return st;
    st = sr_rs_plan(g, off);
    if (st != SR_OK) return st;
    st = sr_dn_plan(g, off);
    if (st != SR_OK) return st;
    g->ws_bytes = off;
    int n_tc = 0, n_direct = 0;
    for (const SrHostNode& n : g->nodes)
        if (!n.is_input) (n.use_tc ? n_tc : n_direct)++;
    g->info.n_tensor_core_nodes = n_tc;
    g->info.n_direct_nodes = n_direct;
    int rs_warps = 0;
    sr_rs_describe(g, &g->info.resident_cluster, &rs_warps, &g->info.resident_smem_bytes, &g->info.resident_heads_on_chip);
    if (sr_dn_available(g)) {
        sr_dn_describe(g, &g->info.resident_cluster, &g->info.resident_smem_bytes);
        g->info.resident_heads_on_chip = 1;
    }
    return SR_OK;
}

// Launches planned for speed may have longer lists (items cut into slices or parts, narrow tiles) and weight matrices with more zero
// rows (joined nodes) than a graph needs.  One that the built-in workspace takes only without them is planned without: lists
// and tables first, then joins.
sr_status plan(sr_graph* g)
{
    if (g->batch <= 0) return SR_ERR_STATE;
    if (g->planned) return SR_OK;                                // asking for the size and binding share one plan
    size_t least = 0;
    g->compact = 0;
    sr_status st = lay_out(g, &least);
    if (st == SR_OK && !g->is_window && !fits_built_in(g, g->ws_bytes) && least <= (size_t)SR_STATIC_WORKSPACE_BYTES) {
        for (g->compact = 1; g->compact <= 2; ++g->compact)
            if (lay_out(g, &least) == SR_OK && fits_built_in(g, g->ws_bytes)) break;
        if (g->compact > 2) {
            g->compact = 0;
            st = lay_out(g, &least);
        }
    }
    g->planned = st == SR_OK;
    return st;
}

bool cuda_ok(cudaError_t e) { return e == cudaSuccess; }


sr_status ready(const sr_graph* g)
{
    if (!g) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    for (const SrHostEdge& e : g->edges)
        if (!e.w_set) return SR_ERR_STATE;
    return SR_OK;
}

// Queue the kernels of `frames` consecutive frame updates, the first of them the one `fr` describes; returns the number of
// launches.  copies, stems_R: what sr_launch_input does for every frame.
int enqueue_frames(sr_graph* g, const SrFrameArgs& fr, int frames, cudaStream_t s, unsigned copies = ~0u, unsigned stems_R = 3u)
{
    int launches = 0;
    // events between two launches of a stream (the timing option) need plain launches around them
    const bool chain = !g->opt_time_tc, overlap = g->opt_overlap != 0;
    // The first launch may start early as well: what comes before it in the stream (an earlier call's kernel, the caller's own
    // work) either lets it or, not knowing, holds it until it has completed.  Not while a capture records the stream.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    bool first = cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    auto follow = [&](bool beside, bool late) {
        SrFollow how;
        how.early = chain && !first;
        how.beside = beside && chain;
        how.late = late && chain;
        first = false;
        return how;
    };
    g->frame = fr;
    const int last = (int)g->groups.size() - 1;
    // The input of a further frame may go beside the last group of the frame before it: it takes the buffers of the frame before
    // that, which only edges that bridge a frame (R = 1) still read.
    bool ahead = g->input_feeds_same_frame && overlap && chain;
    for (const SrHostEdge& e : g->edges)
        if (g->nodes[e.d.src].is_input && e.R == 1 && g->nodes[e.d.tgt].level == last + 1) ahead = false;
    bool there = false;                                          // the input of this frame has been queued
    for (int f = 0; f < frames; ++f, ++g->frame.off) {
        // The frame input: ahead of the first group if the update reads it (with its heads, where they can read the caller's
        // frame themselves; for all frames of a call but the first, beside the last group of the frame before: sequential rollouts
        // of the six-node and ten-node networks at one sample 38.5 -> 35.1 and 67.0 -> 63.2 us per frame), else beside the first group.
        const bool feeds = g->input_feeds_same_frame;
        for (int gi = 0; gi < (int)g->groups.size(); ++gi) {
            // up to four independent launches: one of them leads, the others run beside it
            const bool has_heads = !g->group_head_nodes[gi].empty(), has_items = g->group_item_count[gi] > 0, has_tc = sr_tc_group_has_work(g, gi);
            const bool heads_lead = !has_tc && !has_items;
            const bool merged = gi == 0 && has_heads && (heads_lead || !feeds) && sr_heads_take_input(g, gi, g->frame, copies, stems_R);
            if (merged) ahead = false;
            if (gi == 0 && feeds && !merged && !there) launches += sr_launch_input(g, g->frame, copies, stems_R, follow(false, false), nullptr, s);
            const bool input_beside = gi == 0 && !feeds && !merged;
            const bool next_input = ahead && gi == last && f + 1 < frames;
            const bool late = overlap && (input_beside || next_input || (has_tc + has_items + has_heads > 1));
            if (has_tc) launches += sr_tc_launch_group(g, gi, follow(false, late), s);
            if (has_items) launches += sr_launch_direct_group(g, gi, follow(overlap && has_tc, late && !has_tc), s);
            if (input_beside && !heads_lead) launches += sr_launch_input(g, g->frame, copies, stems_R, follow(overlap, false), nullptr, s);
            if (has_heads) launches += sr_launch_heads(g, gi, merged, copies, stems_R, follow(overlap && !heads_lead, late && heads_lead), s);
            if (input_beside && heads_lead) launches += sr_launch_input(g, g->frame, copies, stems_R, follow(overlap, false), nullptr, s);
            there = next_input;
            if (next_input) {
                ++g->frame.off;
                launches += sr_launch_input(g, g->frame, copies, stems_R, follow(true, false), nullptr, s);
                --g->frame.off;
            }
        }
    }
    return launches;
}

SrFrameCtl make_ctl(const sr_graph* g, const void* const* in, bool sequence, float* out)
{
    SrFrameCtl c{};
    c.t = g->t;
    c.run_t = 0;
    for (size_t i = 0; i < g->input_nodes.size(); ++i) {
        c.in_base[i] = in[i];
        c.in_stride_bytes[i] = sequence ? (int64_t)(node_elems(g, g->input_nodes[i]) * g->elem) : 0;
    }
    c.out_base = out;
    c.out_stride = (int64_t)node_elems(g, g->info.output_node);          // [B][H][W][C] floats per frame
    return c;
}

SrFrameArgs by_value(const SrFrameCtl& c) { return SrFrameArgs{nullptr, 0, c}; }

// The staged copies of the input nodes' current state that the next update reads (edges with R = 1), from the state itself.
void stage_current(sr_graph* g, cudaStream_t s)
{
    SrFrameCtl c{};
    c.t = g->t - 1;                                              // "the input of frame t"
    for (size_t i = 0; i < g->input_nodes.size(); ++i) c.in_base[i] = g->ws + g->nodes[g->input_nodes[i]].state[g->t & 1].offset;
    g->launches += sr_launch_input(g, by_value(c), 0u, 2u, SrFollow(), nullptr, s);
}

// After a resident run they are brought up to date when the launch path is used next.
void refresh_staging(sr_graph* g, cudaStream_t s)
{
    if (g->stage_dirty) stage_current(g, s);
    g->stage_dirty = false;
}

// The states of the last window are the current ones of this graph; an update of all nodes supersedes them.  (It does not read
// them: windows exist only for patterns in which every edge that bridges a frame leaves an input node.)
void leave_window(sr_graph* g) { g->in_window.assign(g->in_window.size(), 0); }

// The dense resident kernel fetches input frames in words of four values (the states lie on larger boundaries).
bool dense_resident_takes(const sr_graph* g, const void* const* in_dev)
{
    if (!sr_dn_available(g)) return false;
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        if (reinterpret_cast<uintptr_t>(in_dev[i]) & 15) return false;
    return true;
}

}  // namespace

// No exception leaves a C entry: what can throw here is the host's memory, for a size that it does not hold.
#define SR_NOTHROW catch (...) { return SR_ERR_INVALID_ARG; }

extern "C" {

sr_status sr_graph_create(const sr_node_desc* nodes, int n_nodes, const sr_edge_desc* edges, int n_edges,
                          const uint8_t* R, int batch, int dtype, sr_graph** out)
{
    if (!out || batch < 0 || (dtype != SR_DTYPE_F32 && dtype != SR_DTYPE_BF16)) return SR_ERR_INVALID_ARG;
    sr_graph* g = new (std::nothrow) sr_graph();
    if (!g) return SR_ERR_INVALID_ARG;
    sr_status st = SR_ERR_INVALID_ARG;
    try {
        st = sr_compile(g, nodes, n_nodes, edges, n_edges, R);
    } catch (...) {
    }
    if (st != SR_OK) {
        delete g;
        return st;
    }
    g->input_feeds_same_frame = false;
    for (const SrHostEdge& e : g->edges)
        if (g->nodes[e.d.src].is_input && e.R == 0) g->input_feeds_same_frame = true;
    g->batch = batch;
    g->dtype = dtype;
    g->elem = dtype == SR_DTYPE_BF16 ? 2 : 4;
    *out = g;
    return SR_OK;
}

void sr_graph_destroy(sr_graph* g)
{
    if (!g) return;
    if (g->window) sr_graph_destroy(g->window);
    g->window = nullptr;
    sr_release_static_workspace(g);
    if (g->graphs) {
        GraphCache* c = static_cast<GraphCache*>(g->graphs);
        if (c->exec) cudaGraphExecDestroy(c->exec);
        if (c->capture_stream) cudaStreamDestroy(c->capture_stream);
        delete c;
    }
    sr_tc_destroy(g);
    sr_rs_destroy(g);
    sr_dn_destroy(g);
    delete g;
}

sr_status sr_graph_info(const sr_graph* g, sr_info* out)
{
    if (!g || !out) return SR_ERR_INVALID_ARG;
    *out = g->info;
    return SR_OK;
}

sr_status sr_graph_levels(const sr_graph* g, int32_t* level)
{
    if (!g || !level) return SR_ERR_INVALID_ARG;
    for (size_t v = 0; v < g->nodes.size(); ++v) level[v] = g->nodes[v].level;
    return SR_OK;
}

sr_status sr_graph_set_option(sr_graph* g, int key, int value)
{
    if (!g) return SR_ERR_INVALID_ARG;
    if (!g->ws) g->planned = false;
    if (key == 0) {
        if (g->ws) return SR_ERR_STATE;
        if (value != 0 && value != 1) return SR_ERR_INVALID_ARG;
        g->opt_engine = value;
        return SR_OK;
    }
    if (key == 1) {
        if (value < 0 || value > 1024) return SR_ERR_INVALID_ARG;
        g->opt_graph_frames = value;
        return SR_OK;
    }
    if (key == 5) {
        if (value != 0 && value != 1) return SR_ERR_INVALID_ARG;
        g->opt_time_tc = value;
        return SR_OK;
    }
    if (key == 4) {
        if (value != 0 && value != 1) return SR_ERR_INVALID_ARG;
        g->opt_overlap = value;
        return SR_OK;
    }
    if (key == 3) {
        if (g->ws) return SR_ERR_STATE;
        if (value != 0 && value != 8 && value != 16 && value != 32) return SR_ERR_INVALID_ARG;
        g->opt_tile_w = value;
        return SR_OK;
    }
    if (key == 2) {
        if (g->ws) return SR_ERR_STATE;
        if (value < 0 || value > 8 || value == 1) return SR_ERR_INVALID_ARG;
        g->opt_b_units = value;
        return SR_OK;
    }
    if (key == 6) {
        if (g->ws) return SR_ERR_STATE;
        if (value != 0 && value != 1) return SR_ERR_INVALID_ARG;
        g->opt_resident = value;
        return SR_OK;
    }
    if (key == 7) {
        if (g->ws) return SR_ERR_STATE;
        if (value != 0 && value != 1 && value != 2 && value != 4) return SR_ERR_INVALID_ARG;
        g->opt_rs_cluster = value;
        return SR_OK;
    }
    if (key == 9) {
        if (g->ws) return SR_ERR_STATE;
        if (value < 0 || value > 2) return SR_ERR_INVALID_ARG;
        g->opt_rs_split = value;
        return SR_OK;
    }
    if (key == 8) {
        if (g->ws) return SR_ERR_STATE;
        if (value != 0 && (value < 4 || value > 32)) return SR_ERR_INVALID_ARG;
        g->opt_rs_warps = value;
        return SR_OK;
    }
    if (key == 11 || key == 12) {                        // accepted, without effect
        if (g->ws) return SR_ERR_STATE;
        return value < 0 || value > 2 ? SR_ERR_INVALID_ARG : SR_OK;
    }
    if (key == 14) {
        if (g->ws) return SR_ERR_STATE;
        if (value < 0 || value > 1) return SR_ERR_INVALID_ARG;
        g->opt_tc_fuse = value;
        return SR_OK;
    }
    if (key == 13) {
        if (g->ws) return SR_ERR_STATE;
        if (value < 0 || value > 1) return SR_ERR_INVALID_ARG;
        g->opt_tc_lists = value;
        return SR_OK;
    }
    if (key == 10) {
        if (value < 0 || value > 60000) return SR_ERR_INVALID_ARG;
        g->opt_wait_ms = value;
        forget_recorded(g);                              // recorded launches carry the old limit
        if (g->window) g->window->opt_wait_ms = value;
        return SR_OK;
    }
    return SR_ERR_INVALID_ARG;
}

sr_status sr_graph_workspace_bytes(const sr_graph* g, size_t* bytes)
try {
    if (!g || !bytes) return SR_ERR_INVALID_ARG;
    if (g->ws) {
        *bytes = g->ws_bytes;
        return SR_OK;
    }
    const sr_status st = plan(const_cast<sr_graph*>(g));
    if (st != SR_OK) return st;
    *bytes = g->ws_bytes;
    return SR_OK;
} SR_NOTHROW

sr_status sr_graph_bind_workspace(sr_graph* g, void* workspace_dev, size_t bytes)
try {
    if (!g || !workspace_dev) return SR_ERR_INVALID_ARG;
    if (g->ws) return SR_ERR_STATE;
    if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return SR_ERR_INVALID_ARG;
    forget_recorded(g);                                  // launches recorded for an earlier binding point at its tables
    sr_status st = plan(g);
    if (st != SR_OK) return st;
    if (bytes < g->ws_bytes) return SR_ERR_INVALID_ARG;
    char* ws = static_cast<char*>(workspace_dev);
    const int n_nodes = (int)g->nodes.size(), n_edges = (int)g->edges.size();
    std::vector<SrDevNode> dn(n_nodes);
    std::vector<SrDevEdge> de(n_edges);
    int pos = 0;
    for (int v = 0; v < n_nodes; ++v) {
        const SrHostNode& n = g->nodes[v];
        SrDevNode& d = dn[v];
        d.state[0] = ws + n.state[0].offset;
        d.state[1] = ws + n.state[1].offset;
        d.bias = reinterpret_cast<const float*>(ws + n.bias.offset);
        d.H = n.d.h; d.W = n.d.w; d.C = n.d.c; d.act = n.d.act;
        d.first_edge = pos;
        d.n_edges = (int)n.in_edges.size();
        d.is_output = v == g->info.output_node;
        d.untiled = sr_direct_untiled(g, v);
        for (int e : n.in_edges) {
            const SrHostEdge& he = g->edges[e];
            const SrHostNode& s = g->nodes[he.d.src];
            SrDevEdge& x = de[pos++];
            x.src[0] = ws + s.state[0].offset;
            x.src[1] = ws + s.state[1].offset;
            x.w = reinterpret_cast<const float*>(ws + he.w_direct.offset);
            x.Hs = s.d.h; x.Ws = s.d.w; x.Cs = s.d.c;
            x.kind = he.d.kind; x.k = he.k_eff; x.stride = he.stride_eff; x.pad = he.pad_eff;
            x.R = he.R; x.K = he.K; x.src_is_input = s.is_input;
        }
    }
    for (SrHostEdge& e : g->edges) e.w_finite = true;
    for (SrHostNode& n : g->nodes) n.w_finite = true;
    if (!cuda_ok(cudaMemset(ws, 0, g->ws_bytes))) return SR_ERR_CUDA;
    if (!cuda_ok(cudaMemcpy(ws + g->r_nodes.offset, dn.data(), sizeof(SrDevNode) * n_nodes, cudaMemcpyHostToDevice)))
        return SR_ERR_CUDA;
    if (!cuda_ok(cudaMemcpy(ws + g->r_edges.offset, de.data(), sizeof(SrDevEdge) * n_edges, cudaMemcpyHostToDevice)))
        return SR_ERR_CUDA;
    if (!g->items.empty() &&
        !cuda_ok(cudaMemcpy(ws + g->r_items.offset, g->items.data(), sizeof(SrDirectItem) * g->items.size(),
                            cudaMemcpyHostToDevice)))
        return SR_ERR_CUDA;
    g->group_heads.assign(g->groups.size(), {});
    g->group_wide.assign(g->groups.size(), {});
    g->group_wide_edges.assign(g->groups.size(), {});
    g->stems.clear();
    g->ws = ws;
    for (size_t gi = 0; gi < g->groups.size(); ++gi) sr_describe_heads(g, (int)gi);
    st = sr_tc_bind(g);
    for (unsigned mask = 0; mask < 4; ++mask) {
        g->stems_of[mask].clear();
        for (const SrStem& stem : g->stems)
            if ((mask >> stem.R) & 1u) g->stems_of[mask].push_back(&stem);
    }
    if (st == SR_OK && g->info.n_tensor_core_nodes > 0 && (!sr_input_share_sm() || !sr_direct_share_sm())) st = SR_ERR_CUDA;
    if (st == SR_OK) st = sr_rs_bind(g);
    if (st == SR_OK) st = sr_dn_bind(g);
    if (st != SR_OK) {
        g->ws = nullptr;
        return st;
    }
    g->t = 0;
    g->in_window.assign(g->nodes.size(), 0);
    return SR_OK;
} catch (...) {
    g->ws = nullptr;                                     // (a bound graph is refused before anything can throw)
    return SR_ERR_INVALID_ARG;
}

sr_status sr_graph_bind_static_workspace(sr_graph* g)
{
    if (!g) return SR_ERR_INVALID_ARG;
    if (g->ws || g->batch <= 0) return SR_ERR_STATE;
    size_t need = 0;
    sr_status st = sr_graph_workspace_bytes(g, &need);
    if (st != SR_OK) return st;
    if (!fits_built_in(g, need)) return SR_ERR_TOO_LARGE;
    int dev = -1;
    if (!cuda_ok(cudaGetDevice(&dev)) || dev < 0 || dev >= 64) return SR_ERR_CUDA;
    std::lock_guard<std::mutex> lock(static_mutex);
    StaticSlot& slot = static_slot[dev];
    if (!slot.address) {
        void* p = nullptr;
        if (!cuda_ok(cudaGetSymbolAddress(&p, sr_static_workspace)) || !p) return SR_ERR_CUDA;
        slot.address = p;
    }
    if (slot.owner && slot.owner != g) unbind(slot.owner);
    slot.owner = nullptr;
    st = sr_graph_bind_workspace(g, slot.address, kStaticBytes);
    if (st != SR_OK) return st;
    slot.owner = g;
    g->static_device = dev;
    return SR_OK;
}

sr_status sr_graph_set_edge_weights(sr_graph* g, int edge, const float* w, int is_device)
try {
    if (!g || !w || edge < 0 || edge >= (int)g->edges.size()) return SR_ERR_INVALID_ARG;
    if (!g->ws) return SR_ERR_STATE;
    SrHostEdge& he = g->edges[edge];
    const SrHostNode& s = g->nodes[he.d.src];
    const SrHostNode& t = g->nodes[he.d.tgt];
    const int Cout = t.d.c, Cs = s.d.c;
    const size_t n_user = (he.d.kind == SR_EDGE_CONV) ? (size_t)Cout * he.d.k * he.d.k * Cs : (size_t)Cout * he.K;
    std::vector<float> u(n_user);
    if (is_device) {
        if (!cuda_ok(cudaMemcpy(u.data(), w, n_user * sizeof(float), cudaMemcpyDeviceToHost))) return SR_ERR_CUDA;
    } else {
        std::memcpy(u.data(), w, n_user * sizeof(float));
    }
    if (g->kept_weights.size() != g->edges.size()) g->kept_weights.assign(g->edges.size(), std::vector<float>());
    g->kept_weights[edge] = u;                                   // as set by the caller: a window graph gets the same
    if (g->dtype == SR_DTYPE_BF16)
        for (float& x : u) x = round_bf16_host(x);
    // the convolution actually executed: [C_out][k'][k'][Cs]; a pooled edge gets the box-filtered kernel
    std::vector<float> eff;
    const int k = he.d.k, ke = he.k_eff;
    if (he.d.kind == SR_EDGE_CONV && he.d.pool == 2) {
        eff.assign((size_t)Cout * ke * ke * Cs, 0.f);
        const int sh = he.d.stride;
        for (int co = 0; co < Cout; ++co)
            for (int dy = 0; dy < 2; ++dy)
                for (int dx = 0; dx < 2; ++dx)
                    for (int ky = 0; ky < k; ++ky)
                        for (int kx = 0; kx < k; ++kx)
                            for (int ci = 0; ci < Cs; ++ci)
                                eff[(((size_t)co * ke + ky + dy * sh) * ke + kx + dx * sh) * Cs + ci] +=
                                    0.25f * u[(((size_t)co * k + ky) * k + kx) * Cs + ci];
    } else {
        eff.swap(u);
    }
    if (!t.use_tc) {
        std::vector<float> d;
        const float* src = eff.data();
        if (he.d.kind == SR_EDGE_CONV) {                        // [C_out][K] -> [K][C_out]
            d.resize((size_t)he.K * Cout);
            for (int co = 0; co < Cout; ++co)
                for (int kk = 0; kk < he.K; ++kk) d[(size_t)kk * Cout + co] = eff[(size_t)co * he.K + kk];
            src = d.data();
        }
        if (!cuda_ok(cudaMemcpy(g->ws + he.w_direct.offset, src, (size_t)he.K * Cout * sizeof(float),
                                cudaMemcpyHostToDevice)))
            return SR_ERR_CUDA;
        // a convolutional node with a weight that is not finite leaves conv_tile, and returns to it with its last one
        he.w_finite = std::all_of(src, src + (size_t)he.K * Cout, [](float v) { return std::isfinite(v); });
        const bool finite = std::all_of(t.in_edges.begin(), t.in_edges.end(), [&](int e) { return g->edges[e].w_finite; });
        if (finite != t.w_finite) {
            const int32_t untiled = sr_direct_untiled(g, he.d.tgt) ? 1 : finite ? 0 : g->dtype == SR_DTYPE_BF16 ? 2 : 4;
            if (!cuda_ok(cudaMemcpy(g->ws + g->r_nodes.offset + sizeof(SrDevNode) * he.d.tgt + offsetof(SrDevNode, untiled), &untiled, sizeof(untiled),
                                    cudaMemcpyHostToDevice)))
                return SR_ERR_CUDA;
            g->nodes[he.d.tgt].w_finite = finite;
            forget_recorded(g);
        }
    } else {
        const sr_status st = sr_tc_set_weights(g, edge, eff.data());
        if (st != SR_OK) return st;
    }
    {
        sr_status st = sr_rs_set_weights(g, edge, eff.data());
        if (st == SR_OK) st = sr_dn_set_weights(g, edge, eff.data());
        if (st != SR_OK) return st;
    }
    he.w_set = true;
    return SR_OK;
} SR_NOTHROW

sr_status sr_graph_set_node_bias(sr_graph* g, int node, const float* bias_host)
try {
    if (!g || !bias_host || node < 0 || node >= (int)g->nodes.size()) return SR_ERR_INVALID_ARG;
    if (!g->ws) return SR_ERR_STATE;
    SrHostNode& n = g->nodes[node];
    if (!cuda_ok(cudaMemcpy(g->ws + n.bias.offset, bias_host, (size_t)n.d.c * sizeof(float), cudaMemcpyHostToDevice)))
        return SR_ERR_CUDA;
    n.bias_set = true;
    if (g->kept_bias.size() != g->nodes.size()) g->kept_bias.assign(g->nodes.size(), std::vector<float>());
    g->kept_bias[node].assign(bias_host, bias_host + n.d.c);
    return SR_OK;
} SR_NOTHROW

sr_status sr_graph_reset(sr_graph* g, const void* const* in0_dev, void* stream)
{
    if (!g || !in0_dev) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        if (!in0_dev[i]) return SR_ERR_INVALID_ARG;
    // Zeroed with the input: the non-input states of frame 0 (those of the other parity are written before they are read), a
    // reported device-side error (an expired wait: the rollout starts over) and the shared work list's counters (every launch
    // leaves them at zero; this covers a launch cut short).
    if (g->window && g->window->ws && !cuda_ok(cudaMemsetAsync(g->window->ws + g->window->r_flags.offset, 0, g->window->r_flags.bytes, s)))
        return SR_ERR_CUDA;
    g->t = 0;
    leave_window(g);
    SrFrameCtl c{};
    c.t = -1;                                                    // "the input of frame 0"
    for (size_t i = 0; i < g->input_nodes.size(); ++i) c.in_base[i] = in0_dev[i];
    const bool resident = sr_rs_available(g) || sr_dn_available(g);      // a resident run does not read staged edges
    g->launches += sr_launch_input(g, by_value(c), ~0u, resident ? 0u : 2u, SrFollow(), &g->r_clear, s);
    g->stage_dirty = resident;
    return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
}

sr_status sr_rollout_step(sr_graph* g, const void* const* in_next_dev, float* out_dev, void* stream)
try {
    sr_status st = ready(g);
    if (st != SR_OK) return st;
    if (!in_next_dev) return SR_ERR_INVALID_ARG;
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        if (!in_next_dev[i]) return SR_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // One frame on the dense resident engine: one launch instead of one per level, whose weights are on their way to shared memory
    // while the step before it still runs.  Measured on the 784-128-128-10 network, steps called from Python, us per step,
    // sequential pattern: 1 / 8 / 56 / 120 sequences 12.5 / 14.4 / 14.5 / 17.2 launched, 8.0 / 8.5 / 10.3 / 12.2 resident;
    // streaming 8.4 / 10.3 / 10.3 / 10.9 and 8.1 / 8.1 / 8.8 / 10.4.  With more clusters than the device holds (256 sequences)
    // every wave loads the weights again: 25.9 and 33.2, streaming 19.3 and 28.2.
    if (sr_dn_one_wave(g) && dense_resident_takes(g, in_next_dev)) {
        st = sr_dn_launch(g, 1, make_ctl(g, in_next_dev, false, out_dev), s);
        if (st != SR_OK) return st;
        g->launches += 1;
        g->stage_dirty = true;
    } else {
        refresh_staging(g, s);
        g->launches += enqueue_frames(g, by_value(make_ctl(g, in_next_dev, false, out_dev)), 1, s);
    }
    g->t += 1;
    leave_window(g);
    return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
} SR_NOTHROW

sr_status sr_rollout_run(sr_graph* g, const void* const* in_seq_dev, int T, float* out_seq_dev, void* stream)
try {
    sr_status st = ready(g);
    if (st != SR_OK) return st;
    if (!in_seq_dev || T < 0) return SR_ERR_INVALID_ARG;
    if (T == 0) return SR_OK;                                    // an empty sequence: nothing to read, nothing changes
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        if (!in_seq_dev[i]) return SR_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    leave_window(g);
    if (sr_rs_available(g)) {
        bool aligned = true;                                     // the resident kernel fetches input rows in 4-byte words
        for (size_t i = 0; i < g->input_nodes.size(); ++i)
            if (reinterpret_cast<uintptr_t>(in_seq_dev[i]) & 3) aligned = false;
        if (aligned) {
            // one launch walks all T frames with the states in shared memory, then the frame counter
            // advances and whatever the launch path derives from the input state is refreshed
            st = sr_rs_launch(g, T, make_ctl(g, in_seq_dev, true, out_seq_dev), s);
            if (st != SR_OK) return st;
            g->launches += 1;
            g->t += T;
            g->stage_dirty = true;             // refreshed when the launch path is used next
            return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
        }
    }
    if (dense_resident_takes(g, in_seq_dev)) {
        st = sr_dn_launch(g, T, make_ctl(g, in_seq_dev, true, out_seq_dev), s);
        if (st != SR_OK) return st;
        g->launches += 1;
        g->t += T;
        g->stage_dirty = true;
        return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
    }
    refresh_staging(g, s);
    SrFrameArgs fr = by_value(make_ctl(g, in_seq_dev, true, out_seq_dev));
    int done = 0;
    const int gf = g->opt_graph_frames;
    if (gf > 0 && T >= gf) {
        GraphCache* c = static_cast<GraphCache*>(g->graphs);
        if (!c) {
            c = new GraphCache();
            g->graphs = c;
        }
        if (c->exec && c->frames != gf) {
            cudaGraphExecDestroy(c->exec);
            c->exec = nullptr;
        }
        if (!c->exec) {
            if (!c->capture_stream && !cuda_ok(cudaStreamCreateWithFlags(&c->capture_stream, cudaStreamNonBlocking)))
                return SR_ERR_CUDA;
            cudaGraph_t graph = nullptr;
            if (!cuda_ok(cudaStreamBeginCapture(c->capture_stream, cudaStreamCaptureModeThreadLocal))) return SR_ERR_CUDA;
            SrFrameArgs rec{};
            rec.ctl = reinterpret_cast<const SrFrameCtl*>(g->ws + g->r_ctl.offset);
            int k = enqueue_frames(g, rec, gf, c->capture_stream);
            sr_launch_advance(g, gf, c->capture_stream);
            ++k;
            // a capture that has begun is always ended, also when a launch inside it failed: a stream left in
            // capture mode would refuse every later use
            const bool queued = cuda_ok(cudaGetLastError());
            const bool ended = cuda_ok(cudaStreamEndCapture(c->capture_stream, &graph));
            if (!queued || !ended || !graph) {
                if (graph) cudaGraphDestroy(graph);
                cudaGetLastError();
                return SR_ERR_CUDA;
            }
            const cudaError_t ie = cudaGraphInstantiate(&c->exec, graph, 0);
            cudaGraphDestroy(graph);
            if (!cuda_ok(ie)) {
                c->exec = nullptr;
                return SR_ERR_CUDA;
            }
            c->frames = gf;
            c->kernels = k;
        }
        sr_launch_set_ctl(g, fr.v, s);
        g->launches += 1;
        while (T - done >= gf) {
            if (!cuda_ok(cudaGraphLaunch(c->exec, s))) return SR_ERR_CUDA;
            g->launches += c->kernels;
            done += gf;
        }
    }
    if (done < T) {
        fr.off = done;
        g->launches += enqueue_frames(g, fr, T - done, s);
    }
    g->t += T;
    return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
} SR_NOTHROW

// ------------------------------------------------------------------ deep windows (W > 1)
sr_status sr_graph_window_tableau(const sr_graph* g, int W, int32_t* T_host)
try {
    if (!g || !T_host || W < 1 || W > 4096) return SR_ERR_INVALID_ARG;
    sr_window_tableau(g, W, T_host);
    return SR_OK;
} SR_NOTHROW

static bool frames_independent(const sr_graph* g)
{
    for (const SrHostEdge& e : g->edges)
        if (e.R == 1 && !g->nodes[e.d.src].is_input) return false;
    return true;
}

sr_status sr_graph_window_workspace_bytes(sr_graph* g, int W, size_t* bytes)
try {
    if (!g || !bytes || W < 1 || W > 4096) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0) return SR_ERR_STATE;
    if (!frames_independent(g)) return SR_ERR_UNSUPPORTED;
    if (g->window && g->window_frames != W) {
        if (g->window->ws) return SR_ERR_STATE;                  // a bound window keeps its size
        sr_graph_destroy(g->window);
        g->window = nullptr;
    }
    if (!g->window) {
        std::vector<sr_node_desc> nd;
        std::vector<sr_edge_desc> ed;
        std::vector<uint8_t> R;
        for (const SrHostNode& n : g->nodes) nd.push_back(n.d);
        for (const SrHostEdge& e : g->edges) {
            ed.push_back(e.d);
            R.push_back((uint8_t)e.R);
        }
        sr_graph* w = nullptr;
        const sr_status st = sr_graph_create(nd.data(), (int)nd.size(), ed.data(), (int)ed.size(), R.data(), g->batch * W, g->dtype, &w);
        if (st != SR_OK) return st;
        w->is_window = true;
        w->opt_engine = g->opt_engine;
        w->opt_b_units = g->opt_b_units;
        w->opt_tile_w = g->opt_tile_w;
        w->opt_overlap = g->opt_overlap;
        w->opt_tc_lists = g->opt_tc_lists;
        w->opt_tc_fuse = g->opt_tc_fuse;
        w->opt_wait_ms = g->opt_wait_ms;
        w->opt_resident = 0;                                     // a window is one update of a large batch: the launch path
        g->window = w;
        g->window_frames = W;
    }
    return sr_graph_workspace_bytes(g->window, bytes);
} SR_NOTHROW

sr_status sr_graph_bind_window(sr_graph* g, int W, void* workspace_dev, size_t bytes)
try {
    if (!g || !workspace_dev) return SR_ERR_INVALID_ARG;
    sr_status st = ready(g);
    if (st != SR_OK) return st;
    size_t need = 0;
    st = sr_graph_window_workspace_bytes(g, W, &need);
    if (st != SR_OK) return st;
    if (g->window->ws) return SR_ERR_STATE;
    if (g->kept_weights.size() != g->edges.size()) return SR_ERR_STATE;
    st = sr_graph_bind_workspace(g->window, workspace_dev, bytes);
    if (st != SR_OK) return st;
    for (size_t e = 0; e < g->edges.size(); ++e) {
        st = sr_graph_set_edge_weights(g->window, (int)e, g->kept_weights[e].data(), 0);
        if (st != SR_OK) return st;
    }
    for (size_t v = 0; v < g->nodes.size() && v < g->kept_bias.size(); ++v)
        if (!g->kept_bias[v].empty()) {
            st = sr_graph_set_node_bias(g->window, (int)v, g->kept_bias[v].data());
            if (st != SR_OK) return st;
        }
    return SR_OK;
} SR_NOTHROW

sr_status sr_rollout_window(sr_graph* g, const void* const* in_seq_dev, int W, float* out_seq_dev, void* stream)
try {
    sr_status st = ready(g);
    if (st != SR_OK) return st;
    sr_graph* w = g->window;
    if (!w || !w->ws || g->window_frames != W) return SR_ERR_STATE;
    if (!in_seq_dev) return SR_ERR_INVALID_ARG;
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        if (!in_seq_dev[i]) return SR_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // frames t .. t+W-1 of the input nodes side by side: what edges that bridge a frame read (Eq. 2: frame i - R(e))
    unsigned bridging = 0;
    for (const SrHostEdge& e : g->edges)
        if (e.R == 1) bridging |= 1u << g->nodes[e.d.src].input_slot;
    for (size_t i = 0; i < g->input_nodes.size(); ++i) {
        if (!((bridging >> i) & 1u)) continue;
        const int v = g->input_nodes[i];
        const size_t frame = node_elems(g, v) * g->elem;
        char* dst = w->ws + w->nodes[v].state[0].offset;
        if (!cuda_ok(cudaMemcpyAsync(dst, g->ws + g->nodes[v].state[g->t & 1].offset, frame, cudaMemcpyDeviceToDevice, s))) return SR_ERR_CUDA;
        if (W > 1 && !cuda_ok(cudaMemcpyAsync(dst + frame, in_seq_dev[i], frame * (size_t)(W - 1), cudaMemcpyDeviceToDevice, s)))
            return SR_ERR_CUDA;
    }
    w->t = 0;
    if (bridging) stage_current(w, s);
    // ONE update of the window graph computes all W frames: its batch is [W][B], which is how in_seq and out_seq lie in memory.
    // Of its input it needs what is read within the frame only.
    w->launches += enqueue_frames(w, by_value(make_ctl(w, in_seq_dev, false, out_seq_dev)), 1, s, w->input_read, 1u);
    // the last frame of the window becomes the current frame of this graph (Sec. 4: windows chain); the non-input states stay
    // where they are (see leave_window)
    const int64_t t_new = g->t + W;
    SrFrameCtl c{};
    c.t = t_new - 1;
    for (size_t i = 0; i < g->input_nodes.size(); ++i)
        c.in_base[i] = static_cast<const char*>(in_seq_dev[i]) + node_elems(g, g->input_nodes[i]) * g->elem * (size_t)(W - 1);
    w->launches += sr_launch_input(g, by_value(c), ~0u, 0u, SrFollow(), nullptr, s);
    for (size_t v = 0; v < g->nodes.size(); ++v) g->in_window[v] = !g->nodes[v].is_input;
    g->t = t_new;
    g->stage_dirty = true;
    g->launches += w->launches;
    w->launches = 0;
    return cuda_ok(cudaGetLastError()) ? SR_OK : SR_ERR_CUDA;
} SR_NOTHROW

sr_status sr_graph_get_state(const sr_graph* g, int node, void* dst_dev, void* stream)
{
    if (!g || !dst_dev || node < 0 || node >= (int)g->nodes.size()) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    const size_t bytes = node_elems(g, node) * g->elem;
    const char* src = g->ws + g->nodes[node].state[g->t & 1].offset;
    if (g->in_window[node]) src = g->window->ws + g->window->nodes[node].state[1].offset + bytes * (size_t)(g->window_frames - 1);
    return cuda_ok(cudaMemcpyAsync(dst_dev, src, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream))) ? SR_OK : SR_ERR_CUDA;
}

sr_status sr_graph_set_state(sr_graph* g, int node, const void* src_dev, void* stream)
{
    if (!g || !src_dev || node < 0 || node >= (int)g->nodes.size()) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    const SrHostNode& n = g->nodes[node];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!cuda_ok(cudaMemcpyAsync(g->ws + n.state[g->t & 1].offset, src_dev, node_elems(g, node) * g->elem,
                                 cudaMemcpyDeviceToDevice, s)))
        return SR_ERR_CUDA;
    g->in_window[node] = 0;
    if (n.is_input && !g->stage_dirty) stage_current(g, s);
    return SR_OK;
}

sr_status sr_graph_frame(const sr_graph* g, int64_t* t)
{
    if (!g || !t) return SR_ERR_INVALID_ARG;
    *t = g->t;
    return SR_OK;
}

sr_status sr_graph_launch_count(const sr_graph* g, int64_t* n)
{
    if (!g || !n) return SR_ERR_INVALID_ARG;
    *n = g->launches;
    return SR_OK;
}

sr_status sr_graph_launch_plan(const sr_graph* g, int group, sr_launch_plan* out)
{
    if (!g || !out || group < 0 || group >= (int)g->groups.size()) return SR_ERR_INVALID_ARG;
    if (!g->planned) return SR_ERR_STATE;
    sr_tc_describe(g, group, out);
    return SR_OK;
}

sr_status sr_graph_kernel_time(sr_graph* g, double* ms, int64_t* launches)
{
    if (!g || !ms || !launches) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    long long n = 0, n_rs = 0;
    double ms_rs = 0.0;
    sr_status st = sr_tc_timing(g, ms, &n);
    if (st == SR_OK) st = sr_rs_timing(g, &ms_rs, &n_rs);
    double ms_dn = 0.0;
    long long n_dn = 0;
    if (st == SR_OK) st = sr_dn_timing(g, &ms_dn, &n_dn);
    *ms += ms_rs + ms_dn;
    *launches = n + n_rs + n_dn;
    return st;
}

sr_status sr_graph_sync_status(sr_graph* g, void* stream)
{
    if (!g) return SR_ERR_INVALID_ARG;
    if (g->batch <= 0 || !g->ws) return SR_ERR_STATE;
    if (!cuda_ok(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)))) return SR_ERR_CUDA;
    for (const sr_graph* q : {static_cast<const sr_graph*>(g), static_cast<const sr_graph*>(g->window)}) {   // a window's launches report to its own word
        int error = 0;
        if (!q || !q->ws) continue;
        if (!cuda_ok(cudaMemcpy(&error, q->ws + q->r_flags.offset, sizeof(error), cudaMemcpyDeviceToHost))) return SR_ERR_CUDA;
        if (error != 0) return SR_ERR_TIMEOUT;
    }
    return SR_OK;
}

const char* sr_status_str(sr_status s)
{
    switch (s) {
        case SR_OK: return "ok";
        case SR_ERR_INVALID_ARG: return "invalid argument";
        case SR_ERR_NOT_A_NETWORK: return "not a network (no edges, or a node is not connected to an input)";
        case SR_ERR_INVALID_ROLLOUT: return "invalid rollout pattern (its rollout window has a cycle)";
        case SR_ERR_SHAPE_MISMATCH: return "an edge does not map its source shape to its target shape";
        case SR_ERR_UNSUPPORTED: return "unsupported configuration";
        case SR_ERR_CUDA: return "CUDA error";
        case SR_ERR_TIMEOUT: return "a device-side wait expired";
        case SR_ERR_STATE: return "call order (workspace not bound, weights not set, or graph is theory-only)";
        case SR_ERR_TOO_LARGE: return "the graph needs more workspace than the built-in workspace holds";
    }
    return "unknown status";
}

}  // extern "C"
