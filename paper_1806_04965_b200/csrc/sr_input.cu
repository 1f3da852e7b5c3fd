// Launches of the frame input (see sr_input.cuh) and of the frame control block.
#include <cuda_runtime.h>

#include "sr_input.cuh"
#include "sr_kernels.h"

namespace {

struct InputParams {
    SrFrameArgs fr;
    SrInputPart in;
    int32_t follow, clear_blocks;                  // blocks behind those of `in` that zero `clear`
    uint4* clear;
    size_t n_clear;                                // 16-byte words
};
static_assert(sizeof(InputParams) <= 4000, "kernel parameters");

// (Registers for six blocks per SM: three of them fit beside a CTA of the tensor-core kernel.)
template <bool CLEAR, bool BESIDE>
__global__ void __launch_bounds__(kInputThreads, CLEAR ? 1 : 6) sr_input_kernel(const __grid_constant__ InputParams P)
{
    __shared__ int2 tap[128];
    sr_begin(P.follow);
    if (!CLEAR || (int)blockIdx.x < P.in.n_blocks) {
        sr_input_block<BESIDE>(P.in, P.fr, sr_frame(P.fr), (int)blockIdx.x, tap);
    } else {
        const size_t nth = (size_t)P.clear_blocks * kInputThreads;
        for (size_t i = (size_t)((int)blockIdx.x - P.in.n_blocks) * kInputThreads + threadIdx.x; i < P.n_clear; i += nth) P.clear[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    sr_end(P.follow);
}

__global__ void sr_set_ctl_kernel(SrFrameCtl* ctl, SrFrameCtl v) { *ctl = v; }

__global__ void sr_advance_kernel(SrFrameCtl* ctl, int n)
{
    ctl->t += n;
    ctl->run_t += n;
}

}  // namespace

// Queues the input of the frame that `fr` describes.  copies: bit i = input node i's state takes it; stems_R: see sr_stems.
// `clear` (or null): a region, in whole 16-byte words, that the same launch zeroes (a reset: as a memset of its own it took
// 2 us of a small network's pass on the GPU, and a launch on the host).  Returns launches.
int sr_launch_input(const sr_graph* g, const SrFrameArgs& fr, unsigned copies, unsigned stems_R, SrFollow how, const SrRegion* clear, cudaStream_t s)
{
    int launches = 0;
    const std::vector<const SrStem*>& stems = sr_stems(g, stems_R);
    size_t next = 0;
    do {
        InputParams P{fr, sr_plan_input(g, launches == 0 ? copies : 0u, stems, next, how.beside), how.flags(), 0, nullptr, 0};
        if (clear && launches == 0) {
            P.clear = reinterpret_cast<uint4*>(g->ws + clear->offset);
            P.n_clear = clear->bytes / 16;
            P.clear_blocks = (int)std::min<size_t>((size_t)g->sm_count * 6, (P.n_clear + 4 * kInputThreads - 1) / (4 * kInputThreads));
        }
        if (P.in.n_blocks + P.clear_blocks == 0) break;
        sr_launch(P.clear_blocks ? sr_input_kernel<true, false> : how.beside ? sr_input_kernel<false, true> : sr_input_kernel<false, false>, P.in.n_blocks + P.clear_blocks, kInputThreads, 0, s, how.early, P);
        ++launches;
        how.early = true;
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
    auto ask = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess; };
    return ask(sr_input_kernel<false, false>) && ask(sr_input_kernel<false, true>);
}
