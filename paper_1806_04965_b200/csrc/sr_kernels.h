// Launch wrappers shared between the API layer and the kernel files.
#pragma once
#include <cuda_runtime.h>

#include "sr_internal.h"

int sr_launch_direct_group(const sr_graph* g, int group, SrFollow how, cudaStream_t s);
int sr_launch_input(const sr_graph* g, const SrFrameArgs& fr, unsigned copies, unsigned stems_R, SrFollow how, const SrRegion* clear, cudaStream_t s);
void sr_launch_set_ctl(const sr_graph* g, const SrFrameCtl& v, cudaStream_t s);
void sr_launch_advance(const sr_graph* g, int n, cudaStream_t s);
bool sr_direct_untiled(const sr_graph* g, int v);
void sr_direct_conv_items(const sr_graph* g, int v, std::vector<SrDirectItem>& items);
bool sr_direct_sliced(const SrDirectItem& it);
int sr_direct_dense_outputs_per_block();
int sr_direct_dense_samples_per_block();
int sr_head_class(const sr_graph* g, int v);
void sr_describe_heads(sr_graph* g, int group);
// The heads of a group; with_input: the frame input goes with them (copies, stems_R as for sr_launch_input).
bool sr_heads_take_input(const sr_graph* g, int group, const SrFrameArgs& fr, unsigned copies, unsigned stems_R);
int sr_launch_heads(const sr_graph* g, int group, bool with_input, unsigned copies, unsigned stems_R, SrFollow how, cudaStream_t s);      // returns launches queued
bool sr_input_share_sm();
bool sr_direct_share_sm();
