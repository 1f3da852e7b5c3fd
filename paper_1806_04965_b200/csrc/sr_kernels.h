// Launch wrappers shared between the API layer and the kernel files.
#pragma once
#include <cuda_runtime.h>

#include "sr_internal.h"

int sr_launch_direct_group(const sr_graph* g, int group, cudaStream_t s);
int sr_launch_input(const sr_graph* g, const SrFrameArgs& fr, unsigned copies, unsigned stems_R, bool beside, cudaStream_t s);
void sr_launch_set_ctl(const sr_graph* g, const SrFrameCtl& v, cudaStream_t s);
void sr_launch_advance(const sr_graph* g, int n, cudaStream_t s);
int sr_direct_conv_pixels_per_block();
int sr_direct_dense_outputs_per_block();
int sr_direct_dense_samples_per_block();
bool sr_head_takes(const sr_graph* g, int v);
int sr_launch_heads(const sr_graph* g, int group, cudaStream_t s);      // returns launches queued
bool sr_input_share_sm();
bool sr_direct_share_sm();
