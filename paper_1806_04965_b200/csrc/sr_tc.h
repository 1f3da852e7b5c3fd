// Tensor-core engine (tcgen05 implicit GEMM) as the API layer sees it.
#pragma once
#include <cuda_runtime.h>

#include "sr_internal.h"

void sr_tc_select_nodes(sr_graph* g);                         // sets SrHostNode::use_tc
sr_status sr_tc_plan(sr_graph* g, size_t& offset);            // reserves workspace regions
sr_status sr_tc_bind(sr_graph* g);                            // uploads tile tables and tensor maps
sr_status sr_tc_set_weights(sr_graph* g, int edge, const float* w_eff /* [C_out][k][k][C_in], host */);
bool sr_tc_stages(const sr_graph* g, int edge);               // the edge is staged (see sr_input.cu): its target reads im2col rows
int sr_tc_launch_group(sr_graph* g, int group, SrFollow how, cudaStream_t s);          // returns launches queued
bool sr_tc_group_has_work(const sr_graph* g, int group);
void sr_tc_describe(const sr_graph* g, int group, sr_launch_plan* out);
sr_status sr_tc_timing(sr_graph* g, double* ms, long long* launches);
void sr_tc_destroy(sr_graph* g);
