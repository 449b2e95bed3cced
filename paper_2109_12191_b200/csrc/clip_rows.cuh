// One flat matrix of per-example gradients, [B, P] with rows that fit the registers of a thread-block cluster: norm, clip
// and sum with every byte read once (clip_rows.cu).
#pragma once
#include "common.cuh"

namespace dp {

bool clip_rows_eligible(int B, long long P);
size_t clip_rows_workspace_bytes(int B, long long P);       // partial sums of the clusters
// acc += sum_n f_n G[n], f_n = min(1, C / ||G[n]||); norms_out, clip_out optional.  A wait that gives up leaves NaN in
// all of acc and in the norms and factors of its cluster's rows.
// DP_ERR_UNSUPPORTED: the current device holds no cluster of the size it takes; nothing has been launched.
dp_status launch_clip_rows(const float *G, int B, long long P, float C, float *acc, float *norms_out, float *clip_out,
                           void *workspace, cudaStream_t stream);

}  // namespace dp
