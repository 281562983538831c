// The FP32 sweeps of a small graph in one thread-block cluster
// (sweep_cluster.cu), for ssm_iterate.
#pragma once
#include "common.cuh"

namespace ssm {

// Enqueues `iters` sweeps on pos (float2[n]) in one launch and sets *blocks to
// the cluster's size; *blocks == 0, and nothing enqueued, when the graph is
// not one for it.  dmax: the largest d_ip entry; long_rows: rows of more than
// kMidDeg entries.
int launch_sweep_cluster(int32_t n, int64_t m, const int32_t *rowptr, const int32_t *colidx, int32_t k,
                         const int32_t *pivots, const uint16_t *dip, const int32_t *cnt_off, const uint32_t *cnt,
                         int32_t dmax, int32_t long_rows, float2 *pos, int32_t iters, double tol, int32_t *iters_done,
                         double *rel_change, int32_t *status, cudaStream_t s, int *blocks);

}  // namespace ssm
