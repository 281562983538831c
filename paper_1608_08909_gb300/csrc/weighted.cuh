// Internal entry points of the weighted-graph search (weighted.cu), shared
// with the stress reducer (distances from sampled sources on weighted graphs).
#pragma once
#include "common.cuh"

namespace ssm {

size_t sssp_slot_bytes(int32_t n);  // the queues of one search
size_t sssp_ws_bytes(int32_t n, int32_t k);  // launch_sssp's workspace
// dist[a*n + v] = least float32 path sum from sources[a] to v, for a < k;
// an unreachable node flags SSM_E_DISCONNECTED.  ws holds
// sssp_ws_bytes(n, k) bytes.
int launch_sssp(int32_t n, const int32_t *rowptr, const int32_t *colidx, const float *elen, int32_t k,
                const int32_t *sources, float *dist, int32_t *status, void *ws, size_t ws_bytes, cudaStream_t s);

// Weighted max/min pivots in one thread-block cluster (wmaxmin_cluster.cu): *ran
// is false, and nothing was enqueued, when the graph is too large for one.
// spill holds wmaxmin_spill_entries(n) words.
size_t wmaxmin_spill_entries(int32_t n);
int launch_wmaxmin_cluster(int32_t n, const int32_t *rowptr, const int32_t *colidx, const float *elen, int32_t k,
                           int32_t start, int32_t *pivots, const float *delta, int32_t *spill, int32_t *status,
                           cudaStream_t s, bool *ran);

}  // namespace ssm
