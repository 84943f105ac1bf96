// BFS sources as a kernel argument, and the one-launch BFS of small graphs.
#pragma once

#include "b2sr_internal.cuh"

namespace b2sr {

constexpr int kParamSources = 64;
struct SourceList {
    int32_t v[kParamSources];
};

// Runs the search in one cluster and sets *taken if the graph is small enough
// for it (tile_dim 4 or 8); *taken false: nothing was done.  At most
// max_rounds rounds, then B2SR_ERR_NOT_CONVERGED.
b2sr_status bfs_cluster(const b2sr_matrix* h, const SourceList& srcs, int nsrc, int32_t* levels, int64_t max_rounds,
                        cudaStream_t s, bool* taken);

}  // namespace b2sr
