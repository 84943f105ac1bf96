// BFS sources as a kernel argument, and the one-launch BFS of small graphs.
#pragma once

#include "b2sr_internal.cuh"

namespace b2sr {

constexpr int kParamSources = 64;
struct SourceList {
    int32_t v[kParamSources];
};

// Runs the search in one cluster if the graph is small enough for it (tile_dim
// 4 or 8): *finished, or *rounds_run rounds (0: none, nothing was done) after
// which kept (device, 2 ceil(n/32) words) holds the frontier and the visited
// set.  active: a device word for the search's use.  At most max_rounds rounds,
// then B2SR_ERR_NOT_CONVERGED.
b2sr_status bfs_cluster(const b2sr_matrix* h, const SourceList& srcs, int nsrc, int32_t* levels, int64_t max_rounds,
                        uint32_t* kept, int32_t* active, cudaStream_t s, bool* finished, int64_t* rounds_run);

}  // namespace b2sr
