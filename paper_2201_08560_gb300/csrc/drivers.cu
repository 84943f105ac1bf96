// Graph algorithms over B2SR (Sec. V): BFS (Boolean semiring, visited set as a
// complemented output mask), BFS from a set of sources (which also runs many
// graphs packed block-diagonally in one arena), multi-source BFS (64 frontiers
// per machine word), SSSP (min-plus relaxation rounds), PageRank (plus-times
// with the column-stochastic matrix), connected components (FastSV hooking
// and shortcutting around the min step) and triangle counting (the masked
// count over the rows up to the diagonal, or over the tiles of the lower
// triangle).
//
// Level-synchronous loops run in batches of several rounds, launched one by one
// at first and as a replayed CUDA graph in a longer loop (captured.cuh); each
// round's kernels are gated on a device flag that the round's update kernel
// clears when nothing changes, until the host reads the flag as 0.  One host
// synchronisation covers a batch.
#include <algorithm>
#include <climits>
#include <vector>

#include "b2sr_internal.cuh"
#include "bfs_cluster.cuh"
#include "captured.cuh"

namespace b2sr {
b2sr_status masked_count(const b2sr_matrix* A, const b2sr_matrix* B, const b2sr_matrix* M, int64_t* count,
                         cudaStream_t s, int64_t* pairs);
bool counts_by_rows(const b2sr_matrix* h);
b2sr_status lower_count(const b2sr_matrix* h, int64_t* count, cudaStream_t s);

// ---------------------------------------------------------------------------
// BFS from a set of sources (all at level 0)
// ---------------------------------------------------------------------------
__global__ void bfs_init_kernel(int32_t* levels, int32_t n, uint32_t* fa, uint32_t* fb, uint32_t* visited,
                                int64_t words, LoopFlags* flags) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n || i < words;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i < n) levels[i] = -1;
        if (i < words) { fa[i] = 0u; fb[i] = 0u; visited[i] = 0u; }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *flags = LoopFlags{1, 0, 0, 0u};
}

// Up to kParamSources sources travel as a kernel argument.
static SourceList source_list(const int32_t* srcs, int nsrc) {
    SourceList l = {};
    for (int i = 0; i < nsrc && i < kParamSources; ++i) l.v[i] = srcs[i];
    return l;
}

__global__ void bfs_seed_kernel(const int32_t* srcs, SourceList few, int nsrc, int32_t* levels, uint32_t* frontier,
                                uint32_t* visited) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nsrc; i += gridDim.x * blockDim.x) {
        const int32_t v = srcs ? srcs[i] : few.v[i];
        levels[v] = 0;
        atomicOr(frontier + (v >> 5), 1u << (v & 31));
        atomicOr(visited + (v >> 5), 1u << (v & 31));
    }
}

// A search goes on after `rounds` rounds: its frontier and visited set are there.
__global__ void bfs_resume_kernel(uint32_t* fb, int64_t words, LoopFlags* flags, int32_t rounds) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (int64_t)gridDim.x * blockDim.x)
        fb[i] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) *flags = LoopFlags{1, 0, rounds, 0u};
}

// visited |= next; levels[v] = level+1 for every new vertex; the frontier just
// used is cleared for the next round's output; ends the round
__global__ void bfs_update_kernel(const uint32_t* __restrict__ next, uint32_t* __restrict__ used,
                                  uint32_t* __restrict__ visited, int32_t* __restrict__ levels, int64_t words,
                                  LoopFlags* flags) {
    if (gate_closed(&flags->active)) return;
    const int32_t lv = *reinterpret_cast<const volatile int32_t*>(&flags->level) + 1;
    int any = 0;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words;
         w += (int64_t)gridDim.x * blockDim.x) {
        uint32_t b = next[w];
        used[w] = 0u;
        if (!b) continue;
        any = 1;
        visited[w] |= b;
        while (b) {
            int c = __ffs(b) - 1;
            b &= b - 1;
            levels[w * 32 + c] = lv;
        }
    }
    finish_round(flags, any);
}

b2sr_status bfs_sources(b2sr_matrix* h, const int32_t* srcs_host, int nsrc, int32_t* levels, int max_iters,
                        cudaStream_t s) {
    const int32_t n = h->n;
    const int64_t words = ceil_div(n, 32);
    const int64_t cap = max_iters > 0 ? max_iters : (int64_t)n + 1;
    DevBuf buf(s);
    B2SR_TRY(buf.alloc(sizeof(LoopFlags) + 3 * words * sizeof(uint32_t) + (size_t)nsrc * sizeof(int32_t)));
    LoopFlags* flags = buf.as<LoopFlags>();
    uint32_t* fa = reinterpret_cast<uint32_t*>(flags + 1);
    uint32_t* vis = fa + words;
    uint32_t* fb = vis + words;
    // the round limit is whole batches of four
    bool finished = false;
    int64_t ran = 0;
    B2SR_TRY(bfs_cluster(h, source_list(srcs_host, nsrc), nsrc, levels, round_up(cap + 1, 4), fa, &flags->active, s,
                         &finished, &ran));
    if (finished) return B2SR_OK;
    if (ran > 0) {
        bfs_resume_kernel<<<grid_for(words), 256, 0, s>>>(fb, words, flags, (int32_t)ran);
        B2SR_LAUNCH_CHECK("bfs_resume_kernel");
    } else {
        int32_t* dsrc = nullptr;
        if (nsrc > kParamSources) {
            dsrc = reinterpret_cast<int32_t*>(fb + words);
            B2SR_CUDA_TRY(cudaMemcpyAsync(dsrc, srcs_host, nsrc * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        }
        bfs_init_kernel<<<grid_for(std::max<int64_t>(n, words)), 256, 0, s>>>(levels, n, fa, fb, vis, words, flags);
        B2SR_LAUNCH_CHECK("bfs_init_kernel");
        bfs_seed_kernel<<<(unsigned)ceil_div(nsrc, 256), 256, 0, s>>>(dsrc, source_list(srcs_host, nsrc), nsrc, levels,
                                                                    fa, vis);
        B2SR_LAUNCH_CHECK("bfs_seed_kernel");
    }
    int64_t rounds = 0;
    return run_captured(s, 4, cap + 1 - ran, &flags->active,
                        [&](cudaStream_t cs, int r) -> b2sr_status {
                            uint32_t* f = (r & 1) ? fb : fa;
                            uint32_t* nx = (r & 1) ? fa : fb;
                            B2SR_TRY(spmv_dispatch(h, B2SR_BOOL_OR_AND, B2SR_VEC_BITS, f, B2SR_VEC_BITS, nx, vis, 1,
                                                   nullptr, cs, &flags->active, false));
                            bfs_update_kernel<<<grid_for(words), 256, 0, cs>>>(nx, f, vis, levels, words, flags);
                            B2SR_LAUNCH_CHECK("bfs_update_kernel");
                            return B2SR_OK;
                        },
                        &rounds);
}

// ---------------------------------------------------------------------------
// multi-source BFS, 64 frontiers per vertex
// ---------------------------------------------------------------------------
// The lane word: 64 frontiers (uint64) or, for at most 32 sources, 32 (uint32:
// half the bytes per gather, and the SpMV takes the k = 4 kernel for 4-byte values).
// The frontier's live tile-columns at k = 4: a bit for every four vertices of
// which one is in some lane's frontier, how many are set, and whether that is
// more than half (the SpMM does not look then).
struct LiveState {
    uint32_t count;
    int32_t dense;
};

// The next frontiers of N rounds, written in turn: round r reads the one before
// (the sources' in round 0 of all) and writes set[r % N].  N is four, or two
// where the device has no room for four.
template <class W, int N>
struct Frontiers {
    W* set[N];
};

// Rows without tiles are written by no SpMM: they are zero from the start.
// Unused lanes count as visited, so a vertex every source has reached is all
// ones in the mask and the SpMM can skip its rows.
template <class W, int N>
__global__ void msbfs_init_kernel(int32_t n, int nsrc, Frontiers<W, N> f, W* vis, uint8_t* live, int64_t live_bytes,
                                  LiveState* state, LoopFlags* flags) {
    constexpr int BITS = 8 * (int)sizeof(W);
    const W unused = nsrc < BITS ? (W)~(((W)1 << nsrc) - (W)1) : (W)0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < N; ++q) f.set[q][i] = (W)0;
        vis[i] = unused;
        if (i < live_bytes) live[i] = 0;  // a byte for 32 vertices, rounded up to 16
    }
    if (blockIdx.x == 0) {
        for (int64_t i = n + threadIdx.x; i < live_bytes; i += blockDim.x) live[i] = 0;
        if (threadIdx.x == 0) {
            *flags = LoopFlags{1, 0, 0, 0u};
            *state = LiveState{0u, 0};
        }
    }
}

template <class W>
__global__ void msbfs_seed_kernel(SourceList srcs, int nsrc, W* X, W* vis, uint32_t* live) {
    int s = threadIdx.x;
    if (s < nsrc) {
        int32_t v = srcs.v[s];
        atomicOr(X + v, (W)1 << s);
        atomicOr(vis + v, (W)1 << s);
        atomicOr(live + (v >> 7), 1u << ((v >> 2) & 31));
    }
}

// visited |= next.  A thread takes four consecutive vertices, which share a live
// bit, so a warp's ballot is a live word.
template <class W>
__global__ void msbfs_update_kernel(const W* __restrict__ Y, W* __restrict__ vis, int32_t n, uint32_t* __restrict__ live,
                                    LiveState* state, LoopFlags* flags) {
    if (gate_closed(&flags->active)) return;
    __shared__ uint32_t block_live;
    if (threadIdx.x == 0) block_live = 0u;
    __syncthreads();
    struct alignas(4 * sizeof(W)) Four {
        W w[4];
    };
    uint32_t nlive = 0;
    const int lane = (int)lane_id();
    const int64_t fours = ((int64_t)n + 3) / 4;
    for (int64_t q0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; q0 < fours;
         q0 += (int64_t)gridDim.x * blockDim.x) {  // warp-uniform
        const int64_t q = q0 + lane;
        Four b = {};
        if (q < fours) {  // the arrays are padded to whole fours; past n nothing is set
            b = reinterpret_cast<const Four*>(Y)[q];
            if (4 * q + 4 > n)
                for (int i = 0; i < 4; ++i)
                    if (4 * q + i >= n) b.w[i] = (W)0;
        }
        const bool some = (b.w[0] | b.w[1] | b.w[2] | b.w[3]) != 0;
        if (some) {
            Four o = reinterpret_cast<const Four*>(vis)[q];
#pragma unroll
            for (int i = 0; i < 4; ++i) o.w[i] |= b.w[i];
            reinterpret_cast<Four*>(vis)[q] = o;
        }
        const uint32_t word = __ballot_sync(0xffffffffu, some);
        if (lane == 0) live[q0 >> 5] = word;
        nlive += __popc(word);
    }
    if (lane == 0 && nlive) atomicAdd(&block_live, nlive);
    __syncthreads();
    if (threadIdx.x == 0 && block_live) atomicAdd(&state->count, block_live);
    if (finish_round(flags, nlive != 0u)) {
        const uint32_t total = atomicExch(&state->count, 0u);
        state->dense = 8 * (int64_t)total > n ? 1 : 0;
    }
}

// The levels of what the last N rounds (fewer at a search's end) found.  After
// the first N every level is written, -1 where nothing was
// found, and the sources' 0; later ones only where a round found something, a
// warp going through the lanes that any of its 32 vertices has.  The levels are
// most of a search's output (R-MAT 22, 64 sources: 1.07 GB): filled with -1
// first and written round by round they took 242 us and 113 us a round; here
// the two launches of such a search take 284 us and a round's update 20.
template <class W, int N>
__global__ void msbfs_levels_kernel(Frontiers<W, N> f, const W* __restrict__ vis, int32_t* __restrict__ levels, int32_t n,
                                    int nsrc, const LoopFlags* flags) {
    const int done = flags->level;
    const int base = (done - 1) & ~(N - 1), run = done - base;
    const int lane = (int)lane_id();
    for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; v0 < n;
         v0 += (int64_t)gridDim.x * blockDim.x) {  // warp-uniform
        const int64_t v = v0 + lane;
        W b[4] = {};
#pragma unroll
        for (int q = 0; q < N; ++q) b[q] = v < n && q < run ? f.set[q][v] : (W)0;
        const W found = b[0] | b[1] | b[2] | b[3], one = b[1] | b[3], two = b[2] | b[3];
        const W seen = base == 0 && v < n ? vis[v] : found;
#pragma unroll
        for (int half = 0; half < (int)sizeof(W) / 4; ++half) {
            const int sh = 32 * half * (int)(sizeof(W) > 4);
            const uint32_t hs = (uint32_t)(seen >> sh), hf = (uint32_t)(found >> sh), h1 = (uint32_t)(one >> sh),
                           h2 = (uint32_t)(two >> sh);
            int32_t* out = levels + (int64_t)sh * n + v;
            if (base == 0) {
                const int lanes = min(32, nsrc - sh);
                if (v < n)
#pragma unroll 8
                    for (int s = 0; s < lanes; ++s)
                        out[(int64_t)s * n] = (int32_t)((hs >> s) & 1u) + (int32_t)((hf >> s) & 1u) +
                                              (int32_t)((h1 >> s) & 1u) + 2 * (int32_t)((h2 >> s) & 1u) - 1;
            } else {
                for (uint32_t lanes = __reduce_or_sync(0xffffffffu, hf); lanes; lanes &= lanes - 1u) {
                    const int s = __ffs(lanes) - 1;
                    if ((hf >> s) & 1u)
                        out[(int64_t)s * n] =
                            base + 1 + (int32_t)((h1 >> s) & 1u) + 2 * (int32_t)((h2 >> s) & 1u);
                }
            }
        }
    }
}

static b2sr_status spmm_lanes(b2sr_matrix* h, const unsigned long long* X, unsigned long long* Y,
                              const unsigned long long* M, cudaStream_t s, const int32_t* gate, bool edges,
                              LiveColumns live) {
    return spmm64_dispatch(h, reinterpret_cast<const uint64_t*>(X), reinterpret_cast<uint64_t*>(Y),
                           reinterpret_cast<const uint64_t*>(M), 1, s, gate, edges, nullptr, live);
}
static b2sr_status spmm_lanes(b2sr_matrix* h, const uint32_t* X, uint32_t* Y, const uint32_t* M, cudaStream_t s,
                              const int32_t* gate, bool edges, LiveColumns live) {
    return spmm32_dispatch(h, X, Y, M, 1, s, gate, edges, live);
}

// no_room: the workspace could not be allocated (nothing was done).
template <class W, int N>
static b2sr_status bfs_multi_lanes(b2sr_matrix* h, const int32_t* srcs_host, int nsrc, int32_t* levels,
                                   int max_iters, cudaStream_t s, bool* no_room) {
    const int32_t n = h->n;
    DevBuf buf(s);
    const size_t vb = round_up((size_t)n * sizeof(W), 256);
    const size_t lb = round_up(ceil_div(n, 32), 16);
    const b2sr_status room = buf.alloc((N + 1) * vb + lb + sizeof(LoopFlags) + sizeof(LiveState));
    *no_room = room == B2SR_ERR_OOM;
    B2SR_TRY(room);
    Frontiers<W, N> f;
    for (int q = 0; q < N; ++q) f.set[q] = reinterpret_cast<W*>(buf.as<char>() + q * vb);
    W* vis = reinterpret_cast<W*>(buf.as<char>() + N * vb);
    uint8_t* live = reinterpret_cast<uint8_t*>(buf.as<char>() + (N + 1) * vb);
    LoopFlags* flags = reinterpret_cast<LoopFlags*>(live + lb);
    LiveState* state = reinterpret_cast<LiveState*>(flags + 1);
    const LiveColumns columns{reinterpret_cast<const uint32_t*>(live), &state->dense};
    W* sources = f.set[N - 1];
    msbfs_init_kernel<W, N><<<grid_for(n), 256, 0, s>>>(n, nsrc, f, vis, live, (int64_t)lb, state, flags);
    B2SR_LAUNCH_CHECK("msbfs_init_kernel");
    msbfs_seed_kernel<W><<<1, 64, 0, s>>>(source_list(srcs_host, nsrc), nsrc, sources, vis,
                                          reinterpret_cast<uint32_t*>(live));
    B2SR_LAUNCH_CHECK("msbfs_seed_kernel");
    const int64_t cap = max_iters > 0 ? max_iters : (int64_t)n + 1;
    int64_t rounds = 0;
    return run_captured(s, 4, cap + 1, &flags->active,
                        [&](cudaStream_t cs, int r) -> b2sr_status {
                            const int q = r % N;
                            W* nxt = f.set[q];
                            // rows without tiles are zero in every set from the start, but for the
                            // last's, which may have sources there until a round has written it
                            B2SR_TRY(spmm_lanes(h, f.set[(q + N - 1) % N], nxt, vis, cs, &flags->active, q == N - 1,
                                                columns));
                            msbfs_update_kernel<W><<<grid_for(ceil_div(n, 4), 4), 256, 0, cs>>>(
                                nxt, vis, n, reinterpret_cast<uint32_t*>(live), state, flags);
                            B2SR_LAUNCH_CHECK("msbfs_update_kernel");
                            if (q < N - 1) return B2SR_OK;
                            msbfs_levels_kernel<W, N><<<grid_for(n), 256, 0, cs>>>(f, vis, levels, n, nsrc, flags);
                            B2SR_LAUNCH_CHECK("msbfs_levels_kernel");
                            return B2SR_OK;
                        },
                        &rounds);
}

b2sr_status bfs_multi(b2sr_matrix* h, const int32_t* srcs_host, int nsrc, int32_t* levels, int max_iters,
                      cudaStream_t s) {
    // five lane words a vertex; where they do not fit, three
    auto search = [&](auto lane_word) -> b2sr_status {
        using W = decltype(lane_word);
        bool no_room = false;
        const b2sr_status st = bfs_multi_lanes<W, 4>(h, srcs_host, nsrc, levels, max_iters, s, &no_room);
        if (!no_room) return st;
        clear_error();
        return bfs_multi_lanes<W, 2>(h, srcs_host, nsrc, levels, max_iters, s, &no_room);
    };
    if (nsrc <= 32) return search(uint32_t(0));
    return search(0ull);
}

// ---------------------------------------------------------------------------
// SSSP: d <- min(d, A min.+ d) until no distance changes
// ---------------------------------------------------------------------------
__global__ void sssp_init_kernel(float* d, int32_t n, int32_t src, LoopFlags* flags) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = (i == src) ? 0.0f : INFINITY;
    if (blockIdx.x == 0 && threadIdx.x == 0) *flags = LoopFlags{1, 0, 0, 0u};
}

// found if a distance changed; the round's result becomes the current vector
__global__ void sssp_update_kernel(const float* __restrict__ nxt, float* __restrict__ cur, int32_t n,
                                   LoopFlags* flags) {
    if (gate_closed(&flags->active)) return;
    int diff = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = nxt[i];
        if (v != cur[i]) { diff = 1; cur[i] = v; }
    }
    finish_round(flags, diff);
}

b2sr_status sssp(b2sr_matrix* h, const float* w, int32_t src, float* dist, int max_iters, cudaStream_t s) {
    const int32_t n = h->n;
    if (w) B2SR_TRY(ensure_voff(h, s));  // built before capture: capture must not allocate for the handle
    DevBuf buf(s);
    B2SR_TRY(buf.alloc(sizeof(LoopFlags) + (size_t)n * sizeof(float)));
    LoopFlags* flags = buf.as<LoopFlags>();
    float* tmp = reinterpret_cast<float*>(flags + 1);
    sssp_init_kernel<<<grid_for(n), 256, 0, s>>>(dist, n, src, flags);
    B2SR_LAUNCH_CHECK("sssp_init_kernel");
    const int64_t cap = max_iters > 0 ? max_iters : (int64_t)n + 1;
    int64_t rounds = 0;
    return run_captured(s, 16, cap + 1, &flags->active,
                        [&](cudaStream_t cs, int) -> b2sr_status {
                            B2SR_TRY(spmv_dispatch(h, B2SR_MIN_PLUS, B2SR_VEC_F32, dist, B2SR_VEC_F32, tmp, nullptr, 0, w,
                                                   cs, &flags->active));
                            sssp_update_kernel<<<grid_for(n), 256, 0, cs>>>(tmp, dist, n, flags);
                            B2SR_LAUNCH_CHECK("sssp_update_kernel");
                            return B2SR_OK;
                        },
                        &rounds);
}

// ---------------------------------------------------------------------------
// PageRank
// ---------------------------------------------------------------------------
// x^0 = 1/n; c_j = x_j / outdeg_j (0 without out-edges).  The rounding of
// every operation is spelled out (no contraction left to the compiler), so the
// batched PageRank of the query server reproduces these values bit for bit.
__global__ void pr_init_kernel(float* x, float* c, const int32_t* __restrict__ outdeg, int32_t n) {
    const float x0 = __fdiv_rn(1.0f, (float)n);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        x[i] = x0;
        int32_t d = outdeg[i];
        c[i] = d > 0 ? __fdiv_rn(x0, (float)d) : 0.0f;
    }
}

// x_i = (1-d) t_i + d y_i; c_i = x_i / outdeg_i
__global__ void pr_step_kernel(const float* __restrict__ y, const float* __restrict__ tele,
                               const int32_t* __restrict__ outdeg, float damp, int32_t n, float* __restrict__ x,
                               float* __restrict__ c) {
    const float tu = __fdiv_rn(1.0f, (float)n);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float ti = tele ? tele[i] : tu;
        float xi = __fmaf_rn(damp, y[i], __fmul_rn(1.0f - damp, ti));
        x[i] = xi;
        int32_t d = outdeg[i];
        c[i] = d > 0 ? __fdiv_rn(xi, (float)d) : 0.0f;
    }
}

b2sr_status pagerank(b2sr_matrix* h, float damp, int iters, const float* tele, float* pr, cudaStream_t s) {
    const int32_t n = h->n;
    if (n == 0) return B2SR_OK;
    B2SR_TRY(ensure_outdeg(h, s));
    DevBuf buf(s);
    B2SR_TRY(buf.alloc(2 * (size_t)n * sizeof(float)));
    float* c = buf.as<float>();
    float* y = c + n;
    pr_init_kernel<<<grid_for(n), 256, 0, s>>>(pr, c, h->outdeg, n);
    B2SR_LAUNCH_CHECK("pr_init_kernel");
    for (int it = 0; it < iters; ++it) {
        B2SR_TRY(spmv_dispatch(h, B2SR_PLUS_TIMES, B2SR_VEC_F32, c, B2SR_VEC_F32, y, nullptr, 0, nullptr, s, nullptr));
        pr_step_kernel<<<grid_for(n), 256, 0, s>>>(y, tele, h->outdeg, damp, n, pr, c);
        B2SR_LAUNCH_CHECK("pr_step_kernel");
    }
    return B2SR_OK;
}

// ---------------------------------------------------------------------------
// connected components: FastSV (Zhang, Azad, Hu; the linear-algebraic CC the
// paper follows in Sec. V), with the min step as a B2SR SpMV
// ---------------------------------------------------------------------------
__global__ void cc_init_kernel(int32_t* f, int32_t* gf, int32_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        f[i] = (int32_t)i;
        gf[i] = (int32_t)i;
    }
}

// stochastic hooking: f[f[i]] = min(f[f[i]], mngf[i])
__global__ void cc_hook_kernel(int32_t* f, const int32_t* __restrict__ mngf, int32_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t fi = f[i];
        int32_t m = mngf[i];
        if (m < fi) atomicMin(f + fi, m);
    }
}

// aggressive hooking and shortcutting: f[i] = min(f[i], mngf[i], gf[i])
__global__ void cc_short_kernel(int32_t* f, const int32_t* __restrict__ mngf, const int32_t* __restrict__ gf,
                                int32_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        f[i] = min(f[i], min(mngf[i], gf[i]));
}

// gf' = f[f]; flag if any grandparent changed
__global__ void cc_grand_kernel(const int32_t* __restrict__ f, const int32_t* __restrict__ gf, int32_t* __restrict__ gfn,
                                int32_t n, int32_t* any) {
    int diff = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t g = f[f[i]];
        gfn[i] = g;
        diff |= (g != gf[i]);
    }
    if (__syncthreads_or(diff) && threadIdx.x == 0) atomicOr(any, 1);
}

b2sr_status cc(b2sr_matrix* h, int32_t* labels, int max_iters, cudaStream_t s) {
    const int32_t n = h->n;
    if (n == 0) return B2SR_OK;
    DevBuf buf(s);
    const size_t vb = round_up((size_t)n * sizeof(int32_t), 256);  // each vector 256-byte aligned
    B2SR_TRY(buf.alloc(3 * vb + 256));
    int32_t* gf = buf.as<int32_t>();
    int32_t* gfn = reinterpret_cast<int32_t*>(buf.as<char>() + vb);
    int32_t* mngf = reinterpret_cast<int32_t*>(buf.as<char>() + 2 * vb);
    int32_t* any = reinterpret_cast<int32_t*>(buf.as<char>() + 3 * vb);
    int32_t* f = labels;
    cc_init_kernel<<<grid_for(n), 256, 0, s>>>(f, gf, n);
    B2SR_LAUNCH_CHECK("cc_init_kernel");
    HostFlag hf;
    const int cap = max_iters > 0 ? max_iters : n;
    for (int it = 0; it <= cap; ++it) {
        B2SR_TRY(spmv_dispatch(h, B2SR_MIN_PLUS, B2SR_VEC_I32, gf, B2SR_VEC_I32, mngf, nullptr, 0, nullptr, s, nullptr));
        cc_hook_kernel<<<grid_for(n), 256, 0, s>>>(f, mngf, n);
        B2SR_LAUNCH_CHECK("cc_hook_kernel");
        cc_short_kernel<<<grid_for(n), 256, 0, s>>>(f, mngf, gf, n);
        B2SR_LAUNCH_CHECK("cc_short_kernel");
        B2SR_CUDA_TRY(cudaMemsetAsync(any, 0, sizeof(int32_t), s));
        cc_grand_kernel<<<grid_for(n), 256, 0, s>>>(f, gf, gfn, n, any);
        B2SR_LAUNCH_CHECK("cc_grand_kernel");
        int32_t got = 0;
        B2SR_TRY(read_flag(any, hf, s, &got));
        std::swap(gf, gfn);
        if (!got) return B2SR_OK;
    }
    return fail(B2SR_ERR_NOT_CONVERGED, "CC exceeded max_iters rounds");
}

// ---------------------------------------------------------------------------
// many graphs in one block-diagonal arena
// ---------------------------------------------------------------------------
// rowptr of graph g placed at rows [base, base + ng), padding rows after it
// empty; its column ids shifted by base.
__global__ void arena_rows_kernel(const int32_t* __restrict__ rp, int32_t ng, int32_t base, int32_t npad,
                                  int64_t eoff, int32_t* __restrict__ out_rp) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < npad;
         i += (int64_t)gridDim.x * blockDim.x)
        out_rp[base + i] = (int32_t)(eoff + rp[i < ng ? i : ng]);
}

__global__ void arena_cols_kernel(const int32_t* __restrict__ ci, int64_t nnz, int32_t base,
                                  int32_t* __restrict__ out_ci) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        out_ci[e] = ci[e] + base;
}

}  // namespace b2sr

using namespace b2sr;

extern "C" b2sr_status b2sr_bfs(b2sr_handle h, int32_t src, int32_t* levels, int max_iters, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (src < 0 || src >= h->n) return fail(B2SR_ERR_INVALID_ARG, "source out of range");
    if (!levels) return fail(B2SR_ERR_INVALID_ARG, "levels is NULL");
    return bfs_sources(h, &src, 1, levels, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_bfs_sources(b2sr_handle h, const int32_t* srcs_host, int nsrc, int32_t* levels,
                                        int max_iters, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (nsrc < 1 || !srcs_host || !levels) return fail(B2SR_ERR_INVALID_ARG, "need at least one source and levels");
    for (int i = 0; i < nsrc; ++i)
        if (srcs_host[i] < 0 || srcs_host[i] >= h->n) return fail(B2SR_ERR_INVALID_ARG, "source out of range");
    return bfs_sources(h, srcs_host, nsrc, levels, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_bfs_multi(b2sr_handle h, const int32_t* srcs_host, int nsrc, int32_t* levels,
                                      int max_iters, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (nsrc < 1 || nsrc > 64) return fail(B2SR_ERR_INVALID_ARG, "nsrc must be in [1, 64]");
    if (!srcs_host || !levels) return fail(B2SR_ERR_INVALID_ARG, "null pointer");
    for (int i = 0; i < nsrc; ++i)
        if (srcs_host[i] < 0 || srcs_host[i] >= h->n) return fail(B2SR_ERR_INVALID_ARG, "source out of range");
    return bfs_multi(h, srcs_host, nsrc, levels, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_sssp(b2sr_handle h, const float* weights, int32_t src, float* dist, int max_iters,
                                 void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (src < 0 || src >= h->n) return fail(B2SR_ERR_INVALID_ARG, "source out of range");
    if (!dist) return fail(B2SR_ERR_INVALID_ARG, "dist is NULL");
    return sssp(h, weights, src, dist, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_pagerank(b2sr_handle h, float d, int iters, const float* teleport, float* pr,
                                     void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (!pr && h->n > 0) return fail(B2SR_ERR_INVALID_ARG, "pr is NULL");
    if (iters < 0 || !(d >= 0.0f && d <= 1.0f)) return fail(B2SR_ERR_INVALID_ARG, "bad iters or damping");
    return pagerank(h, d, iters, teleport, pr, to_stream(stream));
}

extern "C" b2sr_status b2sr_cc(b2sr_handle h, int32_t* labels, int max_iters, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (!labels && h->n > 0) return fail(B2SR_ERR_INVALID_ARG, "labels is NULL");
    return cc(h, labels, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_tc(b2sr_handle h, int64_t* count, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (!count) return fail(B2SR_ERR_INVALID_ARG, "count is NULL");
    if (counts_by_rows(h)) {
        const b2sr_status st = lower_count(h, count, to_stream(stream));
        if (st != B2SR_ERR_OOM) return st;
        clear_error();  // the tile form needs L alone
    }
    b2sr_handle L = nullptr;
    B2SR_TRY(b2sr_lower(h, stream, &L));
    b2sr_status st = masked_count(L, L, L, count, to_stream(stream), nullptr);
    b2sr_destroy(L);
    return st;
}

extern "C" b2sr_status b2sr_from_csr_batch(int ngraphs, const int32_t* n_host, const int32_t* const* rowptrs,
                                           const int32_t* const* colinds, const int64_t* nnz_host, int tile_dim,
                                           void* stream, b2sr_handle* out, int64_t* base_host) {
    clear_error();
    if (!out) return fail(B2SR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (ngraphs < 1 || !n_host || !rowptrs || !colinds || !nnz_host || !base_host)
        return fail(B2SR_ERR_INVALID_ARG, "null pointer or no graphs");
    if (!valid_tile(tile_dim)) return fail(B2SR_ERR_UNSUPPORTED_TILE, "tile_dim must be 4, 8, 16 or 32");
    cudaStream_t s = to_stream(stream);
    int64_t N = 0, NNZ = 0;
    for (int g = 0; g < ngraphs; ++g) {
        if (n_host[g] < 0 || nnz_host[g] < 0 || !rowptrs[g] || (nnz_host[g] > 0 && !colinds[g]))
            return fail(B2SR_ERR_INVALID_ARG, "bad graph " + std::to_string(g));
        base_host[g] = N;
        N += round_up(n_host[g], 32);
        NNZ += nnz_host[g];
    }
    base_host[ngraphs] = N;
    if (N >= (int64_t(1) << 31) || NNZ >= (int64_t(1) << 31)) return fail(B2SR_ERR_INVALID_ARG, "arena too large");
    // every graph's own CSR is checked before it is shifted into the arena: a
    // column outside [0, n_g) would otherwise land in a neighbouring graph
    {
        DevBuf bad(s);
        B2SR_TRY(bad.alloc((size_t)ngraphs * sizeof(int)));
        B2SR_CUDA_TRY(cudaMemsetAsync(bad.p, 0, (size_t)ngraphs * sizeof(int), s));
        for (int g = 0; g < ngraphs; ++g)
            B2SR_TRY(validate_csr_async(n_host[g], rowptrs[g], colinds[g], nnz_host[g], bad.as<int>() + g, s));
        std::vector<int> hbad((size_t)ngraphs);
        B2SR_CUDA_TRY(cudaMemcpyAsync(hbad.data(), bad.p, (size_t)ngraphs * sizeof(int), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        for (int g = 0; g < ngraphs; ++g)
            if (hbad[g]) return fail(B2SR_ERR_INVALID_ARG, "malformed CSR in graph " + std::to_string(g));
    }
    DevBuf rp(s), ci(s);
    B2SR_TRY(rp.alloc((N + 1) * sizeof(int32_t)));
    B2SR_TRY(ci.alloc(std::max<int64_t>(NNZ, 1) * sizeof(int32_t)));
    int64_t eoff = 0;
    for (int g = 0; g < ngraphs; ++g) {
        const int32_t npad = (int32_t)round_up(n_host[g], 32);
        if (npad > 0) {
            arena_rows_kernel<<<grid_for(npad), 256, 0, s>>>(rowptrs[g], n_host[g], (int32_t)base_host[g], npad, eoff,
                                                            rp.as<int32_t>());
            B2SR_LAUNCH_CHECK("arena_rows_kernel");
        }
        if (nnz_host[g] > 0) {
            arena_cols_kernel<<<grid_for(nnz_host[g]), 256, 0, s>>>(colinds[g], nnz_host[g], (int32_t)base_host[g],
                                                                   ci.as<int32_t>() + eoff);
            B2SR_LAUNCH_CHECK("arena_cols_kernel");
        }
        eoff += nnz_host[g];
    }
    const int32_t last = (int32_t)NNZ;
    B2SR_CUDA_TRY(cudaMemcpyAsync(rp.as<int32_t>() + N, &last, sizeof(int32_t), cudaMemcpyHostToDevice, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));  // `last` lives on this stack frame
    return b2sr_from_csr((int32_t)N, rp.as<int32_t>(), ci.as<int32_t>(), NNZ, tile_dim, stream, out);
}
