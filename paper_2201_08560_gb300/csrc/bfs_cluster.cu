// BFS of a small graph in one launch: the level loop of bfs_sources (Sec. V
// BFS, Boolean SpMV with the visited set as a complemented mask) inside one
// thread-block cluster.
//
// A round of the launched loop is three kernels and their gaps, 10 to 15 us
// whatever the graph, so a search of a small graph costs its launches (R-MAT
// 12, k = 8: 194 us, of which the tiles are 0.85 MB a round).  Here the
// cluster's blocks keep the frontier, the visited set and a partial next
// frontier as bitsets in shared memory and meet twice a round at the cluster
// barrier:
//   * the chunks of tiles are dealt to the warps; a lane ORs 8 consecutive
//     tiles row by row into its block's partial next frontier (shared atomics:
//     a row may cross lanes, chunks and blocks, so nothing needs joining);
//   * each block joins a slice of the partial frontiers through distributed
//     shared memory, drops visited vertices, writes their levels, and hands
//     the slice to every block.
// All waits are cluster barriers of co-scheduled blocks.  A launch runs at most
// kLaunchRounds rounds; a longer search keeps its two sets in device memory
// between launches, and goes on in launched rounds if the graph is large: the
// cluster is 16 of 152 SMs, and a round of it takes about 2 us more for every
// chunk that a warp holds, a launched round hardly more (random graphs of 256
// vertices in a row, permuted ids, k = 8, us a search in the cluster / launched
// after 64 rounds: 3 chunks a warp 2,341 / 3,002, 5 chunks 4,937 / 4,837, 6
// chunks 4,221 / 3,749, 8 chunks 6,544 / 5,046, 12 chunks 26,222 / 14,838, after 16 rounds 14,189;
// ring of twelve neighbours a vertex, 6 chunks: 42,641 / 49,234).
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "bfs_cluster.cuh"

namespace cg = cooperative_groups;

namespace b2sr {

constexpr int kClusterThreads = 1024;
constexpr int kClusterWarps = kClusterThreads / 32;
constexpr int kClusterRuns = 16;              // chunks a warp holds at most
constexpr int64_t kClusterMaxN = 256 * 1024;  // three bitsets of n bits a block
constexpr int kMaxCluster = 16;
constexpr int kLaunchRounds = 64;             // multiples of the launched loop's four
constexpr int kShortRuns = 8;                 // and where more than kShortRounds rounds do
constexpr int kShortRounds = 16;
constexpr int kLongRuns = 6;                  // chunks a warp holds where long searches stay here

// dynamic shared memory of a block: frontier, visited and partial bitsets, and
// each lane's first tile-row in each of its chunks
static size_t cluster_smem(int64_t n, int runs) {
    return (size_t)ceil_div(n, 32) * 12 + (size_t)runs * kClusterThreads * sizeof(int32_t);
}

template <int K>
__global__ void __launch_bounds__(kClusterThreads) bfs_cluster_kernel(const int32_t* __restrict__ rowptr,
                                                                      const int32_t* __restrict__ colind,
                                                                      const uint8_t* __restrict__ tiles, int32_t T,
                                                                      int32_t ntr, int32_t n, int32_t nchunks,
                                                                      SourceList srcs, int nsrc, int64_t begin,
                                                                      int rounds, int32_t* __restrict__ levels,
                                                                      uint32_t* __restrict__ kept,
                                                                      int32_t* __restrict__ active) {
    constexpr int TW = K / 4;  // 32-bit words a tile
    constexpr int CT = chunk_tiles(K);
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int found_by[kMaxCluster];
    cg::cluster_group cluster = cg::this_cluster();
    const int blocks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int words = (n + 31) / 32;
    uint32_t* front = smem;
    uint32_t* vis = smem + words;
    uint32_t* part = smem + 2 * words;
    int32_t* first_row = reinterpret_cast<int32_t*>(smem + 3 * words);
    const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
    const int32_t stride = blocks * kClusterWarps;

    const bool fresh = begin == 1;  // the search's first launch
    for (int w = threadIdx.x; w < 3 * words; w += kClusterThreads) smem[w] = fresh || w >= 2 * words ? 0u : kept[w];
    for (int64_t v = fresh ? (int64_t)rank * kClusterThreads + threadIdx.x : n; v < n;
         v += (int64_t)blocks * kClusterThreads)
        levels[v] = -1;
    int run = 0;
    for (int32_t c = rank * kClusterWarps + warp; c < nchunks; c += stride, ++run) {
        const int32_t t = min(c * CT + lane * 8, T - 1);
        int32_t lo = 0, hi = ntr - 1;  // the last tile-row starting at or before t
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo + 1) >> 1);
            if (__ldg(rowptr + mid) <= t) lo = mid; else hi = mid - 1;
        }
        first_row[run * kClusterThreads + threadIdx.x] = lo;
    }
    __syncthreads();
    for (int i = fresh ? threadIdx.x : nsrc; i < nsrc; i += kClusterThreads) {
        const int32_t v = srcs.v[i];
        atomicOr(front + (v >> 5), 1u << (v & 31));
        atomicOr(vis + (v >> 5), 1u << (v & 31));
    }
    cluster.sync();  // every block's sets and all levels are initialised
    if (rank == 0 && fresh)
        for (int i = threadIdx.x; i < nsrc; i += kClusterThreads) levels[srcs.v[i]] = 0;

    const uint8_t* front8 = reinterpret_cast<const uint8_t*>(front);
    const int per = (words + blocks - 1) / blocks;  // words of a block's slice
    bool more = true;
    for (int64_t round = begin; round < begin + rounds && more; ++round) {
        run = 0;
        for (int32_t c = rank * kClusterWarps + warp; c < nchunks; c += stride, ++run) {
            const int32_t tl = c * CT + lane * 8;
            if (tl >= T) continue;
            int32_t row = first_row[run * kClusterThreads + threadIdx.x];
            int32_t next = __ldg(rowptr + row + 1);
            if (next >= tl + 8) {  // one tile-row: nothing to do where all its vertices are visited
                const int left = min(K, n - row * K);
                const uint32_t need = (1u << left) - 1u;
                const uint32_t have = vis[(row * K) >> 5] >> ((row * K) & 31);
                if ((have & need) == need) continue;
            }
            // the arrays are padded to whole chunks
            uint32_t w[8 * TW], cu[8];
            const uint4* src = reinterpret_cast<const uint4*>(tiles + (int64_t)tl * (4 * TW));
#pragma unroll
            for (int q = 0; q < 2 * TW; ++q) {
                const uint4 v = __ldg(src + q);
                w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
            }
            const uint4 c0 = __ldg(reinterpret_cast<const uint4*>(colind + tl));
            const uint4 c1 = __ldg(reinterpret_cast<const uint4*>(colind + tl) + 1);
            cu[0] = c0.x; cu[1] = c0.y; cu[2] = c0.z; cu[3] = c0.w;
            cu[4] = c1.x; cu[5] = c1.y; cu[6] = c1.z; cu[7] = c1.w;
            uint32_t acc[TW];
#pragma unroll
            for (int q = 0; q < TW; ++q) acc[q] = 0u;
            auto flush = [&]() {
                uint32_t hit = 0u;  // bit r: row r of the tile-row has a frontier neighbour
#pragma unroll
                for (int q = 0; q < TW; ++q) {
                    const uint32_t h = (((acc[q] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | acc[q]) & 0x80808080u;
                    hit |= (((h >> 7) * 0x00204081u) >> 21 & 0xFu) << (4 * q);
                    acc[q] = 0u;
                }
                if (hit) atomicOr(part + ((row * K) >> 5), hit << ((row * K) & 31));
            };
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t xs = K == 8 ? front8[cu[i]] : (front8[cu[i] >> 1] >> (4 * (cu[i] & 1u))) & 0xFu;
                const uint32_t rep = xs * 0x01010101u;
#pragma unroll
                for (int q = 0; q < TW; ++q) acc[q] |= w[i * TW + q] & rep;
                if (tl + i + 1 == next) {  // the tile-row ends here; padding tiles after T are zero
                    flush();
                    if (i < 7 && tl + i + 1 < T) {
                        do {
                            ++row;
                            next = __ldg(rowptr + row + 1);
                        } while (next == tl + i + 1);  // empty tile-rows
                    }
                }
            }
            flush();
        }
        cluster.sync();  // the partial frontiers are complete
        int any = 0;
        for (int w = rank * per + threadIdx.x; w < min(words, (rank + 1) * per); w += kClusterThreads) {
            uint32_t b = 0u;
            for (int r = 0; r < blocks; ++r) b |= *cluster.map_shared_rank(part + w, r);
            const uint32_t seen = vis[w];
            b &= ~seen;
            for (int r = 0; r < blocks; ++r) {
                *cluster.map_shared_rank(front + w, r) = b;
                if (b) *cluster.map_shared_rank(vis + w, r) = seen | b;
            }
            any |= b != 0u;
            while (b) {
                const int i = __ffs(b) - 1;
                b &= b - 1;
                levels[w * 32 + i] = (int32_t)round;
            }
        }
        any = __syncthreads_or(any);
        if (threadIdx.x < blocks) *cluster.map_shared_rank(&found_by[rank], threadIdx.x) = any;
        cluster.sync();  // the new frontier is everywhere, and no block reads a partial one any more
        for (int w = threadIdx.x; w < words; w += kClusterThreads) part[w] = 0u;
        more = false;
        for (int r = 0; r < blocks; ++r) more |= found_by[r] != 0;
        __syncthreads();
    }
    if (rank == 0) {
        for (int w = more ? threadIdx.x : 2 * words; w < 2 * words; w += kClusterThreads) kept[w] = smem[w];
        if (threadIdx.x == 0) *active = more ? 1 : 0;
    }
}

// Blocks of the largest cluster the device runs with the kernel's largest
// shared memory (0: none); looked up once per device.
template <int K>
static int cluster_blocks(int device) {
    static std::atomic<int> known[64];  // blocks + 1
    if (device < 0 || device >= 64) return 0;
    int got = known[device].load(std::memory_order_acquire);
    if (got) return got - 1;
    int blocks = 0;
    const int smem = (int)cluster_smem(kClusterMaxN, kClusterRuns);
    if (cudaFuncSetAttribute(bfs_cluster_kernel<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(bfs_cluster_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) {
        for (int want = kMaxCluster; want >= 8 && !blocks; want /= 2) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(want);
            cfg.blockDim = dim3(kClusterThreads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = want;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, bfs_cluster_kernel<K>, &cfg) == cudaSuccess && n > 0) blocks = want;
        }
    }
    cudaGetLastError();  // a device without room for the cluster takes the launched loop
    known[device].store(blocks + 1, std::memory_order_release);
    return blocks;
}

template <int K>
static b2sr_status run_cluster(const b2sr_matrix* h, const SourceList& srcs, int nsrc, int32_t* levels,
                               int64_t max_rounds, uint32_t* kept, int32_t* active, cudaStream_t s, bool* finished,
                               int64_t* rounds_run) {
    const int blocks = cluster_blocks<K>(h->device);
    if (blocks == 0) return B2SR_OK;
    const int64_t runs = ceil_div(h->nchunks, (int64_t)blocks * kClusterWarps);
    if (runs > kClusterRuns) return B2SR_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = cluster_smem(h->n, (int)runs);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const int64_t at_once = runs > kShortRuns ? kShortRounds : kLaunchRounds;
    for (int64_t begin = 1;; begin += at_once) {
        const int rounds = (int)std::min<int64_t>(at_once, max_rounds + 1 - begin);
        B2SR_CUDA_TRY(cudaLaunchKernelEx(&cfg, bfs_cluster_kernel<K>, (const int32_t*)h->rowptr,
                                         (const int32_t*)h->colind, (const uint8_t*)h->tiles, (int32_t)h->T, h->ntr, h->n,
                                         (int32_t)h->nchunks, srcs, nsrc, begin, rounds, levels, kept, active));
        B2SR_LAUNCH_CHECK("bfs_cluster_kernel");
        int32_t more = 0;
        B2SR_CUDA_TRY(cudaMemcpyAsync(&more, active, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        *rounds_run = begin + rounds - 1;
        if (!more) {
            *finished = true;
            return B2SR_OK;
        }
        if (begin + rounds > max_rounds) return fail(B2SR_ERR_NOT_CONVERGED, "exceeded max_iters rounds");
        if (runs > kLongRuns) return B2SR_OK;
    }
}

b2sr_status bfs_cluster(const b2sr_matrix* h, const SourceList& srcs, int nsrc, int32_t* levels, int64_t max_rounds,
                        uint32_t* kept, int32_t* active, cudaStream_t s, bool* finished, int64_t* rounds_run) {
    *finished = false;
    *rounds_run = 0;
    int dev = -1;
    if (h->k > 8 || h->nchunks == 0 || h->n > kClusterMaxN || nsrc > kParamSources ||
        cudaGetDevice(&dev) != cudaSuccess || dev != h->device)
        return B2SR_OK;
    if (h->k == 4)
        return run_cluster<4>(h, srcs, nsrc, levels, max_rounds, kept, active, s, finished, rounds_run);
    return run_cluster<8>(h, srcs, nsrc, levels, max_rounds, kept, active, s, finished, rounds_run);
}

}  // namespace b2sr
