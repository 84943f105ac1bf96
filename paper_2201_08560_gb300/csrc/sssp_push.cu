// SSSP by frontier-driven push relaxation over the transposed bit tiles.
//
// b2sr_sssp relaxes every edge in every round (a min-plus SpMV over the whole
// matrix, Sec. V SSSP).  On graphs of large hop diameter -- a 4096 x 4096
// grid needs about 8,000 rounds -- nearly all of that work is wasted: only
// the vertices whose distance dropped in the previous round can improve a
// neighbour.  This driver keeps that set as a bitset plus a list of the
// tile-rows holding it, and pushes only from them.  It reads B2SR of the
// transpose, A^T: tile-row J of A^T lists, in its bits, the out-edges of the
// vertices kJ .. kJ+k-1 (for a symmetric matrix A^T = A and the handle serves
// as its own transpose).
//
// One round: a warp per active tile-row J deals its tiles to the lanes, the
// active source rows of a tile to several lanes where there are few tiles; for
// every set bit (r, c) in an active row r of a tile (J, I) the target kI+c is
// relaxed with dist[kJ+r] + w by an integer atomicMin on the
// float's bits (non-negative floats order like their bit patterns).  A target
// that improves is marked in the next set: a bitset, and a list of the
// tile-rows that hold its bits, appended by whoever sets the first bit of a
// tile-row.  With delta > 0 the rounds keep a threshold: a vertex whose
// distance is at or past it goes to a far set instead, where it costs nothing
// until the near set runs dry; then the threshold rises by delta and the far
// set becomes the next round's active set (delta-stepping's buckets as a
// near/far pair of worklists).  The three sets change roles through words in
// device memory, so nothing is copied between them, and a set is cleared as it
// is read.  Distances only decrease, and every value written is the length of
// a path, so the result is the shortest-path fixed point whatever the order of
// the atomics: bit-exact and the same as b2sr_sssp's.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "b2sr_internal.cuh"
#include "captured.cuh"

namespace cg = cooperative_groups;

namespace b2sr {

constexpr int kPushThreads = 256;
constexpr int kPushWarps = kPushThreads / 32;

// A vertex set: bitset, and the tile-rows holding its bits, each once.
struct PushSet {
    uint32_t* act;
    int32_t* list;
};

// Loop state (device).  Round r reads state[r & 1], written by round r - 1,
// works out its own from it, and its first block writes state[(r + 1) & 1]: no
// block waits for another.  cur, nxt and far name the sets in their roles.
struct PushState {
    int32_t cur, nxt, far;
    int32_t active;  // 0: nothing was left to do
    int32_t epoch;   // which far counters are in use
    float theta;     // threshold (infinite without buckets)
    int32_t rounds;  // rounds run
    int32_t busy;    // the cluster left a round with too many rows for it
    unsigned long long worked;  // active tile-rows summed over the rounds
};
// Counters, each on a line of its own.  near[r & 3] is the length of the list
// that round r builds; a round clears the one of the round after it.  far and
// farmin (the least distance in the far set, float bits) go by epoch, which
// changes when the far set becomes the active one; the change clears the
// epoch after the new one.  So no round changes what its late blocks read.
struct alignas(128) PushCounter {
    int32_t v;
};
struct PushControl {
    alignas(128) PushState state[2];
    PushCounter near[4], far[4], farmin[4];
};

// Position of the i-th set bit of m (i below the number of set bits).
__device__ __forceinline__ int nth_bit(uint32_t m, int i) {
    int pos = 0;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const int below = __popc((m >> pos) & ((1u << w) - 1u));
        if (i >= below) {
            i -= below;
            pos += w;
        }
    }
    return pos;
}

// Row r of tile t, and the set bits of its earlier rows (the row's first weight
// is that far from the tile's).
template <int K>
__device__ __forceinline__ uint32_t tile_row_of(const uint8_t* __restrict__ tiles, int32_t t, int r) {
    if constexpr (K == 4) return (__ldg(reinterpret_cast<const uint32_t*>(tiles) + t) >> (8 * r)) & 0xFu;
    else if constexpr (K == 8) return (uint32_t)(__ldg(reinterpret_cast<const unsigned long long*>(tiles) + t) >> (8 * r)) & 0xFFu;
    else if constexpr (K == 16) return __ldg(reinterpret_cast<const uint16_t*>(tiles) + (int64_t)t * 16 + r);
    else return __ldg(reinterpret_cast<const uint32_t*>(tiles) + (int64_t)t * 32 + r);
}
template <int K>
__device__ __forceinline__ int ones_before(const uint8_t* __restrict__ tiles, int32_t t, int r) {
    if constexpr (K == 4) {
        return __popc(__ldg(reinterpret_cast<const uint32_t*>(tiles) + t) & ((1u << (8 * r)) - 1u));
    } else if constexpr (K == 8) {
        return __popcll(__ldg(reinterpret_cast<const unsigned long long*>(tiles) + t) & ((1ull << (8 * r)) - 1ull));
    } else {
        constexpr int TB = K == 16 ? 32 : 128;
        const uint4* p = reinterpret_cast<const uint4*>(tiles + (int64_t)t * TB);
        const int bits = r * K;  // of the tile
        int ones = 0;
        for (int q = 0; 128 * q < bits; ++q) {
            const uint4 v = __ldg(p + q);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int left = bits - 128 * q - 32 * i;
                if (left > 0) ones += __popc(left >= 32 ? w[i] : w[i] & ((1u << left) - 1u));
            }
        }
        return ones;
    }
}

// Rows of tile t that are not empty, k = 16 and 32.
template <int K>
__device__ __forceinline__ uint32_t rows_with_bits(const uint8_t* __restrict__ tiles, int32_t t) {
    constexpr int TB = K == 16 ? 32 : 128;
    const uint4* p = reinterpret_cast<const uint4*>(tiles + (int64_t)t * TB);
    uint32_t rows = 0u;
#pragma unroll
    for (int q = 0; q < TB / 16; ++q) {
        const uint4 v = __ldg(p + q);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (K == 32) {
                if (w[i]) rows |= 1u << (4 * q + i);
            } else {
                if (w[i] & 0xFFFFu) rows |= 1u << (8 * q + 2 * i);
                if (w[i] >> 16) rows |= 2u << (8 * q + 2 * i);
            }
        }
    }
    return rows;
}

// The tile-rows a block appends to one list: kept in shared memory, appended
// at the block's end with one global atomic (directly once the buffer is full).
template <int CAP>
struct Appends {
    int32_t n, base;
    int32_t row[CAP];
};
constexpr int kPushBuffer = 512;

template <int K, int CAP>
__device__ __forceinline__ void mark_bits(const PushSet& s, int32_t* count, Appends<CAP>& ap, int32_t J, uint32_t bits) {
    constexpr int per = 32 / K;
    constexpr uint32_t seg = K == 32 ? 0xFFFFFFFFu : (1u << (K & 31)) - 1u;
    const int sh = (J % per) * K;
    const uint32_t old = atomicOr(s.act + J / per, bits << sh);
    if (((old >> sh) & seg) != 0u) return;  // listed by whoever set the tile-row's first bit
    const int32_t at = atomicAdd(&ap.n, 1);
    if (at < CAP) ap.row[at] = J;
    else s.list[atomicAdd(count, 1)] = J;
}

// Entries a tile from which lanes take single rows: R-MAT 12 and 14, k = 32 (7 and
// 4 a tile), unit weights, us a search by pairs / by tiles: 430 / 661, 1,190 /
// 1,448; R-MAT 14, k = 16 (2.4), is no faster by pairs.
constexpr int64_t kPairEntries = 3;

struct PushGraph {  // the transpose's arrays, the edge weights (w null: 1) and the distances
    const int32_t *rowptr, *colind;
    const uint8_t* tiles;
    const int32_t* voff;
    const float* w;
    float* dist;
    int32_t n;
    int pairs;  // tiles hold kPairEntries or more on average
};

// When the near list has run dry: the threshold rises by delta -- or, past a
// gap in the distances, to the least far distance plus delta, so that the
// nearest waiting vertex always gets in -- and the far set becomes the active
// one (whatever is still past the threshold moves back).
__device__ __forceinline__ void raise_threshold(PushState& p, float fm, float delta) {
    const float th = p.theta;
    float nt = fmaxf(th + delta, fm + delta);
    if (!(nt > fm)) nt = nextafterf(fm, INFINITY);  // delta below the spacing of floats there
    if (!(nt > th)) nt = nextafterf(th, INFINITY);
    p.theta = nt;
    const int32_t t = p.cur;
    p.cur = p.far;
    p.far = t;
    p.epoch = (p.epoch + 1) & 3;
}

// Relaxes the out-edges of tile-row J's active vertices; called by the `width`
// lanes of `group`, `sub` within it; du: a float for each of them in shared
// memory.  A chain of dependent memory accesses (segment, row pointers and
// distances; tiles; weights; two atomics), so a lane issues up to kBatch
// relaxations side by side, and the lanes take one (tile, active row) pair each
// where a tile-row has few of them (a mesh's has five tiles) or tiles hold
// several entries (g.pairs).  Elsewhere most pairs are empty, and a tile goes to
// one lane with all its active rows, or to as many as there are to a tile: one
// lane a pair went through every tile once an active row (random graph of 2^15
// vertices, k = 16: 6.3 ms against 1.3).  far_seen: the least distance sent to
// the far set.
template <int K, int NEAR, int FAR>
__device__ __forceinline__ void push_row(const PushGraph& g, const PushSet& cur, const PushSet& nxt, const PushSet& far,
                                         int32_t* near_count, int32_t* far_count, Appends<NEAR>& add_near,
                                         Appends<FAR>& add_far, float th, int buckets, int32_t J, int width,
                                         unsigned group, int sub, float* du, float& far_seen) {
    constexpr int per = 32 / K;
    constexpr uint32_t seg = K == 32 ? 0xFFFFFFFFu : (1u << (K & 31)) - 1u;
    constexpr int kBatch = 4;
    const int sh = (J % per) * K;
    uint32_t amask = (__ldcg(cur.act + J / per) >> sh) & seg;
    const int32_t t0 = __ldg(g.rowptr + J), t1 = __ldg(g.rowptr + J + 1);
    // the sources' distances (the bitset has no bits past n)
    float mine_du = 0.0f;
    if (sub < K && (int64_t)J * K + sub < g.n) mine_du = __ldcg(g.dist + (int64_t)J * K + sub);
    __syncwarp(group);  // every lane has read the segment, and is done with the row before
    if (sub == 0) atomicAnd(cur.act + J / per, ~(seg << sh));
    if (buckets) {
        // active vertices at or past the threshold move to the far set
        const bool late = sub < K && ((amask >> sub) & 1u) && mine_du >= th;
        const uint32_t defer = __ballot_sync(group, late) >> (lane_id() - sub);
        if (late) far_seen = fminf(far_seen, mine_du);
        const uint32_t mine = defer & seg;
        if (mine && sub == 0) mark_bits<K>(far, far_count, add_far, J, mine);
        amask &= ~mine;
    }
    const int na = __popc(amask);
    if (na == 0) return;
    const int32_t nt = t1 - t0;
    // a batch of relaxations: targets' columns (-1: none) and distances through the tile
    int c[kBatch];
    float cand[kBatch];
    auto relax = [&](int32_t I) {
        int old[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
            if (c[q] >= 0)
                old[q] = atomicMin(reinterpret_cast<int*>(g.dist) + (int64_t)I * K + c[q], __float_as_int(cand[q]));
        uint32_t near_bits = 0u, far_bits = 0u;
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
            if (c[q] >= 0 && cand[q] < __int_as_float(old[q])) {
                if (cand[q] >= th) {
                    far_seen = fminf(far_seen, cand[q]);
                    far_bits |= 1u << c[q];
                } else {
                    near_bits |= 1u << c[q];
                }
            }
        if (near_bits) mark_bits<K>(nxt, near_count, add_near, I, near_bits);
        if (far_bits) mark_bits<K>(far, far_count, add_far, I, far_bits);
    };
    // the entries of one row, from distance d; wt: the row's weights
    auto relax_row = [&](int32_t I, uint32_t bits, float d, const float* wt) {
        while (bits) {
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                c[q] = -1;
                if (bits) {
                    c[q] = __ffs(bits) - 1;
                    bits &= bits - 1;
                    cand[q] = d + (wt ? __ldg(wt + q) : 1.0f);
                }
            }
            if (wt) wt += kBatch;
            relax(I);
        }
    };
    if (g.pairs || (int64_t)nt * na <= 2 * width) {  // the same for the group
        const int64_t pairs = (int64_t)nt * na;
        int32_t ti = sub / na;
        int ri = sub - ti * na;
        const int32_t dt = width / na;
        const int dr = width - dt * na;
        for (int64_t p = 0; p < pairs; p += width) {
            const bool live = p + sub < pairs;
            const int r = live ? nth_bit(amask, ri) : 0;
            const float d = __shfl_sync(group, mine_du, r, width);
            if (live) {
                const int32_t t = t0 + ti;
                const int32_t I = __ldg(g.colind + t);
                const float* wt = g.w ? g.w + __ldg(g.voff + t) : nullptr;
                const uint32_t bits = tile_row_of<K>(g.tiles, t, r);
                if (wt && bits) wt += ones_before<K>(g.tiles, t, r);
                relax_row(I, bits, d, wt);
            }
            ti += dt;
            ri += dr;
            if (ri >= na) {
                ri -= na;
                ++ti;
            }
        }
        return;
    }
    du[sub] = mine_du;
    __syncwarp(group);
    // 2^lg lanes a tile, no more than it has active rows
    auto log_up = [](int v) { return 32 - __clz(v - 1); };
    const int lg = min(log_up(na), 31 - __clz(width) - log_up(min(nt, width)));
    uint32_t mine_rows = amask;
    if (lg > 0) {
        mine_rows = 0u;
        for (int i = sub & ((1 << lg) - 1); i < na; i += 1 << lg) mine_rows |= 1u << nth_bit(amask, i);
    }
    for (int32_t t = t0 + (sub >> lg); t < t1; t += width >> lg) {
        const int32_t I = __ldg(g.colind + t);
        const float* wt = g.w ? g.w + __ldg(g.voff + t) : nullptr;
        if constexpr (K <= 8) {  // the tile is one word, a byte a row
            using W = typename std::conditional<K == 4, uint32_t, unsigned long long>::type;
            constexpr W ones = (W)0x0101010101010101ull;
            const W w = __ldg(reinterpret_cast<const W*>(g.tiles) + t);
            const W row_bytes = ((((mine_rows * ones) & (W)0x8040201008040201ull) + 0x7F * ones) >> 7) & ones;
            W bits = w & (row_bytes * (W)0xFF);
            while (bits) {
#pragma unroll
                for (int q = 0; q < kBatch; ++q) {
                    c[q] = -1;
                    if (bits) {
                        const W low = bits & (~bits + 1);
                        bits ^= low;
                        const int at = sizeof(W) == 4 ? __ffs((int)low) - 1 : __ffsll((long long)low) - 1;
                        const W below = w & (low - 1);
                        c[q] = at & 7;
                        cand[q] = du[at >> 3] +
                                  (wt ? __ldg(wt + (sizeof(W) == 4 ? __popc((uint32_t)below) : __popcll(below))) : 1.0f);
                    }
                }
                relax(I);
            }
        } else {
            for (uint32_t rows = mine_rows & rows_with_bits<K>(g.tiles, t); rows; rows &= rows - 1) {
                const int row = __ffs(rows) - 1;
                relax_row(I, tile_row_of<K>(g.tiles, t, row), du[row],
                          wt ? wt + ones_before<K>(g.tiles, t, row) : nullptr);
            }
        }
    }
}

// Resident blocks an SM, which are all that are launched: a round of many rows is
// bound by the loads in flight, and one of few costs no more for the blocks that
// leave at once.  Random graph of 2^20 vertices, us a search with 2 / 3 / 4 blocks:
// k = 4 3,308 / 2,374 / 1,914, k = 16 4,040 / 2,965 / 2,522; grid of 2048 x 2048,
// delta 400, k = 8 35,162 / 34,861 / 34,865, k = 32 44,525 / 44,534 / 46,648 (four
// blocks spill there).
template <int K>
constexpr int push_blocks() { return K <= 8 ? 4 : 3; }

// One round over the whole chip, a warp per active tile-row.  The roles of the
// sets follow from the previous round: its near list is this round's active
// set; when that is empty but far vertices wait, the threshold rises; when both
// are empty the loop is done.
template <int K>
__global__ void __launch_bounds__(kPushThreads, push_blocks<K>()) push_round_kernel(PushGraph g, PushSet s0, PushSet s1, PushSet s2,
                                                                  PushControl* ctl, int round, int buckets, float delta) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ PushState me;
    __shared__ int32_t ncur, block_min;
    __shared__ Appends<kPushBuffer> add_near, add_far;
    __shared__ float du[kPushThreads];
    if (threadIdx.x == 0) {
        PushState p = ctl->state[round & 1];
        const int32_t nn = ctl->near[(round + 3) & 3].v;
        const int32_t nf = ctl->far[p.epoch].v;
        const float fm = __int_as_float(ctl->farmin[p.epoch].v);
        int32_t len = 0;
        bool moved = false;
        if (p.active) {
            if (nn > 0) {
                len = nn;
                const int32_t t = p.cur;
                p.cur = p.nxt;
                p.nxt = t;
            } else if (buckets && nf > 0) {
                len = nf;
                moved = true;
                raise_threshold(p, fm, delta);
            }
            p.active = len > 0 ? 1 : 0;
            p.rounds += len > 0 ? 1 : 0;
            p.worked += (unsigned long long)len;
        }
        if (blockIdx.x == 0) {
            ctl->state[(round + 1) & 1] = p;
            ctl->near[(round + 1) & 3].v = 0;
            if (moved) {
                ctl->far[(p.epoch + 1) & 3].v = 0;
                ctl->farmin[(p.epoch + 1) & 3].v = __float_as_int(INFINITY);
            }
        }
        me = p;
        ncur = len;
        block_min = __float_as_int(INFINITY);
        add_near.n = add_far.n = 0;
    }
    __syncthreads();
    if ((int64_t)blockIdx.x * kPushWarps >= ncur) return;
    const PushSet cur = me.cur == 0 ? s0 : (me.cur == 1 ? s1 : s2);
    const PushSet nxt = me.nxt == 0 ? s0 : (me.nxt == 1 ? s1 : s2);
    const PushSet far = me.far == 0 ? s0 : (me.far == 1 ? s1 : s2);
    int32_t* near_count = &ctl->near[round & 3].v;
    int32_t* far_count = &ctl->far[me.epoch].v;
    const float th = me.theta;
    const int lane = (int)lane_id();
    const int64_t warps = (int64_t)gridDim.x * kPushWarps;
    float far_seen = INFINITY;
    for (int64_t e = (int64_t)blockIdx.x * kPushWarps + (threadIdx.x >> 5); e < ncur; e += warps)
        push_row<K>(g, cur, nxt, far, near_count, far_count, add_near, add_far, th, buckets, cur.list[e], 32, FULL, lane,
                    du + (threadIdx.x & ~31), far_seen);
    if (far_seen < INFINITY) atomicMin(&block_min, __float_as_int(far_seen));
    __syncthreads();
    const int m_near = min(add_near.n, kPushBuffer), m_far = min(add_far.n, kPushBuffer);
    if (threadIdx.x == 0 && m_near > 0) add_near.base = atomicAdd(near_count, m_near);
    if (threadIdx.x == 32 && m_far > 0) add_far.base = atomicAdd(far_count, m_far);
    if (threadIdx.x == 64 && block_min < __float_as_int(INFINITY)) atomicMin(&ctl->farmin[me.epoch].v, block_min);
    __syncthreads();
    for (int i = threadIdx.x; i < m_near; i += kPushThreads) nxt.list[add_near.base + i] = add_near.row[i];
    for (int i = threadIdx.x; i < m_far; i += kPushThreads) far.list[add_far.base + i] = add_far.row[i];
}

// ---------------------------------------------------------------------------
// rounds with few active tile-rows, many to a launch
// ---------------------------------------------------------------------------
// A launched round takes 6 to 7 us however few rows it has: the launch, the
// state and the lists' way through device memory on top of the relaxations' own
// chain.  Here one thread-block cluster runs up to kClusterRounds rounds with a
// cluster barrier between them.  A block keeps the tile-rows it marks in shared
// memory; the next round's work is dealt over all blocks by the prefix of their
// counts, and a row is read from the block that holds it through distributed
// shared memory.  Far marks are buffered until the near lists run dry.  A row
// gets 8 to 32 lanes, by how many rows there are.  Weighted grids, us a round
// launched / here: 31 rows a round 5.9 / 4.3, 107 rows 6.6 / 4.4, 400 rows 5.8 /
// 5.5, 770 rows 6.4 / 7.3.  So a search starts here and, once a few hundred
// rounds averaged more than 25 rows a block, launches the others: the rows of a
// round go up and down with every bucket, and changing to and fro cost more
// (115 ms against 88 on a 4096 x 4096 grid) than either.
//
// To the launched rounds the kernel is one round: it reads and leaves the same
// state and lists, and it leaves a round with more than `most` rows (or one
// whose marks did not fit) to them unrun.  Every decision is made from counts
// that no block changes before the next barrier, so all blocks take it alike.
constexpr int kClusterThreads = 1024;
constexpr int kClusterWarps = kClusterThreads / 32;
constexpr int kMaxCluster = 16;
constexpr int kClusterRounds = 128;
constexpr int kNearBuffer = 2048;
constexpr int kFarBuffer = 2048;
constexpr int kClusterAverage = 25;  // rows a block and round
constexpr int kMeshTiles = 5;        // tiles a row of the grids that both limits were measured on
constexpr int64_t kFewTiles = 128 * 1024;

struct ClusterShared {
    PushState me;
    int32_t from[kMaxCluster + 1];  // first index of each block's rows in the round's order
    int32_t len;                    // rows of the round
    int32_t listed;                 // they are in the set's list in device memory
    int32_t stop;
    int32_t block_min;
    float du[kClusterThreads];  // distances of the rows at work
    Appends<kNearBuffer> near[2];  // by the parity of the round that marks
    Appends<kFarBuffer> far;
};

static cudaLaunchConfig_t cluster_config(int blocks, cudaLaunchAttribute* at, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = sizeof(ClusterShared);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <int K>
__global__ void __launch_bounds__(kClusterThreads) push_cluster_kernel(PushGraph g, PushSet s0, PushSet s1, PushSet s2,
                                                                       PushControl* ctl, int slot, int buckets,
                                                                       float delta, int32_t most, int64_t max_rounds) {
    extern __shared__ __align__(16) unsigned char raw[];
    ClusterShared& sh = *reinterpret_cast<ClusterShared*>(raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int blocks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
    int32_t* near_count = &ctl->near[slot & 3].v;
    auto set = [&](int i) { return i == 0 ? s0 : (i == 1 ? s1 : s2); };
    // the buffered far marks go to the far set's list; called by all threads
    auto flush_far = [&]() {
        __syncthreads();
        const int m = min(sh.far.n, kFarBuffer);
        if (threadIdx.x == 0) {
            if (m > 0) sh.far.base = atomicAdd(&ctl->far[sh.me.epoch].v, m);
            if (sh.block_min < __float_as_int(INFINITY)) atomicMin(&ctl->farmin[sh.me.epoch].v, sh.block_min);
        }
        __syncthreads();
        const PushSet far = set(sh.me.far);
        for (int i = threadIdx.x; i < m; i += kClusterThreads) far.list[sh.far.base + i] = sh.far.row[i];
        __syncthreads();
        if (threadIdx.x == 0) {
            sh.far.n = 0;
            sh.block_min = __float_as_int(INFINITY);
        }
    };
    const int32_t given = __ldcg(&ctl->near[(slot + 3) & 3].v);  // rows that the round before left
    if (threadIdx.x == 0) {
        sh.me = ctl->state[slot & 1];
        sh.near[0].n = sh.near[1].n = sh.far.n = 0;
        sh.block_min = __float_as_int(INFINITY);
        sh.listed = 1;
        sh.len = given;
        sh.stop = sh.me.active ? 0 : 1;
    }
    cluster.sync();  // every block has read the state
    int done = 0;
    for (;; ++done) {
        const int q = done & 1;  // near[q] holds the rows that the last round marked
        if (done > 0 && warp == 0) {
            const int32_t n = lane < blocks ? cluster.map_shared_rank(&sh, lane)->near[q].n : 0;
            int32_t end = n;
#pragma unroll
            for (int d = 1; d < kMaxCluster; d <<= 1) {
                const int32_t o = __shfl_up_sync(0xffffffffu, end, d);
                if (lane >= d) end += o;
            }
            const bool full = __any_sync(0xffffffffu, n > kNearBuffer);
            if (lane < blocks) sh.from[lane + 1] = end;
            if (lane == blocks - 1) {
                sh.from[0] = 0;
                sh.len = end;
                sh.listed = 0;
                sh.stop = full ? 1 : 0;
            }
            if (lane == 0) sh.near[q ^ 1].n = 0;
        }
        __syncthreads();
        if (sh.stop) break;
        if (sh.len == 0) {  // near is dry
            flush_far();
            cluster.sync();
            const int32_t nf = buckets ? __ldcg(&ctl->far[sh.me.epoch].v) : 0;
            const float fm = __int_as_float(__ldcg(&ctl->farmin[sh.me.epoch].v));
            __syncthreads();
            if (nf > most || (nf > 0 && (done >= kClusterRounds || sh.me.rounds >= max_rounds))) {
                if (threadIdx.x == 0) sh.len = nf;
                break;
            }
            if (threadIdx.x == 0) {
                sh.len = nf;
                sh.listed = 1;
                if (nf > 0) {
                    raise_threshold(sh.me, fm, delta);
                    if (rank == 0) {
                        ctl->far[(sh.me.epoch + 1) & 3].v = 0;
                        ctl->farmin[(sh.me.epoch + 1) & 3].v = __float_as_int(INFINITY);
                    }
                } else {
                    sh.me.active = 0;
                }
            }
            __syncthreads();
            if (nf == 0) break;
        } else {
            if (sh.len > most || done >= kClusterRounds || sh.me.rounds >= max_rounds) break;
            if (sh.far.n > kFarBuffer / 2) flush_far();
            __syncthreads();
            if (threadIdx.x == 0) {
                const int32_t t = sh.me.cur;
                sh.me.cur = sh.me.nxt;
                sh.me.nxt = t;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            sh.me.rounds += 1;
            sh.me.worked += (unsigned long long)sh.len;
        }
        const PushSet cur = set(sh.me.cur), nxt = set(sh.me.nxt), far = set(sh.me.far);
        const int32_t len = sh.len;
        const int all = blocks * kClusterWarps;
        const int width = K == 32 || len <= all ? 32 : (K == 16 || len <= 2 * all ? 16 : 8);
        const int sub = lane & (width - 1);
        const unsigned group = (width == 32 ? 0xffffffffu : ((1u << width) - 1u)) << (lane - sub);
        float far_seen = INFINITY;
        // neighbouring rows go to different blocks
        for (int32_t e = (lane / width) * all + warp * blocks + rank; e < len; e += all * (32 / width)) {
            int32_t J;
            if (sh.listed) {
                J = __ldcg(cur.list + e);
            } else {
                int b = 0;
                for (int step = kMaxCluster / 2; step; step >>= 1)
                    if (b + step < blocks && sh.from[b + step] <= e) b += step;
                J = cluster.map_shared_rank(&sh, b)->near[q].row[e - sh.from[b]];
            }
            push_row<K>(g, cur, nxt, far, near_count, &ctl->far[sh.me.epoch].v, sh.near[q ^ 1], sh.far, sh.me.theta,
                        buckets, J, width, group, sub, sh.du + threadIdx.x - sub, far_seen);
        }
        if (far_seen < INFINITY) atomicMin(&sh.block_min, __float_as_int(far_seen));
        cluster.sync();  // all marks are made
    }
    // what is left goes to the lists in device memory
    flush_far();
    const int q = done & 1;
    if (done > 0) {
        const int m = min(sh.near[q].n, kNearBuffer);
        if (threadIdx.x == 0 && m > 0) sh.near[q].base = atomicAdd(near_count, m);
        __syncthreads();
        const PushSet nxt = set(sh.me.nxt);
        for (int i = threadIdx.x; i < m; i += kClusterThreads) nxt.list[sh.near[q].base + i] = sh.near[q].row[i];
    }
    if (rank == 0 && threadIdx.x == 0) {
        sh.me.busy = sh.me.active && sh.len > most ? 1 : 0;
        ctl->state[(slot + 1) & 1] = sh.me;
        ctl->near[(slot + 1) & 3].v = 0;
        if (done == 0) *near_count = given;
    }
    cluster.sync();  // no block reads this one's counts any more
}

// Distances, and the loop state before round 0: the source in set 0 as the
// list that the round before would have built.
__global__ void push_init_kernel(float* dist, int32_t n, int32_t src, int k, PushSet s0, PushControl* ctl, float theta) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dist[i] = (i == src) ? 0.0f : INFINITY;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        s0.act[src >> 5] = 1u << (src & 31);
        s0.list[0] = src / k;
        PushState z = {};
        z.cur = 1;
        z.far = 2;
        z.active = 1;
        z.theta = theta;
        ctl->state[0] = z;
        for (int i = 0; i < 4; ++i) {
            ctl->near[i].v = i == 3 ? 1 : 0;
            ctl->far[i].v = 0;
            ctl->farmin[i].v = __float_as_int(INFINITY);
        }
    }
}

thread_local int64_t g_last_push_rounds = 0;
thread_local int64_t g_last_push_rows = 0;

// Blocks of the largest cluster the device runs (0: none); looked up once per
// device.
template <int K>
static int push_cluster_blocks(int device) {
    static std::atomic<int> known[64];  // blocks + 1
    if (device < 0 || device >= 64) return 0;
    int got = known[device].load(std::memory_order_acquire);
    if (got) return got - 1;
    int blocks = 0;
    if (cudaFuncSetAttribute(push_cluster_kernel<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(push_cluster_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(ClusterShared)) == cudaSuccess) {
        for (int want = kMaxCluster; want >= 8 && !blocks; want /= 2) {
            cudaLaunchAttribute at[1];
            const cudaLaunchConfig_t cfg = cluster_config(want, at, nullptr);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, push_cluster_kernel<K>, &cfg) == cudaSuccess && n > 0) blocks = want;
        }
    }
    cudaGetLastError();  // a device without room for the cluster launches every round
    known[device].store(blocks + 1, std::memory_order_release);
    return blocks;
}

b2sr_status sssp_push(b2sr_matrix* hT, const float* w, int32_t src, float* dist, float delta, int max_iters,
                      cudaStream_t s) {
    g_last_push_rounds = 0;
    g_last_push_rows = 0;
    const int32_t n = hT->n;
    const int32_t ntr = hT->ntr;
    if (w) B2SR_TRY(ensure_voff(hT, s));  // before capture: capture must not allocate for the handle
    const size_t bw = round_up((size_t)ceil_div(n, 32) * 4, 256);
    const size_t lw = round_up((size_t)ntr * 4, 256);
    DevBuf buf(s);
    B2SR_TRY(buf.alloc(3 * (bw + lw) + sizeof(PushControl)));
    char* base = buf.as<char>();
    PushSet set[3];
    for (int i = 0; i < 3; ++i)
        set[i] = PushSet{reinterpret_cast<uint32_t*>(base + i * bw), reinterpret_cast<int32_t*>(base + 3 * bw + i * lw)};
    PushControl* ctl = reinterpret_cast<PushControl*>(base + 3 * (bw + lw));
    const int buckets = delta > 0.0f ? 1 : 0;
    B2SR_CUDA_TRY(cudaMemsetAsync(base, 0, 3 * bw, s));
    push_init_kernel<<<grid_for(n), 256, 0, s>>>(dist, n, src, hT->k, set[0], ctl, buckets ? delta : INFINITY);
    B2SR_LAUNCH_CHECK("push_init_kernel");
    // default round limit: without buckets at most n rounds improve anything;
    // with them every raise of the threshold settles at least one vertex and
    // costs a few rounds beyond the improving ones, so 4n covers both
    const int64_t cap = max_iters > 0 ? max_iters : (buckets ? 4 * (int64_t)n + 4 : (int64_t)n + 1);
    constexpr int kBatch = 32;  // launched rounds between two looks at the state
    const int64_t limit = ceil_div(cap + 1, kBatch) * kBatch;  // rounds with work: whole batches
    const PushGraph g{hT->rowptr, hT->colind, hT->tiles, w ? hT->voff : nullptr, w, dist, n,
                      hT->nnz >= kPairEntries * hT->T};
    PushState now = {};
    auto look = [&]() -> b2sr_status {
        B2SR_CUDA_TRY(cudaMemcpyAsync(&now, &ctl->state[0], sizeof(now), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        return B2SR_OK;
    };
    B2SR_TRY(with_tile(hT->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        int dev = -1;
        const int blocks = cudaGetDevice(&dev) == cudaSuccess ? push_cluster_blocks<K>(dev) : 0;
        // both limits are in tile-rows of kMeshTiles tiles: a round's work is in its
        // tiles, unless the graph has too few to matter
        const double scale = hT->T <= kFewTiles ? 1.0 : std::max(1.0, (double)hT->T / ((double)kMeshTiles * ntr));
        // rows it serves in two turns
        const int32_t most = (int32_t)(blocks * kClusterWarps * (K <= 8 ? 4 : 32 / K) * 2 / scale);
        const double average = blocks * kClusterAverage / scale;
        now.active = 1;
        for (bool few = blocks > 0; few && now.active;) {
            const int64_t rounds = now.rounds, worked = (int64_t)now.worked;
            cudaLaunchAttribute at[1];
            const cudaLaunchConfig_t cfg = cluster_config(blocks, at, s);
            for (int slot = 0; slot < 4; ++slot) {  // four: the near counters go round once
                B2SR_CUDA_TRY(cudaLaunchKernelEx(&cfg, push_cluster_kernel<K>, g, set[0], set[1], set[2], ctl, slot,
                                                 buckets, delta, most, limit));
                B2SR_LAUNCH_CHECK("push_cluster_kernel");
            }
            B2SR_TRY(look());
            if (now.active && now.rounds >= limit) return fail(B2SR_ERR_NOT_CONVERGED, "exceeded max_iters rounds");
            few = !now.busy && (double)((int64_t)now.worked - worked) <= (double)(now.rounds - rounds) * average;
        }
        if (!now.active) return B2SR_OK;
        const int grid = sm_count() * push_blocks<K>();  // warps stride over the active list
        int64_t replayed = 0;
        B2SR_TRY(run_captured(s, kBatch, limit + 1 - now.rounds, &ctl->state[0].active,
                              [&](cudaStream_t cs, int r) -> b2sr_status {
                                  push_round_kernel<K><<<grid, kPushThreads, 0, cs>>>(g, set[0], set[1], set[2], ctl, r,
                                                                                     buckets, delta);
                                  B2SR_LAUNCH_CHECK("push_round_kernel");
                                  return B2SR_OK;
                              },
                              &replayed));
        B2SR_TRY(look());
        return now.rounds > limit ? fail(B2SR_ERR_NOT_CONVERGED, "exceeded max_iters rounds") : B2SR_OK;
    }));
    g_last_push_rounds = now.rounds;
    g_last_push_rows = (int64_t)now.worked;
    return B2SR_OK;
}

}  // namespace b2sr

using namespace b2sr;

extern "C" b2sr_status b2sr_sssp_push(b2sr_handle hT, const float* weights_t, int32_t src, float* dist, float delta,
                                      int max_iters, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(hT));
    if (src < 0 || src >= hT->n) return fail(B2SR_ERR_INVALID_ARG, "source out of range");
    if (!dist) return fail(B2SR_ERR_INVALID_ARG, "dist is NULL");
    if (!(delta == delta)) return fail(B2SR_ERR_INVALID_ARG, "delta is NaN");
    return sssp_push(hT, weights_t, src, dist, delta, max_iters, to_stream(stream));
}

extern "C" b2sr_status b2sr_sssp_push_rounds(int64_t* rounds, int64_t* active_tile_rows) {
    clear_error();
    if (!rounds) return fail(B2SR_ERR_INVALID_ARG, "rounds is NULL");
    *rounds = g_last_push_rounds;
    if (active_tile_rows) *active_tile_rows = g_last_push_rows;
    return B2SR_OK;
}
