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
// One round: a warp per active tile-row J deals its (tile, active source row)
// pairs to the lanes; for every set bit (r, c) of a pair's tile (J, I) the
// target kI+c is relaxed with dist[kJ+r] + w by an integer atomicMin on the
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
#include <algorithm>
#include <type_traits>

#include "b2sr_internal.cuh"
#include "captured.cuh"

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
    int32_t pad;
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

// Row r of tile t, and the set bits of its earlier rows (the row's first
// weight is that far from the tile's).
template <int K>
__device__ __forceinline__ uint32_t pushed_row(const uint8_t* __restrict__ tiles, int32_t t, int r, bool weighted,
                                               int* before) {
    if constexpr (K == 4) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(tiles) + t);
        *before = __popc(w & ((1u << (8 * r)) - 1u));
        return (w >> (8 * r)) & 0xFu;
    } else if constexpr (K == 8) {
        const unsigned long long w = __ldg(reinterpret_cast<const unsigned long long*>(tiles) + t);
        *before = __popcll(w & ((1ull << (8 * r)) - 1ull));
        return (uint32_t)(w >> (8 * r)) & 0xFFu;
    } else if constexpr (K == 16) {
        const uint16_t* p = reinterpret_cast<const uint16_t*>(tiles) + (int64_t)t * 16;
        *before = 0;
        if (weighted)
            for (int q = 0; q < r; ++q) *before += __popc((uint32_t)__ldg(p + q));
        return __ldg(p + r);
    } else {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(tiles) + (int64_t)t * 32;
        *before = 0;
        if (weighted)
            for (int q = 0; q < r; ++q) *before += __popc(__ldg(p + q));
        return __ldg(p + r);
    }
}

// The tile-rows a block appends to one list: kept in shared memory, appended
// at the block's end with one global atomic (directly once the buffer is full).
constexpr int kPushBuffer = 512;
struct Appends {
    int32_t n, base;
    int32_t row[kPushBuffer];
};

template <int K>
__device__ __forceinline__ void mark_bits(const PushSet& s, int32_t* count, Appends& ap, int32_t J, uint32_t bits) {
    constexpr int per = 32 / K;
    constexpr uint32_t seg = K == 32 ? 0xFFFFFFFFu : (1u << (K & 31)) - 1u;
    const int sh = (J % per) * K;
    const uint32_t old = atomicOr(s.act + J / per, bits << sh);
    if (((old >> sh) & seg) != 0u) return;  // listed by whoever set the tile-row's first bit
    const int32_t at = atomicAdd(&ap.n, 1);
    if (at < kPushBuffer) ap.row[at] = J;
    else s.list[atomicAdd(count, 1)] = J;
}

// One round.  It is a chain of dependent memory accesses (state, list, segment
// and row pointers, tiles, weights, two atomics, list length), so the lanes
// take one (tile, source row) pair each and issue up to kBatch relaxations
// side by side; a lane that walked all rows of a tile paid the chain once per
// active row and bit.  The roles of the sets follow from the previous round:
// its near list is this round's active set; when that is empty but far
// vertices wait, the threshold rises by delta -- or, past a gap in the
// distances, to the least far distance plus delta, so that the nearest waiting
// vertex always gets in -- and the whole far set is this round's active set
// (whatever is still past the threshold moves back); when both are empty the
// loop is done.
template <int K>
__global__ void __launch_bounds__(kPushThreads) push_round_kernel(const int32_t* __restrict__ rowptr,
                                                                  const int32_t* __restrict__ colind,
                                                                  const uint8_t* __restrict__ tiles,
                                                                  const int32_t* __restrict__ voff,
                                                                  const float* __restrict__ w, PushSet s0, PushSet s1,
                                                                  PushSet s2, PushControl* ctl, int round, float* dist,
                                                                  int buckets, float delta) {
    constexpr int per = 32 / K;
    constexpr uint32_t seg = K == 32 ? 0xFFFFFFFFu : (1u << (K & 31)) - 1u;
    constexpr int kBatch = 4;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ PushState me;
    __shared__ int32_t ncur, block_min;
    __shared__ Appends add_near, add_far;
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
    float fmin_seen = INFINITY;  // least distance this lane sent to the far set
    for (int64_t e = (int64_t)blockIdx.x * kPushWarps + (threadIdx.x >> 5); e < ncur; e += warps) {
        const int32_t J = cur.list[e];
        const int sh = (J % per) * K;
        uint32_t amask = (cur.act[J / per] >> sh) & seg;
        const int32_t t0 = __ldg(rowptr + J), t1 = __ldg(rowptr + J + 1);
        float du = 0.0f;  // the sources' distances (the bitset has no bits past n)
        if (lane < K && ((amask >> lane) & 1u)) du = dist[(int64_t)J * K + lane];
        __syncwarp();  // every lane has read the segment
        if (lane == 0) atomicAnd(cur.act + J / per, ~(seg << sh));
        if (buckets) {
            // active vertices at or past the threshold move to the far set
            const bool late = lane < K && ((amask >> lane) & 1u) && du >= th;
            const uint32_t defer = __ballot_sync(FULL, late);
            if (late) fmin_seen = fminf(fmin_seen, du);
            if (defer && lane == 0) mark_bits<K>(far, far_count, add_far, J, defer);
            amask &= ~defer;
        }
        const int na = __popc(amask);
        if (na == 0) continue;
        const int64_t pairs = (int64_t)(t1 - t0) * na;
        int32_t ti = lane / na;
        int ri = lane - ti * na;
        const int32_t dt = 32 / na;
        const int dr = 32 - dt * na;
        for (int64_t p = 0; p < pairs; p += 32) {
            const bool live = p + lane < pairs;
            const int r = live ? nth_bit(amask, ri) : 0;
            const float d = __shfl_sync(FULL, du, r);
            if (live) {
                const int32_t t = t0 + ti;
                int before = 0;
                uint32_t bits = pushed_row<K>(tiles, t, r, w != nullptr, &before);
                const int32_t I = __ldg(colind + t);
                const float* wt = w ? w + __ldg(voff + t) + before : nullptr;
                while (bits) {
                    int c[kBatch];
                    float cand[kBatch];
                    int old[kBatch];
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
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (c[q] >= 0)
                            old[q] = atomicMin(reinterpret_cast<int*>(dist) + (int64_t)I * K + c[q],
                                               __float_as_int(cand[q]));
                    uint32_t near_bits = 0u, far_bits = 0u;
#pragma unroll
                    for (int q = 0; q < kBatch; ++q)
                        if (c[q] >= 0 && cand[q] < __int_as_float(old[q])) {
                            if (cand[q] >= th) {
                                fmin_seen = fminf(fmin_seen, cand[q]);
                                far_bits |= 1u << c[q];
                            } else {
                                near_bits |= 1u << c[q];
                            }
                        }
                    if (near_bits) mark_bits<K>(nxt, near_count, add_near, I, near_bits);
                    if (far_bits) mark_bits<K>(far, far_count, add_far, I, far_bits);
                }
            }
            ti += dt;
            ri += dr;
            if (ri >= na) {
                ri -= na;
                ++ti;
            }
        }
    }
    if (fmin_seen < INFINITY) atomicMin(&block_min, __float_as_int(fmin_seen));
    __syncthreads();
    const int m_near = min(add_near.n, kPushBuffer), m_far = min(add_far.n, kPushBuffer);
    if (threadIdx.x == 0 && m_near > 0) add_near.base = atomicAdd(near_count, m_near);
    if (threadIdx.x == 32 && m_far > 0) add_far.base = atomicAdd(far_count, m_far);
    if (threadIdx.x == 64 && block_min < __float_as_int(INFINITY)) atomicMin(&ctl->farmin[me.epoch].v, block_min);
    __syncthreads();
    for (int i = threadIdx.x; i < m_near; i += kPushThreads) nxt.list[add_near.base + i] = add_near.row[i];
    for (int i = threadIdx.x; i < m_far; i += kPushThreads) far.list[add_far.base + i] = add_far.row[i];
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
    const int grid = sm_count() * 2;  // warps stride over the active list
    // default round limit: without buckets at most n rounds improve anything;
    // with them every raise of the threshold settles at least one vertex and
    // costs a few rounds beyond the improving ones, so 4n covers both
    const int64_t cap = max_iters > 0 ? max_iters : (buckets ? 4 * (int64_t)n + 4 : (int64_t)n + 1);
    int64_t replayed = 0;
    const int32_t* voff = w ? hT->voff : nullptr;
    B2SR_TRY(with_tile(hT->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        return run_captured(s, 32, cap + 1, &ctl->state[0].active,
                            [&](cudaStream_t cs, int r) -> b2sr_status {
                                push_round_kernel<K><<<grid, kPushThreads, 0, cs>>>(hT->rowptr, hT->colind, hT->tiles,
                                                                                   voff, w, set[0], set[1], set[2], ctl,
                                                                                   r, dist, buckets, delta);
                                B2SR_LAUNCH_CHECK("push_round_kernel");
                                return B2SR_OK;
                            },
                            &replayed);
    }));
    PushState end;
    B2SR_CUDA_TRY(cudaMemcpyAsync(&end, &ctl->state[0], sizeof(end), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    g_last_push_rounds = end.rounds;
    g_last_push_rows = (int64_t)end.worked;
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
