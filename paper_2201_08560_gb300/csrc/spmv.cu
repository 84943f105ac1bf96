// B2SR SpMV: the BMV schemes of Table 2 over the semirings of Table 4, and the
// 64-lane Boolean SpMM used by multi-source BFS.
//
// Design (GB300).  The paper maps one tile-row to one warp (Listing 1) or 32
// tile-rows to a 1024-thread block (Sec. IV, bmv_bin_full_full).  Power-law
// graphs make any row mapping badly imbalanced (a scale-20 R-MAT tile-row can
// hold 10^5 tiles), so the unit of work here is a fixed-size chunk of
// consecutive tiles:
//   * one warp per chunk of 32*P tiles, and four kernels that walk it: the
//     small-tile one (bits at k = 4 and 8, unweighted values at k = 4; a lane a
//     run of tiles, whole input segments), the row-lane one (values at k = 16 and
//     32, the 64-lane OR at k = 8; a lane a row of the tile), the staged one
//     (values at k <= 16 under that schedule; one cp.async gather per set bit
//     into shared memory) and the general one (the rest; registers hold a lane's
//     k row results);
//   * every load a lane needs is issued up front, so each warp keeps several KB
//     in flight;
//   * rows that cross lanes are joined by shuffles in a fixed order; rows that
//     cross chunks leave per-chunk partials that a second kernel joins, one warp
//     per row, in a fixed order (Boolean rows at k = 4 and 8 are ORed into the
//     cleared output instead).
// Every reduction order is fixed by the data, so floating-point results are
// bitwise reproducible and independent of launch geometry and stream.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "b2sr_internal.cuh"
#include "tile_bits.cuh"

namespace b2sr {

// ---------------------------------------------------------------------------
// tile words.  A lane holds its P tiles as 32-bit words: TW words per tile
// (k=4: 1, k=8: 2, k=16: 8, k=32: 32); row r of a tile is byte r (k<=8),
// half-word r (k=16) or word r (k=32).
// ---------------------------------------------------------------------------
template <int K>
struct ChunkShape {
    static constexpr int P = tiles_per_lane(K);
    static constexpr int CT = 32 * P;
    static constexpr int TB = K * (K <= 8 ? 1 : (K == 16 ? 2 : 4));
    static constexpr int TW = TB / 4;
    static constexpr int TILE_V4 = P * TB / 16;  // uint4 loads per lane for its tiles
    static constexpr int ROW_BITS = K <= 8 ? 8 : K;  // bits per row slot in a word
};

// Bit r of the result is set iff row r of the tile shares a bit with xs (the
// k-bit segment of the input vector under the tile's column).
template <int K>
__device__ __forceinline__ uint32_t rows_hit(const uint32_t* w, uint32_t xs) {
    if (K == 4 || K == 8) {
        // four rows per word, one per byte: flag the non-zero bytes (high bit
        // per byte), then gather the four flags with one multiply
        const uint32_t rep = xs * 0x01010101u;
        uint32_t out = 0;
#pragma unroll
        for (int q = 0; q < K / 4; ++q) {
            uint32_t m = w[q] & rep;
            uint32_t h = (((m & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | m) & 0x80808080u;
            out |= (((h >> 7) * 0x00204081u) >> 21 & 0xFu) << (4 * q);
        }
        return out;
    } else if (K == 16) {
        const uint32_t rep = xs | (xs << 16);
        uint32_t out = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint32_t m = w[q] & rep;
            out |= ((m & 0xFFFFu) ? 1u : 0u) << (2 * q);
            out |= ((m >> 16) ? 1u : 0u) << (2 * q + 1);
        }
        return out;
    } else {
        uint32_t out = 0;
#pragma unroll
        for (int r = 0; r < 32; ++r) out |= ((w[r] & xs) ? 1u : 0u) << r;
        return out;
    }
}

__device__ __forceinline__ bool mask_allows(const uint32_t* __restrict__ mask, int comp, int64_t v) {
    if (!mask) return true;
    bool b = (__ldg(mask + (v >> 5)) >> (v & 31)) & 1u;
    return comp ? !b : b;
}

// Every output row in [r0, r1) is excluded by a bitset mask (bits all 0, or
// all 1 for a complemented mask): the masked store writes the semiring's
// identity there whatever the tiles hold.  Rows past n store nothing; spans
// of more than 2048 rows are not tested (false).
// Warp-collective.  Semirings whose masked calls sit on a level loop (BFS,
// MIS, colouring) use it; in the others the test's registers cost more
// occupancy than the skip saves, and saturated() is constant false.
__device__ __forceinline__ bool rows_masked_out(const uint32_t* __restrict__ mask, int comp, int32_t n, int64_t r0,
                                                int64_t r1) {
    if (!mask || r1 - r0 > 2048) return false;  // at most two mask words a lane
    r1 = min(r1, (int64_t)n);
    bool ok = true;
    for (int64_t w = (r0 >> 5) + lane_id(); w * 32 < r1; w += 32) {
        const int64_t lo = max(r0, w * 32), hi = min(r1, w * 32 + 32);
        const uint32_t need = (hi - lo >= 32) ? 0xFFFFFFFFu : (((1u << (hi - lo)) - 1u) << (lo - w * 32));
        const uint32_t m = comp ? __ldg(mask + w) : ~__ldg(mask + w);
        ok &= (m & need) == need;
    }
    return __all_sync(0xffffffffu, ok);
}

// ---------------------------------------------------------------------------
// accumulator storage: registers (static row index) or shared memory (one
// column per lane, any row index)
// ---------------------------------------------------------------------------
template <class V, int NV>
struct RegAcc {
    V a[NV];
    __device__ __forceinline__ V get(int v) const { return a[v]; }
    __device__ __forceinline__ void set(int v, V x) { a[v] = x; }
};

template <class V, int NV>
struct SmemAcc {
    V* p;  // element v at p[v * 32]
    __device__ __forceinline__ V get(int v) const { return p[v * 32]; }
    __device__ __forceinline__ void set(int v, V x) { p[v * 32] = x; }
};

// ---------------------------------------------------------------------------
// warp shuffles of accumulator values (scalars, and the four-column blocks of
// SemPlus4 one component at a time)
// ---------------------------------------------------------------------------
// Join type of the plus-times partials of rows that cross chunks: a
// compensated fp32 sum.  Each addition is Knuth's TwoSum of the leading parts
// (the exact rounding error, whatever the magnitudes), added to the carried
// error terms; the rounding is spelled out so no contraction or reordering
// can change it.  fp32 keeps the join off the fp64 pipe, which is narrow on
// GB300; the compensation keeps it as accurate as an fp64 join for the few
// hundred partials a row can have.
struct CSum {
    float s, c;
    CSum() = default;
    __device__ __forceinline__ CSum(float a) : s(a), c(0.0f) {}
    // an infinite or NaN sum has no rounding error: its c is NaN
    __device__ __forceinline__ explicit operator float() const { return isfinite(s) ? __fadd_rn(s, c) : s; }
};

__device__ __forceinline__ CSum csum_add(CSum a, CSum b) {
    const float t = __fadd_rn(a.s, b.s);
    const float bp = __fsub_rn(t, a.s);
    const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(b.s, bp));
    CSum r;
    r.s = t;
    r.c = __fadd_rn(__fadd_rn(a.c, b.c), e);
    return r;
}

struct CSum4 {  // the same for a four-column block, column by column
    CSum v[4];
    CSum4() = default;
    __device__ __forceinline__ CSum4(float4 a) : v{CSum(a.x), CSum(a.y), CSum(a.z), CSum(a.w)} {}
    __device__ __forceinline__ explicit operator float4() const {
        return make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
    }
};

template <class T>
__device__ __forceinline__ T shfl_up(T v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }
template <class T>
__device__ __forceinline__ T shfl_xor(T v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float4 shfl_up(float4 v, int d) {
    return make_float4(shfl_up(v.x, d), shfl_up(v.y, d), shfl_up(v.z, d), shfl_up(v.w, d));
}
__device__ __forceinline__ float4 shfl_xor(float4 v, int o) {
    return make_float4(shfl_xor(v.x, o), shfl_xor(v.y, o), shfl_xor(v.z, o), shfl_xor(v.w, o));
}
__device__ __forceinline__ CSum shfl_xor(CSum a, int o) {
    CSum r;
    r.s = shfl_xor(a.s, o);
    r.c = shfl_xor(a.c, o);
    return r;
}
__device__ __forceinline__ CSum4 shfl_xor(CSum4 a, int o) {
    CSum4 r;
#pragma unroll
    for (int i = 0; i < 4; ++i) r.v[i] = shfl_xor(a.v[i], o);
    return r;
}

// ---------------------------------------------------------------------------
// semirings.  Each provides V (accumulator value), NV (values per tile-row
// accumulator), ident(), comb(a, b) (a earlier in the fixed order),
// store(R, acc) (self term, mask, overwrite; empty tile-rows are stored with
// the identity) and a join type J for the cross-chunk join.
//   bit-vector schemes (kGather = false): xseg(J) and tile(acc, words, xs);
//   value schemes (kGather = true): one gathered input per set bit, src(),
//     weighted, wts(), voffs() and apply(acc, x_j, w_ij).
// ---------------------------------------------------------------------------

// Row mask of OR-accumulated, input-masked tile words (k <= 8: a row per
// byte): bit r is set iff byte r is non-zero.  The non-zero bytes get their
// high bit, and one multiply gathers the four high bits of a word.
template <int K>
__device__ __forceinline__ uint32_t nonzero_rows(const uint32_t* w) {
    uint32_t out = 0;
#pragma unroll
    for (int q = 0; q < K / 4; ++q) {
        const uint32_t m = w[q];
        const uint32_t h = (((m & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | m) & 0x80808080u;
        out |= (((h >> 7) * 0x00204081u) >> 21 & 0xFu) << (4 * q);
    }
    return out;
}

// bmv_bin_bin_bin[_masked]: bitset in, bitset out.  For k <= 8 the
// accumulator is the OR of the tile words ANDed with the input segment (one
// word per four rows); OR commutes with "row is non-zero", so the row mask is
// formed only when a row is stored.  For k >= 16 it is the k-bit row mask.
// For k <= 8 every store ORs into a cleared output: a row that crosses chunks
// is stored by each, so there are no partials, no join and no rows to fill in
// (three launches, an allocation and a free before; the clear and one launch
// now).
template <int K>
struct SemBool {
    using V = uint32_t;
    using J = uint32_t;
    static constexpr int NV = K <= 8 ? K / 4 : 1;
    static constexpr bool kGather = false;
    static constexpr bool kOrsInto = K <= 8;
    const uint32_t* x;
    uint32_t* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ V ident() const { return 0u; }
    __device__ V comb(V a, V b) const { return a | b; }
    __device__ J jcomb(J a, J b) const { return a | b; }
    __device__ uint32_t xseg(int32_t Jc) const { return ld_bits(x, (int64_t)Jc * K, K); }
    __device__ bool saturated(int64_t r0, int64_t r1) const { return rows_masked_out(mask, comp, n, r0, r1); }
    template <class A>
    __device__ void tile(A& acc, const uint32_t* w, uint32_t xs) const {
        if constexpr (K <= 8) {
            const uint32_t rep = xs * 0x01010101u;
#pragma unroll
            for (int q = 0; q < NV; ++q) acc.set(q, acc.get(q) | (w[q] & rep));
        } else {
            acc.set(0, acc.get(0) | rows_hit<K>(w, xs));
        }
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
        uint32_t v;
        if constexpr (K <= 8) {
            uint32_t w[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) w[q] = acc.get(q);
            v = nonzero_rows<K>(w);
        } else {
            v = acc.get(0);
        }
        if (mask) {
            uint32_t mb = ld_bits(mask, (int64_t)R * K, K);
            v &= comp ? ~mb : mb;
        }
        if constexpr (kOrsInto) {
            if (v) atomicOr(y + (((int64_t)R * K) >> 5), v << ((R * K) & 31));
        } else if (K == 32) {
            y[R] = v;
        } else {
            reinterpret_cast<uint16_t*>(y)[R] = (uint16_t)v;
        }
    }
};

// bmv_bin_bin_full[_masked]: bitset in, int32 counts out (popc of Sec. IV)
template <int K>
struct SemCount {
    using V = int32_t;
    using J = int32_t;
    static constexpr int NV = K;
    static constexpr bool kGather = false;
    const uint32_t* x;
    int32_t* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ V ident() const { return 0; }
    __device__ V comb(V a, V b) const { return a + b; }
    __device__ J jcomb(J a, J b) const { return a + b; }
    __device__ uint32_t xseg(int32_t Jc) const { return ld_bits(x, (int64_t)Jc * K, K); }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    template <class A>
    __device__ void tile(A& acc, const uint32_t* w, uint32_t xs) const {
#pragma unroll
        for (int r = 0; r < K; ++r) acc.set(r, acc.get(r) + __popc(tile_row<K>(w, r) & xs));
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) {
            int64_t i = (int64_t)R * K + r;
            if (i < n) y[i] = mask_allows(mask, comp, i) ? acc.get(r) : 0;
        }
    }
};

// ones per row: the count of a vector of ones, which needs no input; the rows
// without tiles are zero beforehand
template <int K>
struct SemOnes : SemCount<K> {
    static constexpr bool kNoInput = true;
    __device__ uint32_t xseg(int32_t) const { return K == 32 ? 0xFFFFFFFFu : (1u << (K & 31)) - 1u; }
};

// bmv_bin_full_full over plus-times: float in, float out; partials of rows
// that cross chunks are joined with a compensated fp32 sum (CSum)
template <int K>
struct SemPlus {
    using V = float;
    using G = float;
    using J = CSum;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const float* x;
    float* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ const float* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return 0.0f; }
    __device__ V comb(V a, V b) const { return a + b; }
    __device__ J jcomb(J a, J b) const { return csum_add(a, b); }
    __device__ V apply(V acc, G xv, float) const { return acc + xv; }
    __device__ V contrib(G xv, float) const { return xv; }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : 0.0f;
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// plus-times over a block of four fp32 columns (vertex-major: x[v] holds the
// four columns' values of vertex v).  Every component is added in exactly the
// order SemPlus adds a single column, and joined the same way, so column b
// of the result is bitwise the SemPlus result for column b.
template <int K>
struct SemPlus4 {
    using V = float4;
    using G = float4;
    using J = CSum4;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const float4* x;
    float4* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ const float4* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
    __device__ V comb(V a, V b) const { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
    __device__ J jcomb(J a, J b) const {
        J r;
#pragma unroll
        for (int i = 0; i < 4; ++i) r.v[i] = csum_add(a.v[i], b.v[i]);
        return r;
    }
    __device__ V apply(V acc, G xv, float) const { return comb(acc, xv); }
    __device__ V contrib(G xv, float) const { return xv; }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : ident();
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// bmv_bin_full_full over min-plus (relaxation, Sec. V SSSP): float in/out;
// weights in set-bit order (voff[t] = set bits before tile t), or w = 1.  The
// chunk kernels store the minimum over the neighbours; the diagonal's self
// term min(x_i, .) is applied by spmv_self_kernel once the rows are joined
// (kept out of the chunk kernels, where its extra load per row cost registers
// and spills)
template <int K>
struct SemMinPlus {
    using V = float;
    using G = float;
    using J = float;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kSelfTerm = true;  // x_i joins y_i in spmv_self_kernel
    static constexpr bool kMayWeight = true;
    const float* x;
    float* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    const float* w;
    const int32_t* voff;
    bool weighted;
    __device__ const float* src() const { return x; }
    __device__ const float* wts() const { return w; }
    __device__ const int32_t* voffs() const { return voff; }
    __device__ V ident() const { return INFINITY; }
    __device__ V comb(V a, V b) const { return fminf(a, b); }
    __device__ J jcomb(J a, J b) const { return fminf(a, b); }
    __device__ V apply(V acc, G xv, float wv) const { return fminf(acc, xv + wv); }
    __device__ V contrib(G xv, float wv) const { return xv + wv; }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : INFINITY;
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// min over neighbours of int32 labels (min-plus with weight 0: the CC step);
// the self term x_i is applied after the join, as for SemMinPlus
template <int K>
struct SemMinI32 {
    using V = int32_t;
    using G = int32_t;
    using J = int32_t;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kSelfTerm = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const int32_t* x;
    int32_t* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ const int32_t* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return INT_MAX; }
    __device__ V comb(V a, V b) const { return min(a, b); }
    __device__ J jcomb(J a, J b) const { return min(a, b); }
    __device__ V apply(V acc, G xv, float) const { return min(acc, xv); }
    __device__ V contrib(G xv, float) const { return xv; }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : INT_MAX;
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// bmv_bin_full_full over tropical max-times (Table 4: the local-maximum step
// of MIS and colouring): y_i = max over neighbours j of x_j (A_ij = 1 is the
// multiplicative identity, so x_j passes unchanged); -inf where no neighbour
// or masked out.  max is exact, so the result does not depend on the order.
template <int K>
struct SemMaxF32 {
    using V = float;
    using G = float;
    using J = float;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const float* x;
    float* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ const float* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return -INFINITY; }
    __device__ V comb(V a, V b) const { return fmaxf(a, b); }
    __device__ J jcomb(J a, J b) const { return fmaxf(a, b); }
    __device__ V apply(V acc, G xv, float) const { return fmaxf(acc, xv); }
    __device__ V contrib(G xv, float) const { return xv; }
    __device__ bool saturated(int64_t, int64_t) const { return false; }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : -INFINITY;
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// max over neighbours of 64-bit keys (priority bits above the vertex id: the
// local-maximum test of MIS and colouring with ties broken by id); 0 is
// below every key and stands for "no undecided neighbour"
template <int K>
struct SemMaxKey {
    using V = unsigned long long;
    using G = unsigned long long;
    using J = unsigned long long;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const unsigned long long* x;
    unsigned long long* y;
    const uint32_t* mask;
    int comp;
    int32_t n;
    __device__ const unsigned long long* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return 0ull; }
    __device__ V comb(V a, V b) const { return a > b ? a : b; }
    __device__ J jcomb(J a, J b) const { return a > b ? a : b; }
    __device__ V apply(V acc, G xv, float) const { return acc > xv ? acc : xv; }
    __device__ V contrib(G xv, float) const { return xv; }
    __device__ bool saturated(int64_t r0, int64_t r1) const { return rows_masked_out(mask, comp, n, r0, r1); }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) y[i] = mask_allows(mask, comp, i) ? v : 0ull;
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// Boolean frontiers packed in one word per vertex (lane b of X_j: vertex j is
// in frontier b): Y_i = OR_j X_j, masked by M_i or ~M_i
template <int K, class W>
struct SemOrLanes {
    using V = W;
    using G = W;
    using J = W;
    static constexpr int NV = K;
    static constexpr bool kGather = true;
    static constexpr bool kMayWeight = false;
    static constexpr bool weighted = false;
    const W* x;
    W* y;
    const W* mask;
    int comp;
    int32_t n;
    // optional: bit J set where one of x[4J .. 4J+3] is not zero, and a flag
    // that says not to look (most are set)
    const uint32_t* live = nullptr;
    const int32_t* dense = nullptr;
    __device__ const W* src() const { return x; }
    __device__ const float* wts() const { return nullptr; }
    __device__ const int32_t* voffs() const { return nullptr; }
    __device__ V ident() const { return (W)0; }
    __device__ V comb(V a, V b) const { return a | b; }
    __device__ J jcomb(J a, J b) const { return a | b; }
    __device__ V apply(V acc, G xv, float) const { return acc | xv; }
    __device__ V contrib(G xv, float) const { return xv; }
    // Every output row in [r0, r1) is fully masked out (complemented mask of
    // all ones): zero whatever the tiles hold.  Warp-collective.
    __device__ bool saturated(int64_t r0, int64_t r1) const {
        if (!mask || !comp || r1 - r0 > 9 * K) return false;  // up to nine tile-rows
        r1 = min(r1, (int64_t)n);
        bool ok = true;
        for (int64_t i = r0 + lane_id(); i < r1; i += 32) ok &= __ldg(mask + i) == (W)~(W)0;
        return __all_sync(0xffffffffu, ok);
    }
    __device__ void store_row(int32_t R, int r, V v) const {
        int64_t i = (int64_t)R * K + r;
        if (i < n) {
            if (mask) v &= comp ? ~__ldg(mask + i) : __ldg(mask + i);
            y[i] = v;
        }
    }
    template <class A>
    __device__ void store(int32_t R, const A& acc) const {
#pragma unroll
        for (int r = 0; r < K; ++r) store_row(R, r, acc.get(r));
    }
};

// 64 and 32 lanes: the batched BFS packs up to 64 (or, for at most 32
// sources, 32) frontiers into one word per vertex.
template <int K>
using SemOr64 = SemOrLanes<K, unsigned long long>;
template <int K>
using SemOr32 = SemOrLanes<K, uint32_t>;

// schemes that read no input vector
template <class S, class = void>
struct NoInput : std::false_type {};
template <class S>
struct NoInput<S, std::void_t<decltype(S::kNoInput)>> : std::bool_constant<S::kNoInput> {};

// schemes whose stores OR into a cleared output
template <class S, class = void>
struct OrsInto : std::false_type {};
template <class S>
struct OrsInto<S, std::void_t<decltype(S::kOrsInto)>> : std::bool_constant<S::kOrsInto> {};

// ---------------------------------------------------------------------------
// kernel arguments and shared-memory layout
// ---------------------------------------------------------------------------
struct SpmvGeom {
    const int32_t* rowptr;
    const int32_t* colind;
    const uint8_t* tiles;
    const int32_t* chunk_row;
    int64_t T;
    int64_t nchunks;
    int32_t ntr;
    // optional device flag: when it reads 0 the launch does nothing (lets a
    // captured loop of SpMVs run past the point where its driver is done)
    const int32_t* gate;
};

__device__ __forceinline__ bool gated_off(const int32_t* gate) { return gate && *gate == 0; }

template <class V>
struct Partials {
    V* val_first;  // [nchunks * NV]: the chunk's first row, begun in an earlier chunk
    V* val_last;   // [nchunks * NV]: the chunk's last row, continued in a later chunk
};

template <int BYTES>
__device__ __forceinline__ void cp_async_gather(void* smem, const void* gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

constexpr int kSpmvThreads = 256;
constexpr int kSpmvWarps = kSpmvThreads / 32;
constexpr int64_t kMaxBlockSmem = 227 * 1024;  // dynamic shared memory a block can have

// Shared memory per warp for the gather schemes (k <= 16): the lanes' tile
// words and tile columns (lane-private, so the flat bit walk can index them),
// NG staged input values (+ NG weights for min-plus) and a one-byte
// (tile, row) tag per staged value.  A chunk with more than NG set bits reads
// its values straight from global memory instead.
template <int K, class SEM, bool GATHER = SEM::kGather>
struct GatherLayout {
    static constexpr int NG = 0;
    static constexpr int bytes = 0;
};
template <int K, class SEM>
struct GatherLayout<K, SEM, true> {
    using G = typename SEM::G;
    using S = ChunkShape<K>;
    // the same for every value type: whether a chunk is staged decides its
    // summation order, and the four-column block must sum like one column
    static constexpr int NG = 512;
    static constexpr int words_off = 0;                                    // [P*TW][32] u32
    static constexpr int col_off = words_off + S::CT * S::TW * 4;          // [P][32] i32
    static constexpr int x_off = col_off + S::CT * 4;                      // [NG] G
    static constexpr int w_off = x_off + NG * (int)sizeof(G);              // [NG] f32 (min-plus)
    static constexpr int tag_off = w_off + (SEM::kMayWeight ? NG * 4 : 0);  // [NG] u8
    static constexpr int pre_off = (tag_off + NG + 15) / 16 * 16;           // [P][32] i32: first slot of each tile
    static constexpr int bytes = pre_off + S::CT * 4;
    static_assert(x_off % 16 == 0 && bytes % 16 == 0, "16-byte staging slots");
};

// ---------------------------------------------------------------------------
// pieces shared by the chunk kernels
// ---------------------------------------------------------------------------
// Tile indices fit in int32 (T < 2^31: TileColInd and TileRowPtr are int32),
// which keeps the walk's compares and shuffles single-word.
struct LaneSpan {
    int32_t cs, ce, tl;
    int cnt;
};

// Tile-row of the lane's first tile, and rowptr[row], rowptr[row+1]; the
// chunk's rows r0..r1 come from the schedule, a window of row pointers from
// one coalesced load, and the search is a shuffle binary search.
struct RowCursor {
    int32_t row;
    int32_t row_start, next;
    bool head_cs;
};

// Row pointers of a chunk's tile-rows r0 .. r0+span+1 that fit one warp
// (lane j holds rowptr[r0 + j]); the search loads any further windows itself.
__device__ __forceinline__ int32_t row_window(const SpmvGeom& g, int32_t r0, int32_t span, int lane) {
    return lane <= span + 1 ? __ldg(g.rowptr + r0 + lane) : INT32_MAX;
}

__device__ __forceinline__ RowCursor locate_row_win(const SpmvGeom& g, int32_t r0, int32_t span, int32_t win,
                                                    const LaneSpan& ls, int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    RowCursor rc;
    rc.head_cs = __shfl_sync(FULL, win, 0) == ls.cs;
    int32_t row = r0;
    if (span > 0) {
        // first window: the row starts are lanes 1..31 (lane 0 is rowptr[r0])
        const int32_t b = lane == 0 ? INT32_MIN : win;
        int pos = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            const int32_t v = __shfl_sync(FULL, b, pos + step - 1);
            if (v <= ls.tl) pos += step;
        }
        pos += (__shfl_sync(FULL, b, pos) <= ls.tl) ? 1 : 0;
        int32_t add = pos - 1;  // lane 0 is always counted
        int32_t last = __shfl_sync(FULL, win, 31);
        for (int32_t base = 32; base <= span && last < ls.ce; base += 32) {
            // further windows (rare: many tile-rows in one chunk)
            const int32_t j = base + lane;
            const int32_t bb = j <= span ? __ldg(g.rowptr + r0 + j) : INT32_MAX;
            int p2 = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int32_t v = __shfl_sync(FULL, bb, p2 + step - 1);
                if (v <= ls.tl) p2 += step;
            }
            p2 += (__shfl_sync(FULL, bb, p2) <= ls.tl) ? 1 : 0;
            add += p2;
            last = __shfl_sync(FULL, bb, 31);
        }
        row = r0 + add;
    }
    const int d = row - r0;
    const int32_t a0 = __shfl_sync(FULL, win, d < 32 ? d : 0);
    const int32_t a1 = __shfl_sync(FULL, win, d + 1 < 32 ? d + 1 : 0);
    rc.row = row;
    rc.row_start = d < 32 ? a0 : __ldg(g.rowptr + row);
    rc.next = d + 1 < 32 ? a1 : __ldg(g.rowptr + row + 1);
    return rc;
}

__device__ __forceinline__ RowCursor locate_row(const SpmvGeom& g, int32_t c, const LaneSpan& ls, int lane) {
    const int32_t r0 = __ldg(g.chunk_row + c);
    const int32_t span = __ldg(g.chunk_row + c + 1) - r0;
    return locate_row_win(g, r0, span, row_window(g, r0, span, lane), ls, lane);
}

// Per-lane walk state: the tile-row being accumulated, where it ends, the
// values of the lane's first tile-row (F) once that row has ended.
template <class SEM, class Acc>
struct Walk {
    int32_t row;
    int32_t next;
    bool has_end = false;
    bool open = false;
    // called after tile t (the lane's i-th of cnt) has been accumulated
    __device__ __forceinline__ void end_tile(const SpmvGeom& g, const SEM& sem, Acc& acc, Acc& F, int32_t t, int i,
                                             int cnt, const RegAcc<typename SEM::V, SEM::NV>& idv) {
        open = true;
        if (t + 1 == next) {  // tile-row `row` ends with tile t
            if (!has_end) {
#pragma unroll
                for (int v = 0; v < SEM::NV; ++v) F.set(v, acc.get(v));
                has_end = true;
            } else {
                sem.store(row, acc);
            }
#pragma unroll
            for (int v = 0; v < SEM::NV; ++v) acc.set(v, sem.ident());
            open = false;
            if (i + 1 < cnt) {
                int32_t R = row + 1;
                while (__ldg(g.rowptr + R + 1) == next) { sem.store(R, idv); ++R; }
                row = R;
                next = __ldg(g.rowptr + row + 1);
            }
        }
    }
};

// Warp segmented scan of (reset = has_end, value = acc), then: lanes that end
// their first tile-row store it (or leave it as the chunk's first partial if
// it began in an earlier chunk); lane 31 leaves the still-open tail.
template <class SEM, class Acc, class First>
__device__ __forceinline__ void close_chunk(const SEM& sem, Partials<typename SEM::V> part, int64_t c,
                                            const LaneSpan& ls, int lane, bool head_cs, int32_t first_row,
                                            bool has_end, bool open, Acc& acc, First& F, int P,
                                            int32_t tail_row = 0) {
    using V = typename SEM::V;
    constexpr int NV = SEM::NV;
    constexpr unsigned FULL = 0xffffffffu;
    // The reset pattern does not depend on the values, so which scan steps
    // take a neighbour's value is worked out once, then applied per value.
    bool take[5];
    bool inc_r = has_end;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int d = 1 << k;
        const bool o = __shfl_up_sync(FULL, inc_r, d);
        take[k] = lane >= d && !inc_r;
        if (take[k]) inc_r = o;
    }
    bool ex_r = __shfl_up_sync(FULL, inc_r, 1);
    if (lane == 0) ex_r = false;
    const int la = (int)((ls.ce - 1 - ls.cs) / P);
    const bool tail_open = __shfl_sync(FULL, open, la);
    const bool tail_r = __shfl_sync(FULL, inc_r, 31);
    const bool close_here = has_end && (OrsInto<SEM>::value || ex_r || head_cs);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        V x = acc.get(v);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const V o = shfl_up(x, 1 << k);
            if (take[k]) x = sem.comb(o, x);
        }
        const V ex = shfl_up(x, 1);
        if (has_end && lane > 0) F.set(v, sem.comb(ex, F.get(v)));
        if constexpr (OrsInto<SEM>::value) {
            acc.set(v, x);  // lane 31: the open tail
            continue;
        }
        if (has_end && !close_here) part.val_first[c * NV + v] = F.get(v);
        if (lane == 31 && tail_open) {
            if (tail_r || head_cs) part.val_last[c * NV + v] = x;
            else part.val_first[c * NV + v] = x;
        }
    }
    if (close_here) sem.store(first_row, F);
    if constexpr (OrsInto<SEM>::value)
        if (lane == 31 && tail_open) sem.store(tail_row, acc);
}

// 32 bytes from global memory in one load, not allocated in L1: each tile
// is read once, and L1 is left to the input-vector gathers.  A whole 32-byte
// sector per instruction: narrower no-allocate loads would fetch a sector
// again for every part of it.
__device__ __forceinline__ void ld32_stream(const void* p, uint32_t (&v)[8]) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p));
}

// The same load without `volatile`: the compiler may schedule it with the
// other loads of the lane (the data is read-only while a kernel runs).
__device__ __forceinline__ void ld32_stream_free(const void* p, uint32_t (&v)[8]) {
    asm("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "l"(p));
}

// 16 bytes, not allocated in L1.
__device__ __forceinline__ uint4 ld16_stream(const void* p) {
    uint4 v;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}

template <int K>
__device__ __forceinline__ void load_lane_tiles(const SpmvGeom& g, int32_t tl, uint4 (&tv)[ChunkShape<K>::TILE_V4],
                                                int32_t (&col)[ChunkShape<K>::P]) {
    using S = ChunkShape<K>;
    constexpr int P = S::P;
    // a lane's P tiles are P * TB = 32, 64, 128 or 256 bytes, 32-byte aligned (tl is a multiple of P)
    static_assert(S::TILE_V4 % 2 == 0, "whole 32-byte sectors of tiles per lane");
    const uint8_t* src = g.tiles + (int64_t)tl * S::TB;
    if constexpr (K == 4) {
        // k = 4 (32 bytes of tiles and of columns a lane): two 16-byte loads
        // each measured faster here than one 32-byte load (161 against 166 us
        // for the plus-times SpMV on R-MAT 20); from k = 8 the 32-byte load wins
#pragma unroll
        for (int q = 0; q < S::TILE_V4; ++q) tv[q] = ld16_stream(src + 16 * q);
        const uint4 c0 = ld16_stream(g.colind + tl), c1 = ld16_stream(g.colind + tl + 4);
        col[0] = (int32_t)c0.x; col[1] = (int32_t)c0.y; col[2] = (int32_t)c0.z; col[3] = (int32_t)c0.w;
        col[4] = (int32_t)c1.x; col[5] = (int32_t)c1.y; col[6] = (int32_t)c1.z; col[7] = (int32_t)c1.w;
        return;
    }
#pragma unroll
    for (int q = 0; q < S::TILE_V4 / 2; ++q) {
        uint32_t v[8];
        ld32_stream_free(src + 32 * q, v);
        tv[2 * q] = make_uint4(v[0], v[1], v[2], v[3]);
        tv[2 * q + 1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
    if constexpr (P == 8) {  // 32 bytes of column indices: one sector
        uint32_t v[8];
        ld32_stream_free(g.colind + tl, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) col[i] = (int32_t)v[i];
    } else if constexpr (P % 4 == 0) {  // lanes share sectors: cached loads
        const int4* cs = reinterpret_cast<const int4*>(g.colind + tl);
#pragma unroll
        for (int q = 0; q < P / 4; ++q) {
            int4 v = __ldg(cs + q);
            col[4 * q] = v.x; col[4 * q + 1] = v.y; col[4 * q + 2] = v.z; col[4 * q + 3] = v.w;
        }
    } else {
        const int2* cs = reinterpret_cast<const int2*>(g.colind + tl);
#pragma unroll
        for (int q = 0; q < P / 2; ++q) {
            int2 v = __ldg(cs + q);
            col[2 * q] = v.x; col[2 * q + 1] = v.y;
        }
    }
}

// ---------------------------------------------------------------------------
// chunk kernel for the bit-vector schemes at k = 16 and 32, for counts at k = 8
// where rows are short, and for the value schemes that neither the small-tile,
// the row-lane nor the staged kernel takes: registers hold the accumulators
// (static row indices)
// ---------------------------------------------------------------------------
template <int K, class SEM>
__global__ void __launch_bounds__(kSpmvThreads) spmv_chunks_kernel(SpmvGeom g, SEM sem,
                                                                   Partials<typename SEM::V> part) {
    using S = ChunkShape<K>;
    using V = typename SEM::V;
    constexpr int NV = SEM::NV;
    constexpr int P = S::P;
    const int warp = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    const int32_t c = (int32_t)blockIdx.x * kSpmvWarps + warp;
    if (c >= g.nchunks || gated_off(g.gate)) return;  // whole warps leave together

    LaneSpan ls;
    ls.cs = c * S::CT;
    ls.ce = min(ls.cs + S::CT, (int32_t)g.T);
    ls.tl = ls.cs + lane * P;
    ls.cnt = max(0, min(P, ls.ce - ls.tl));

    uint4 tv[S::TILE_V4];
    int32_t col[P];
    // a chunk whose every output row is masked out reads no tiles (zero words:
    // the walk still stores its rows and partials, all the identity)
    bool sat = false;
    {
        const int32_t ra = __ldg(g.chunk_row + c), rb = __ldg(g.chunk_row + c + 1);
        sat = sem.saturated((int64_t)ra * K, ((int64_t)rb + 1) * K);
    }
    if (!sat) {
        load_lane_tiles<K>(g, ls.tl, tv, col);
    } else {
#pragma unroll
        for (int q = 0; q < S::TILE_V4; ++q) tv[q] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int i = 0; i < P; ++i) col[i] = 0;
    }
    const uint32_t* words = reinterpret_cast<const uint32_t*>(tv);
    uint32_t xs[SEM::kGather ? 1 : P];
    if constexpr (!SEM::kGather) {
#pragma unroll
        for (int i = 0; i < P; ++i) xs[i] = sem.xseg(col[i]);
    }
    const RowCursor rc = locate_row(g, c, ls, lane);

    RegAcc<V, NV> acc, F, idv;
#pragma unroll
    for (int v = 0; v < NV; ++v) { acc.set(v, sem.ident()); F.set(v, sem.ident()); idv.set(v, sem.ident()); }
    Walk<SEM, RegAcc<V, NV>> wk;
    wk.row = rc.row;
    wk.next = rc.next;
    if (ls.cnt > 0) {
        // empty tile-rows just before a row that starts at this lane's first tile
        if (ls.tl > 0 && rc.row_start == ls.tl)
            for (int32_t R = rc.row - 1; R >= 0 && __ldg(g.rowptr + R) == ls.tl; --R) sem.store(R, idv);
#pragma unroll
        for (int i = 0; i < P; ++i) {
            if (i < ls.cnt) {
                const int32_t t = ls.tl + i;
                if constexpr (!SEM::kGather) {
                    sem.tile(acc, words + i * S::TW, xs[i]);
                } else {
                    using G = typename SEM::G;
                    const G* xt = sem.src() + (int64_t)col[i] * K;
                    const float* wt = sem.weighted ? sem.wts() + __ldg(sem.voffs() + t) : nullptr;
                    int qb = 0;
#pragma unroll
                    for (int q = 0; q < S::TW; ++q) {
                        uint32_t b = words[i * S::TW + q];
                        while (b) {
                            const int bit = __ffs(b) - 1;
                            b &= b - 1;
                            const int r = q * (32 / S::ROW_BITS) + bit / S::ROW_BITS;
                            const float wv = sem.weighted ? __ldg(wt + qb) : 1.0f;
                            const G xv = __ldg(xt + bit % S::ROW_BITS);
                            if constexpr (sizeof(V) == 8 && NV <= 8) {
                                // 8-byte accumulators: a predicated update of
                                // each row keeps the indices constant (a
                                // runtime index puts the array in local memory)
#pragma unroll
                                for (int v = 0; v < NV; ++v)
                                    if (v == r) acc.set(v, sem.apply(acc.get(v), xv, wv));
                            } else {
                                acc.set(r, sem.apply(acc.get(r), xv, wv));
                            }
                            ++qb;
                        }
                    }
                }
                wk.end_tile(g, sem, acc, F, t, i, ls.cnt, idv);
            }
        }
    }
    close_chunk(sem, part, c, ls, lane, rc.head_cs, rc.row, wk.has_end, wk.open, acc, F, P);
}

// ---------------------------------------------------------------------------
// small-tile chunk kernel: the bit-vector schemes (Boolean and count SpMVs) at
// k = 4 and 8, and at k = 4 the unweighted value schemes with 4- and 8-byte
// values (plus-times, label min, fp32 max, 32- and 64-lane OR).  A tile is one
// 32- or 64-bit word there, 256 tiles a chunk, so the kernel is bound by
// instructions and by the input gathers, not by the tile stream:
//   * persistent warps: warp gw takes chunks gw, gw + W, ... and loads the
//     next chunk's tile stream into registers before it works on the current
//     one, so every warp keeps a chunk in flight;
//   * a value scheme loads the whole 4-value input segment under a tile in
//     one 16- or 32-byte load (a gather costs a 32-byte sector whatever its
//     width) and adds it under the tile's 16 bits, with no loop over set bits:
//     nothing diverges, and every load of a lane is in flight at once;
//   * the chunk's row ends become a 256-bit mask and a table of row numbers in
//     shared memory, made from one coalesced load of row pointers, so the walk
//     tests one bit per tile and loads no row pointers;
//   * a chunk inside one tile-row (more than half of them on a power-law
//     graph) needs no walk: one fixed-order tree joins the lanes.
// What bounds the value schemes is the L1 data pipe: a gather takes one
// wavefront per distinct 128-byte line, 32 a warp for scattered columns (79%
// of the pipe, 27.2M wavefronts an SpMV on R-MAT 20 before the tiles of
// one-row chunks were dealt out).  R-MAT 20, k = 4, direct schedule, SpMV call
// in us before / after (one gather per set bit, a row search and a row-pointer
// walk per lane before): plus-times 173 / 118 (permuted ids 148 / 138), label
// min 183 / 129 (154 / 144), 64-lane OR 238 / 176, four fp32 columns 312 / 224
// (236 / 194); Boolean 86 / 59 at k = 4 and 99 / 63 at k = 8.  Warp
// instructions of the plus-times kernel: 98M / 59M.
// ---------------------------------------------------------------------------
// lane-word schemes
template <class S>
struct LaneWords : std::false_type {};
template <int K, class W>
struct LaneWords<SemOrLanes<K, W>> : std::true_type {};

// min and max schemes
template <class S>
struct MinMax : std::false_type {};
template <int K>
struct MinMax<SemMinI32<K>> : std::true_type {};
template <int K>
struct MinMax<SemMaxF32<K>> : std::true_type {};

// How a scheme reads its input: bits from global memory, bits from the
// block's copy of the whole bitset in shared memory, whole aligned segments of
// values, one value per set column (an input that is not aligned to a segment,
// or whose last segment is ragged; 16-byte values, whose segment would be two
// sectors), or one value per set bit in a loop (8- and 16-byte values where
// tiles hold hardly more than one: the 16 predicated updates are 32 and 64
// instructions then), or segments where the block's copy of `live` says that
// they are not all zero (the sparse levels of a batched BFS).
enum { kSmBits = 0, kSmBitsShared = 1, kSmSegs = 2, kSmVals = 3, kSmEach = 4, kSmSegsLive = 5, kRowLanes = 6 };
// Threads a block, and the resident blocks the registers are budgeted for
// (every lane holds two chunks' tile words and columns; with 16-byte values
// one).  R-MAT 20, k = 4, in
// us with 4 / 3 blocks an SM: plus-times 126 / 128, label min 145 / 135 (four
// blocks spill there), 16-source BFS 1,265 / 1,330; four columns by bit with 4
// / 3 / 2 blocks 237 / 269 / 385.  The shared bitset leaves
// room for one block: k = 8 with 512 / 640 / 768 threads 83 / 74 / 72.5.
template <int K, class SEM, int MODE>
constexpr int small_threads() {
    if (MODE == kSmSegsLive) return sizeof(typename SEM::V) == 8 ? 768 : 1024;
    if (MODE != kSmBitsShared) return kSpmvThreads;
    return K == 4 ? 1024 : (SEM::NV == 8 ? 640 : 768);  // eight counts a row need the registers
}
template <int K, class SEM, int MODE>
constexpr int small_min_blocks() {
    if (MODE == kSmBitsShared || MODE == kSmSegsLive) return 1;
    if (MODE == kRowLanes) return sizeof(typename SEM::V) == 16 ? 4 : 6;
    if (sizeof(typename SEM::V) == 16) return MODE == kSmEach ? 4 : 3;
    if (SEM::NV == 8) return 2;
    return K == 8 || sizeof(typename SEM::V) == 8 || MinMax<SEM>::value ? 3 : 4;
}

// The tile stream of one chunk as a lane holds it: the chunk's first tile-row
// and that of the next chunk, their row pointers (lane j: rowptr[ra + j]),
// and the lane's 8 tiles and columns.  Words are zero where every output row
// of the chunk is masked out (no tiles are read then; the walk still stores
// its rows and partials, all the identity).
template <int K>
struct SmallTiles {
    static constexpr int TW = ChunkShape<K>::TW;
    int32_t ra, rb;
    int32_t win;
    bool dead;  // every row is masked out
    uint32_t w[8 * TW], cu[8];
};

__device__ __forceinline__ uint32_t ld4_stream(const void* p) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];\n" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void ld8_stream(const void* p, uint32_t& a, uint32_t& b) {
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];\n" : "=r"(a), "=r"(b) : "l"(p));
}

// ra, rb: chunk_row[c], chunk_row[c + 1]
template <int K, class SEM>
__device__ __forceinline__ void small_load(const SpmvGeom& g, const SEM& sem, int32_t c, int lane, int32_t ra,
                                           int32_t rb, SmallTiles<K>& t) {
    constexpr int TW = SmallTiles<K>::TW;
    t.ra = ra;
    t.rb = rb;
    t.win = row_window(g, ra, rb - ra, lane);
    const int64_t c0 = (int64_t)c * chunk_tiles(K);
    const uint32_t* tiles = reinterpret_cast<const uint32_t*>(g.tiles);
    // the arrays are padded to whole chunks, so every lane's bytes exist
    t.dead = sem.saturated((int64_t)ra * K, ((int64_t)rb + 1) * K);
    if (t.dead) {
#pragma unroll
        for (int i = 0; i < 8 * TW; ++i) t.w[i] = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) t.cu[i] = 0u;
    } else if (ra == rb) {
        // inside one tile-row the tiles are dealt to the lanes (lane l: tiles l,
        // l + 32, ...): a gather's 32 lanes then have neighbouring columns and
        // share lines (R-MAT 20: 23 distinct 128-byte lines instead of 32)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int64_t tl = c0 + 32 * i + lane;
            if constexpr (TW == 1) t.w[i] = ld4_stream(tiles + tl);
            else ld8_stream(tiles + 2 * tl, t.w[2 * i], t.w[2 * i + 1]);
            t.cu[i] = ld4_stream(g.colind + tl);
        }
    } else {
        const int64_t tl = c0 + lane * 8;
#pragma unroll
        for (int q = 0; q < TW; ++q) {
            uint32_t v[8];
            ld32_stream(tiles + tl * TW + 8 * q, v);
#pragma unroll
            for (int i = 0; i < 8; ++i) t.w[8 * q + i] = v[i];
        }
        ld32_stream(g.colind + tl, t.cu);
    }
}

// Row ends of a chunk, per warp: bit t of `mask` is set iff tile cs + t is the
// last of its tile-row; row[j] is the tile-row of the j-th such tile.
struct ChunkRows {
    uint32_t mask[8];
    int32_t row[256];
};

// Fills s from the chunk's row pointers, 31 rows a step (lane j of a step: the
// row starting at its pointer, ending at lane j + 1's); stores the identity
// for the empty tile-rows between ra and rb, which hold the first tiles of
// this and the next chunk, so that each is stored by one chunk.  The row count,
// whose empty rows need no store, looks up every tile's row instead where most
// rows are empty (2^26 rows with 2,000 entries, k = 4: the steps took 42 ms).
template <class SEM, class Acc>
__device__ __forceinline__ void chunk_ends(const SpmvGeom& g, const SEM& sem, int32_t ra, int32_t rb, int32_t win,
                                           int32_t cs, int32_t ce, int lane, const Acc& idv, ChunkRows& s) {
    constexpr unsigned FULL = 0xffffffffu;
    __syncwarp();  // the previous chunk's readers are done
    if (lane < 8) s.mask[lane] = 0u;
    __syncwarp();
    const int32_t span = rb - ra;
    int found = 0;
    if constexpr (NoInput<SEM>::value) {
        if (span > 1024) {
            for (int i = 0; cs + 32 * i < ce; ++i) {
                const int32_t t = cs + 32 * i + lane;
                int32_t lo = ra, hi = rb;
                while (lo < hi) {
                    const int32_t mid = lo + ((hi - lo + 1) >> 1);
                    if (__ldg(g.rowptr + mid) <= t) lo = mid; else hi = mid - 1;
                }
                const bool end = t < ce && __ldg(g.rowptr + lo + 1) == t + 1;
                const unsigned ends = __ballot_sync(FULL, end);
                if (end) s.row[found + __popc(ends & ((1u << lane) - 1u))] = lo;
                if (lane == 0) s.mask[i] = ends;
                found += __popc(ends);
            }
            __syncwarp();
            return;
        }
    }
    for (int32_t j0 = 0; j0 <= span; j0 += 31) {
        const int32_t j = j0 + lane;
        const int32_t a = j0 == 0 ? win : (j <= span + 1 ? __ldg(g.rowptr + ra + j) : INT32_MAX);
        const int32_t b = __shfl_down_sync(FULL, a, 1);
        const bool row = lane < 31 && j <= span;
        const bool end = row && b > a && b > cs && b <= ce;
        const unsigned ends = __ballot_sync(FULL, end);
        if (end) {
            s.row[found + __popc(ends & ((1u << lane) - 1u))] = ra + j;
            atomicOr(&s.mask[(b - 1 - cs) >> 5], 1u << ((b - 1 - cs) & 31));
        } else if (!OrsInto<SEM>::value && !NoInput<SEM>::value && row && a == b) {
            sem.store(ra + j, idv);
        }
        found += __popc(ends);
    }
    __syncwarp();
}

// The four input values under a k = 4 tile.
template <class G, int MODE>
__device__ __forceinline__ void load_seg(const G* __restrict__ x, uint32_t J, uint32_t w, G (&v)[4]) {
    if constexpr (MODE == kSmSegs || MODE == kSmSegsLive) {
        if constexpr (sizeof(G) == 4) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(x) + J);
            const uint32_t u[4] = {q.x, q.y, q.z, q.w};
            memcpy(v, u, sizeof(v));
        } else {
            uint32_t u[8];
            asm("ld.global.nc.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
                : "l"(x + 4 * (int64_t)J));
            memcpy(v, u, sizeof(v));
        }
    } else {
        const uint32_t cols = w | (w >> 8) | (w >> 16) | (w >> 24);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if ((cols >> c) & 1u) v[c] = __ldg(x + 4 * (int64_t)J + c);
            else v[c] = G();
    }
}

// Adds the tile's rows (row r in byte r of w) to the row accumulators, columns
// in increasing order.
template <class SEM, class G, class Acc>
__device__ __forceinline__ void seg_add(const SEM& sem, Acc& acc, uint32_t w, const G (&v)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (w & (1u << (8 * r + c))) acc.set(r, sem.apply(acc.get(r), v[c], 1.0f));
    }
}

// One value per set bit; the first bit's (most tiles have no other) is loaded
// beforehand, so that those of several tiles are in flight together.
template <class G>
__device__ __forceinline__ G first_value(const G* __restrict__ x, uint32_t J, uint32_t w) {
    return w ? __ldg(x + 4 * (int64_t)J + ((__ffs(w) - 1) & 7)) : G();
}
template <class SEM, class G, class Acc>
__device__ __forceinline__ void each_add(const SEM& sem, Acc& acc, uint32_t J, uint32_t w, G v) {
    while (w) {
        const int r = (__ffs(w) - 1) >> 3;
        w &= w - 1;
        G more = G();
        if (w) more = first_value(sem.src(), J, w);
#pragma unroll
        for (int u = 0; u < 4; ++u)  // constant indices keep the accumulators in registers
            if (u == r) acc.set(u, sem.apply(acc.get(u), v, 1.0f));
        v = more;
    }
}

// Joins the lanes' NV values with the tree of a butterfly (lane pairs, then
// pairs of pairs, ...: the order of the segmented scan's last lane).  Value
// schemes: the first levels halve the values a lane carries, so lane l < NV
// ends with value joined_value<NV>(l) in slot 0; bit schemes: every lane ends
// with all.
template <int NV>
__device__ __forceinline__ int joined_value(int lane) {
    int v = 0;
#pragma unroll
    for (int d = 1, half = NV / 2; half >= 1; d <<= 1, half >>= 1) v += (lane & d) ? half : 0;
    return v;
}

template <class SEM, class Acc>
__device__ __forceinline__ void join_lanes(const SEM& sem, Acc& acc, int lane) {
    using V = typename SEM::V;
    constexpr int NV = SEM::NV;
    constexpr unsigned FULL = 0xffffffffu;
    if constexpr (!SEM::kGather) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
            acc.set(v, std::is_signed<V>::value ? (V)__reduce_add_sync(FULL, (int)acc.get(v))
                                                : (V)__reduce_or_sync(FULL, (unsigned)acc.get(v)));
    } else {
#pragma unroll
        for (int d = 1, half = NV / 2; d < 32; d <<= 1, half = half > 1 ? half / 2 : 0) {
            const bool hi = lane & d;
            if (half >= 1) {
#pragma unroll
                for (int v = 0; v < half; ++v) {
                    const V send = hi ? acc.get(v) : acc.get(v + half), keep = hi ? acc.get(v + half) : acc.get(v);
                    const V o = shfl_xor(send, d);
                    acc.set(v, hi ? sem.comb(o, keep) : sem.comb(keep, o));
                }
            } else {
                const V o = shfl_xor(acc.get(0), d);
                acc.set(0, hi ? sem.comb(o, acc.get(0)) : sem.comb(acc.get(0), o));
            }
        }
    }
}

// A chunk (not the last) without a contribution, of a lane-word scheme: zeros
// for the rows that end here and began here or are empty, which are neighbours,
// and for the chunk's shares of the rows that it cuts.  Such chunks are most of
// the first and the last levels of a batched BFS, whose walks found nothing to
// add: the SpMMs of a search, with 16 sources on R-MAT 20, 967 to 858 us, with
// 64 on R-MAT 22, 4,571 to 3,949 (811 and 3,755 with a loop for each case in
// small_body).
template <class SEM>
__device__ __forceinline__ void zero_chunk(const SpmvGeom& g, const SEM& sem, Partials<typename SEM::V> part, int32_t c,
                                           int32_t cs, int lane, int32_t ra, int32_t rb, int32_t start) {
    using V = typename SEM::V;
    constexpr int K = SEM::NV;
    if (lane < K) {
        part.val_first[(int64_t)c * K + lane] = V(0);
        part.val_last[(int64_t)c * K + lane] = V(0);
    }
    const int64_t end = min((int64_t)rb * K, (int64_t)sem.n);  // row rb goes on after the chunk or begins there
    for (int64_t i = ((int64_t)ra + (start == cs ? 0 : 1)) * K + lane; i < end; i += 32) sem.y[i] = V(0);
}

// One chunk from its loaded tile stream.
template <int K, class SEM, int MODE>
__device__ __forceinline__ void small_chunk(const SpmvGeom& g, const SEM& sem, Partials<typename SEM::V> part,
                                            int32_t c, int lane, const SmallTiles<K>& t, ChunkRows& s,
                                            const uint8_t* sx, typename SEM::V* first) {
    using Sh = ChunkShape<K>;
    using V = typename SEM::V;
    constexpr int NV = SEM::NV;
    constexpr int TW = Sh::TW;
    static_assert(Sh::P == 8 && TW <= 2, "eight tiles of one or two words a lane");
    const int32_t cs = c * Sh::CT;
    const int32_t ce = min(cs + Sh::CT, (int32_t)g.T);
    uint32_t on = 0xFFu;  // kSmSegsLive: the lane's tiles under which a segment is not all zero
    if constexpr (LaneWords<SEM>::value) {
        bool dead = t.dead;
        if constexpr (MODE == kSmSegsLive) {
            if (!dead) {
                on = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    on |= ((reinterpret_cast<const uint32_t*>(sx)[t.cu[i] >> 5] >> (t.cu[i] & 31)) & 1u) << i;
                dead = !__any_sync(0xffffffffu, on != 0u);
            }
        }
        if (dead && c + 1 < g.nchunks) {
            zero_chunk(g, sem, part, c, cs, lane, t.ra, t.rb, __shfl_sync(0xffffffffu, t.win, 0));
            return;
        }
    }
    RegAcc<V, NV> acc, idv;
    // the values of the lane's first tile-row: in shared memory where they are wide
    typename std::conditional<sizeof(V) == 16, SmemAcc<V, NV>, RegAcc<V, NV>>::type F;
    if constexpr (sizeof(V) == 16) F.p = first + lane;
#pragma unroll
    for (int v = 0; v < NV; ++v) { acc.set(v, sem.ident()); F.set(v, sem.ident()); idv.set(v, sem.ident()); }
    const bool one_row = t.ra == t.rb;  // warp-uniform: the whole chunk lies in tile-row ra
    uint32_t ends = 0u;
    int rank = 0;
    if (!one_row) {
        chunk_ends(g, sem, t.ra, t.rb, t.win, cs, ce, lane, idv, s);
        ends = reinterpret_cast<const uint8_t*>(s.mask)[lane];
        rank = __popc(ends);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, rank, d);
            if (lane >= d) rank += o;
        }
        rank -= __popc(ends);  // row ends before the lane's tiles
    }
    const int rank0 = rank;
    bool has_end = false;
    auto end_tile = [&](int i) {
        if (!((ends >> i) & 1u)) return;
        if (!has_end) {  // the lane's first row: joined with earlier lanes below
#pragma unroll
            for (int v = 0; v < NV; ++v) F.set(v, acc.get(v));
            has_end = true;
        } else {
            sem.store(s.row[rank], acc);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) acc.set(v, sem.ident());
        ++rank;
    };
    if constexpr (SEM::kGather) {
        // tiles whose segments are loaded together (plus-times on R-MAT 20: 1, 2,
        // 4 tiles 127, 126, 130 us; the loads of more cost registers)
        constexpr int GRP = MODE == kSmVals && sizeof(V) == 16 ? 1 : 2;
        using G = typename SEM::G;
#pragma unroll
        for (int i0 = 0; i0 < 8; i0 += GRP) {
            if constexpr (MODE == kSmEach) {
                G x[GRP];
#pragma unroll
                for (int i = 0; i < GRP; ++i) x[i] = first_value(sem.src(), t.cu[i0 + i], t.w[i0 + i]);
#pragma unroll
                for (int i = 0; i < GRP; ++i) {
                    each_add(sem, acc, t.cu[i0 + i], t.w[i0 + i], x[i]);
                    if (!one_row) end_tile(i0 + i);
                }
            } else {
                G x[GRP][4];
                bool any = true;  // warp-uniform: some lane's segments are not all zero
                if constexpr (MODE == kSmSegsLive) {
                    any = __any_sync(0xffffffffu, ((on >> i0) & ((1u << GRP) - 1u)) != 0u);
                    if (any) {
#pragma unroll
                        for (int i = 0; i < GRP; ++i) {
                            if ((on >> (i0 + i)) & 1u) {
                                load_seg<G, MODE>(sem.src(), t.cu[i0 + i], t.w[i0 + i], x[i]);
                            } else {
#pragma unroll
                                for (int c = 0; c < 4; ++c) x[i][c] = G();
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < GRP; ++i)
                        load_seg<G, MODE>(sem.src(), t.cu[i0 + i], t.w[i0 + i], x[i]);
                }
#pragma unroll
                for (int i = 0; i < GRP; ++i) {
                    if (any) seg_add(sem, acc, t.w[i0 + i], x[i]);
                    if (!one_row) end_tile(i0 + i);
                }
            }
        }
    } else {
        uint32_t xs[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if constexpr (MODE == kSmBitsShared)
                xs[i] = K == 8 ? sx[t.cu[i]] : (sx[t.cu[i] >> 1] >> (4 * (t.cu[i] & 1u))) & 0xFu;
            else
                xs[i] = sem.xseg((int32_t)t.cu[i]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sem.tile(acc, t.w + i * TW, xs[i]);
            if (!one_row) end_tile(i);
        }
    }
    if (one_row) {
        const bool head = __shfl_sync(0xffffffffu, t.win, 0) == cs;  // the row begins with this chunk
        join_lanes(sem, acc, lane);
        if constexpr (OrsInto<SEM>::value) {
            if (lane == 0) sem.store(t.ra, acc);
            return;
        }
        if (head && c + 1 == g.nchunks) {  // begins and ends in this chunk (the matrix's last)
            if constexpr (SEM::kGather) {
                if (lane < NV) sem.store_row(t.ra, joined_value<NV>(lane), acc.get(0));
            } else if (lane == 0) {
                sem.store(t.ra, acc);
            }
            return;
        }
        // continued by later chunks (head) or begun in earlier ones
        V* dst = (head ? part.val_last : part.val_first) + (int64_t)c * NV;
        if constexpr (SEM::kGather) {
            if (lane < NV) dst[joined_value<NV>(lane)] = acc.get(0);
        } else if (lane == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) dst[v] = acc.get(v);
        }
        return;
    }
    LaneSpan ls;
    ls.cs = cs;
    ls.ce = ce;
    const bool head_cs = __shfl_sync(0xffffffffu, t.win, 0) == cs;
    // a tail after the chunk's last row end is continued by the next chunk
    const bool open = !((s.mask[(ce - 1 - cs) >> 5] >> ((ce - 1 - cs) & 31)) & 1u);
    const int32_t first_row = has_end ? s.row[rank0] : 0;
    close_chunk(sem, part, c, ls, lane, head_cs, first_row, has_end, open, acc, F, Sh::P, t.rb);
}

// Dynamic shared memory a warp: its ChunkRows, and for 16-byte values the
// lanes' first rows.
template <class SEM>
constexpr int small_warp_smem() {
    return (int)sizeof(ChunkRows) + (sizeof(typename SEM::V) == 16 ? 32 * SEM::NV * 16 : 0);
}

// Dynamic shared memory: that for every warp, then (kSmBitsShared,
// kSmSegsLive) the input bitset.
template <int K, class SEM, int MODE>
__device__ __forceinline__ void small_body(const SpmvGeom& g, const SEM& sem, Partials<typename SEM::V> part) {
    constexpr int WARPS = small_threads<K, SEM, MODE>() / 32;
    extern __shared__ __align__(16) uint8_t small_smem[];
    if (gated_off(g.gate)) return;
    uint8_t* mine = small_smem + (threadIdx.x >> 5) * small_warp_smem<SEM>();
    ChunkRows* rows = reinterpret_cast<ChunkRows*>(mine);
    typename SEM::V* first = reinterpret_cast<typename SEM::V*>(mine + sizeof(ChunkRows));  // 16-byte values only
    const uint8_t* sx = small_smem + WARPS * small_warp_smem<SEM>();
    const int lane = (int)lane_id();
    const int32_t W = (int32_t)gridDim.x * WARPS;
    int32_t c = (int32_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    SmallTiles<K> cur, nxt;
    // tile-rows of the chunk after the loaded one: its loads depend on them
    int32_t na = 0, nb = 0;
    if (c < g.nchunks) {
        small_load<K>(g, sem, c, lane, __ldg(g.chunk_row + c), __ldg(g.chunk_row + c + 1), cur);
        if (c + W < g.nchunks) {
            na = __ldg(g.chunk_row + c + W);
            nb = __ldg(g.chunk_row + c + W + 1);
        }
    }
    bool filter = false;
    if constexpr (MODE == kSmSegsLive) filter = __ldg(sem.dense) == 0;
    if (MODE == kSmBitsShared || filter) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(small_smem + WARPS * small_warp_smem<SEM>());
        const uint32_t* bits;
        int words;
        if constexpr (MODE == kSmSegsLive) {
            bits = sem.live;
            words = (g.ntr + 31) / 32;
        } else {
            bits = reinterpret_cast<const uint32_t*>(sem.x);
            words = (sem.n + 31) / 32;
        }
        int at = 0;
        if (reinterpret_cast<uintptr_t>(bits) % 16 == 0) {
            const uint4* src = reinterpret_cast<const uint4*>(bits);
            for (int i = threadIdx.x; i < words / 4; i += WARPS * 32) reinterpret_cast<uint4*>(dst)[i] = __ldg(src + i);
            at = words & ~3;
        }
        for (int i = at + threadIdx.x; i < words; i += WARPS * 32) dst[i] = __ldg(bits + i);
        __syncthreads();
    }
    if (c >= g.nchunks) return;  // whole warps leave together
    if constexpr (sizeof(typename SEM::V) == 16) {
        // one chunk at a time: more warps hide its loads better than the
        // registers of a second chunk would (R-MAT 20: 225 and 270 us)
        for (;;) {
            small_chunk<K, SEM, MODE>(g, sem, part, c, lane, cur, *rows, sx, first);
            c += W;
            if (c >= g.nchunks) return;
            small_load<K>(g, sem, c, lane, na, nb, cur);
            if (c + W < g.nchunks) {
                na = __ldg(g.chunk_row + c + W);
                nb = __ldg(g.chunk_row + c + W + 1);
            }
        }
    }
    auto loop = [&](auto mode) {
        for (;;) {
            const int32_t cn = c + W;
            const bool more = cn < g.nchunks;
            if (more) small_load<K>(g, sem, cn, lane, na, nb, nxt);
            if (cn + W < g.nchunks) {
                na = __ldg(g.chunk_row + cn + W);
                nb = __ldg(g.chunk_row + cn + W + 1);
            }
            small_chunk<K, SEM, decltype(mode)::value>(g, sem, part, c, lane, cur, *rows, sx, first);
            if (!more) break;
            c = cn;
            cur = nxt;
        }
    };
    if constexpr (MODE == kSmSegsLive) {  // a loop for each, so that the dense levels pay for no test
        if (filter) loop(std::integral_constant<int, kSmSegsLive>());
        else loop(std::integral_constant<int, kSmSegs>());
    } else {
        loop(std::integral_constant<int, MODE>());
    }
}

// ---------------------------------------------------------------------------
// row-lane chunk kernel: the value schemes at k = 16 and 32, the 64-lane OR at
// k = 8.  Few of a tile's rows hold a bit there, and k accumulators a lane are
// too many to join across lanes, so the lanes of a warp are the rows: lane l
// takes row l % k of every (32/k)-th tile, one accumulator, and a tile-row's
// end joins the 32/k lanes of a row by at most two shuffles and stores k
// neighbouring values.  A step is 32/k tiles; the tiles and columns of a
// segment (2 KB of tiles) are copied to shared memory asynchronously, where a
// step's rows are 32 neighbouring bytes, half-words or words.  Steps go in
// groups of four, whose first gathers are in flight together (most rows of a
// tile hold one bit; the others loop).
// R-MAT 20, k = 32, plus-times: 2034 us with k accumulators a lane, 661 here
// (k = 16: 654, 439); bound by latency and instructions (2.1 an SM a cycle,
// DRAM 37%, L1 25%), so the registers are cut to 40 for six blocks an SM (four
// with 16-byte values, which spill then): 638 us before the sums were
// compensated, against 738 with four blocks and groups of eight, whose gathers
// in flight a warp are twice as many.  The compensation costs 2 to 4% (four
// columns 10%) and takes the error below that of the k accumulators (relative
// to a 64-bit sum, root mean square 2.0e-8 against 2.1e-8 on R-MAT 20, 2.8e-8
// against 3.3e-8 on 3607 vertices; without it 2.2e-8 and 3.8e-8).
// ---------------------------------------------------------------------------
template <int K>
struct RowLaneShape {
    static constexpr int SUBS = 32 / K;                            // tiles a step
    static constexpr int SEG = 2048 / ChunkShape<K>::TB;           // tiles a segment: 256, 64, 16
    static constexpr int STEPS = SEG / SUBS;                       // 64, 32, 16
    static constexpr int SEGS = ChunkShape<K>::CT / SEG;           // segments a chunk: 1, 2, 4
    static constexpr int GRP = 4;                                  // steps a group
};

template <int K>
struct RowLaneSegment {
    __align__(16) uint8_t tiles[2048];
    __align__(16) int32_t col[RowLaneShape<K>::SEG];
};

__device__ __forceinline__ void cp_async_stream16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// Copies the segment from tile t0 (the arrays are padded to whole chunks).
template <int K>
__device__ __forceinline__ void rowlane_copy(const SpmvGeom& g, int64_t t0, int lane, RowLaneSegment<K>& s) {
    const uint8_t* src = g.tiles + t0 * ChunkShape<K>::TB;
#pragma unroll
    for (int j = 0; j < 4; ++j) cp_async_stream16(s.tiles + 512 * j + 16 * lane, src + 512 * j + 16 * lane);
    constexpr int PIECES = RowLaneShape<K>::SEG / 4;
#pragma unroll
    for (int j = 0; j < PIECES; j += 32)
        if (j + lane < PIECES) cp_async_stream16(s.col + 4 * (j + lane), g.colind + t0 + 4 * (j + lane));
    cp_async_commit();
}

// Joins the lanes of a row (lanes l, l + k, ...), earlier tiles first.
template <int K, class SEM>
__device__ __forceinline__ typename SEM::V rowlane_join(const SEM& sem, typename SEM::V v, int lane) {
#pragma unroll
    for (int d = K; d < 32; d <<= 1) {
        const typename SEM::V o = shfl_xor(v, d);
        v = (lane & d) ? sem.comb(o, v) : sem.comb(v, o);
    }
    return v;
}

// A lane's running value of its row.  fp32 sums are compensated, as a lane's
// chain is as long as its tile-row.
template <class SEM, class J>
struct RowLaneAcc {
    typename SEM::V a;
    __device__ __forceinline__ void clear(const SEM& sem) { a = sem.ident(); }
    __device__ __forceinline__ void add(const SEM& sem, typename SEM::V v) { a = sem.comb(a, v); }
    __device__ __forceinline__ typename SEM::V value() const { return a; }
};
__device__ __forceinline__ void csum_push(CSum& a, float v) {
    const float t = __fadd_rn(a.s, v);
    const float bp = __fsub_rn(t, a.s);
    a.c = __fadd_rn(a.c, __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(v, bp)));
    a.s = t;
}
template <class SEM>
struct RowLaneAcc<SEM, CSum> {
    CSum a;
    __device__ __forceinline__ void clear(const SEM&) { a = CSum(0.0f); }
    __device__ __forceinline__ void add(const SEM&, float v) { csum_push(a, v); }
    __device__ __forceinline__ float value() const { return (float)a; }
};
template <class SEM>
struct RowLaneAcc<SEM, CSum4> {
    CSum4 a;
    __device__ __forceinline__ void clear(const SEM& sem) { a = CSum4(sem.ident()); }
    __device__ __forceinline__ void add(const SEM&, float4 v) {
        csum_push(a.v[0], v.x);
        csum_push(a.v[1], v.y);
        csum_push(a.v[2], v.z);
        csum_push(a.v[3], v.w);
    }
    __device__ __forceinline__ float4 value() const { return (float4)a; }
};

template <int K, class SEM>
__device__ __forceinline__ void rowlane_body(const SpmvGeom& g, const SEM& sem, Partials<typename SEM::V> part) {
    using S = RowLaneShape<K>;
    using V = typename SEM::V;
    using G = typename SEM::G;
    using Rows = typename std::conditional<K == 8, uint8_t, typename std::conditional<K == 16, uint16_t, uint32_t>::type>::type;
    constexpr int CT = ChunkShape<K>::CT;
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int GRP = RowLaneShape<K>::GRP;
    static_assert(GRP == 4, "the group's tiles are added in pairs");
    __shared__ ChunkRows rows[kSpmvWarps];
    __shared__ RowLaneSegment<K> segs[kSpmvWarps];
    if (gated_off(g.gate)) return;
    ChunkRows& cr = rows[threadIdx.x >> 5];
    RowLaneSegment<K>& seg = segs[threadIdx.x >> 5];
    const Rows* bits = reinterpret_cast<const Rows*>(seg.tiles);
    const int lane = (int)lane_id();
    const int r = lane % K, sub = lane / K;
    const int32_t W = (int32_t)gridDim.x * kSpmvWarps;
    RegAcc<V, SEM::NV> idv;
#pragma unroll
    for (int v = 0; v < SEM::NV; ++v) idv.set(v, sem.ident());
    for (int32_t c = (int32_t)blockIdx.x * kSpmvWarps + (threadIdx.x >> 5); c < g.nchunks; c += W) {
        const int32_t ra = __ldg(g.chunk_row + c), rb = __ldg(g.chunk_row + c + 1);
        const int32_t cs = c * CT, ce = cs + min(CT, (int32_t)g.T - cs);
        const bool skip = sem.saturated((int64_t)ra * K, ((int64_t)rb + 1) * K);  // every row masked out
        if (!skip) rowlane_copy<K>(g, cs, lane, seg);
        const int32_t win = row_window(g, ra, rb - ra, lane);
        const bool one_row = ra == rb;
        const bool head = __shfl_sync(FULL, win, 0) == cs;  // tile-row ra begins with this chunk
        if (!one_row) chunk_ends(g, sem, ra, rb, win, cs, ce, lane, idv, cr);
        RowLaneAcc<SEM, typename SEM::J> acc;
        acc.clear(sem);
        int rank = 0;  // row ends so far
        // the row that ends here: stored, or the chunk's first partial
        auto end_row = [&]() {
            const V v = rowlane_join<K>(sem, acc.value(), lane);
            if (lane < K) {
                if (rank > 0 || head) sem.store_row(cr.row[rank], lane, v);
                else part.val_first[(int64_t)c * K + lane] = v;
            }
            ++rank;
            acc.clear(sem);
        };
#pragma unroll 1
        for (int q = 0; q < S::SEGS; ++q) {
            if (!skip) {
                cp_async_wait_all();
                __syncwarp();
            }
#pragma unroll 1
            for (int i0 = 0; i0 < S::STEPS; i0 += GRP) {
                uint32_t b[GRP];
                int32_t at[GRP];  // first input value under the tile
                int32_t wat[GRP];
                G x[GRP];
                float wv[GRP];
#pragma unroll
                for (int i = 0; i < GRP; ++i) {
                    const int tile = (i0 + i) * S::SUBS + sub;  // in the segment
                    b[i] = skip ? 0u : (uint32_t)bits[(i0 + i) * 32 + lane];
                    at[i] = (skip ? 0 : seg.col[tile]) * K;
                    wat[i] = 0;
                    wv[i] = 1.0f;
                    if constexpr (SEM::kMayWeight) {
                        if (sem.weighted) {  // the tile's bits in earlier rows, then the row's own
                            int before = __popc(b[i]);
#pragma unroll
                            for (int d = 1; d < K; d <<= 1) {
                                const int o = __shfl_up_sync(FULL, before, d, K);
                                if (r >= d) before += o;
                            }
                            const int32_t t = cs + min(q * S::SEG + tile, (int32_t)g.T - 1 - cs);
                            wat[i] = __ldg(sem.voffs() + t) + (before - __popc(b[i]));
                        }
                    }
                    if (b[i]) {
                        x[i] = __ldg(sem.src() + (at[i] + __ffs(b[i]) - 1));
                        if constexpr (SEM::kMayWeight)
                            if (sem.weighted) wv[i] = __ldg(sem.wts() + wat[i]);
                    }
                }
                const int t0 = q * S::SEG + i0 * S::SUBS;  // the group's first tile in the chunk
                uint32_t ends = 0u;                          // row ends among its tiles
                if (!one_row)
                    ends = (cr.mask[t0 >> 5] >> (t0 & 31)) & (GRP * S::SUBS == 32 ? FULL : (1u << (GRP * S::SUBS % 32)) - 1u);
                // the lane's row of a tile: its first bit's value, then the others'
                auto tile_sum = [&](int i) {
                    V v = sem.ident();
                    if (b[i] == 0u) return v;
                    v = sem.apply(v, x[i], wv[i]);
                    for (uint32_t more = b[i] & (b[i] - 1u); more; more &= more - 1u) {
                        float w2 = 1.0f;
                        if constexpr (SEM::kMayWeight)
                            if (sem.weighted) w2 = __ldg(sem.wts() + ++wat[i]);
                        v = sem.apply(v, __ldg(sem.src() + (at[i] + __ffs(more) - 1)), w2);
                    }
                    return v;
                };
                if (ends == 0u) {  // warp-uniform
                    const V v = sem.comb(tile_sum(0), tile_sum(1));
                    acc.add(sem, sem.comb(v, sem.comb(tile_sum(2), tile_sum(3))));
                } else {
                    // tile by tile: a lane adds its row of a tile before that
                    // tile's end and after the ends of earlier ones
#pragma unroll
                    for (int i = 0; i < GRP; ++i) {
                        const V v = tile_sum(i);
#pragma unroll
                        for (int u = 0; u < S::SUBS; ++u) {
                            if (sub == u) acc.add(sem, v);
                            if ((ends >> (i * S::SUBS + u)) & 1u) end_row();
                        }
                    }
                }
            }
            __syncwarp();  // every lane has read the segment
            if (q + 1 < S::SEGS && !skip) rowlane_copy<K>(g, (int64_t)cs + (q + 1) * S::SEG, lane, seg);
        }
        // the open row: all of a chunk inside one row, or the tail
        const bool open = one_row || !((cr.mask[(ce - 1 - cs) >> 5] >> ((ce - 1 - cs) & 31)) & 1u);
        if (open) {
            const V v = rowlane_join<K>(sem, acc.value(), lane);
            if (lane < K) {
                if (one_row && c + 1 == g.nchunks && head) sem.store_row(ra, lane, v);
                else if (one_row && !head) part.val_first[(int64_t)c * K + lane] = v;
                else part.val_last[(int64_t)c * K + lane] = v;
            }
        }
    }
}

// k = 4 with the bit-vector schemes and 4-byte values; the other small-tile
// cases (k = 8, 8-byte values).
template <class SEM, int MODE>
__global__ void __launch_bounds__((small_threads<4, SEM, MODE>()), (small_min_blocks<4, SEM, MODE>()))
    spmv_k4_kernel(SpmvGeom g, SEM sem, Partials<typename SEM::V> part) {
    small_body<4, SEM, MODE>(g, sem, part);
}
template <int K, class SEM, int MODE>
__global__ void __launch_bounds__((small_threads<K, SEM, MODE>()), (small_min_blocks<K, SEM, MODE>()))
    spmv_chunks_kernel(SpmvGeom g, SEM sem, Partials<typename SEM::V> part) {
    if constexpr (MODE == kRowLanes) rowlane_body<K, SEM>(g, sem, part);
    else small_body<K, SEM, MODE>(g, sem, part);
}

// ---------------------------------------------------------------------------
// chunk kernel for the value schemes at k <= 16.  Pass 1: each lane walks
// the set bits of its tiles in one flat loop (tile words copied to lane-private
// shared memory so a running word index can address them) and issues one
// cp.async gather per bit, so a warp's input values are all in flight at once;
// each staged value is tagged with its (tile, row).  Pass 2: a second flat
// loop over the tags adds each value to its row's register accumulator (a
// predicated select over the k rows keeps every register index static) and
// closes tiles as the walk passes them.  Lanes with fewer set bits finish
// early instead of idling through per-word loops.
// ---------------------------------------------------------------------------
// Resident blocks the gather kernel is compiled for: wide (16-byte) values
// need the registers of two blocks per SM rather than three.
template <int K, class SEM>
constexpr int gather_min_blocks() {
    return (K >= 16 || sizeof(typename SEM::V) > 8) ? 2 : 3;
}

template <int K, class SEM>
__global__ void __launch_bounds__(kSpmvThreads, (gather_min_blocks<K, SEM>())) spmv_gather_kernel(SpmvGeom g, SEM sem,
                                                                   Partials<typename SEM::V> part) {
    using S = ChunkShape<K>;
    using V = typename SEM::V;
    using G = typename SEM::G;
    using L = GatherLayout<K, SEM>;
    constexpr int NV = SEM::NV;
    constexpr int P = S::P;
    constexpr int TW = S::TW;
    constexpr int RB = S::ROW_BITS;
    constexpr int RPW = 32 / RB;  // rows per 32-bit word
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) uint8_t smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    const int32_t c = (int32_t)blockIdx.x * kSpmvWarps + warp;
    if (c >= g.nchunks || gated_off(g.gate)) return;  // whole warps leave together

    uint8_t* wsm = smem + warp * L::bytes;
    // lane-interleaved (element e of lane l at [e * 32 + l]): conflict-free
    uint32_t* swords = reinterpret_cast<uint32_t*>(wsm + L::words_off) + lane;
    int32_t* scol = reinterpret_cast<int32_t*>(wsm + L::col_off) + lane;
    G* sx = reinterpret_cast<G*>(wsm + L::x_off);
    float* sw = reinterpret_cast<float*>(wsm + L::w_off);
    uint8_t* stag = wsm + L::tag_off;

    LaneSpan ls;
    ls.cs = c * S::CT;
    ls.ce = min(ls.cs + S::CT, (int32_t)g.T);
    ls.tl = ls.cs + lane * P;
    ls.cnt = max(0, min(P, ls.ce - ls.tl));

    uint4 tv[S::TILE_V4];
    int32_t col[P];
    // a chunk whose every output row is masked out reads no tiles (zero words:
    // the walk still stores its rows and partials, all the identity)
    bool sat = false;
    {
        const int32_t ra = __ldg(g.chunk_row + c), rb = __ldg(g.chunk_row + c + 1);
        sat = sem.saturated((int64_t)ra * K, ((int64_t)rb + 1) * K);
    }
    if (!sat) {
        load_lane_tiles<K>(g, ls.tl, tv, col);
    } else {
#pragma unroll
        for (int q = 0; q < S::TILE_V4; ++q) tv[q] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int i = 0; i < P; ++i) col[i] = 0;
    }
    const uint32_t* words = reinterpret_cast<const uint32_t*>(tv);

    // set bits of the lane's tiles and their slots in the warp's staging area
    int nb = 0;
#pragma unroll
    for (int i = 0; i < P; ++i)
        if (i < ls.cnt) {
#pragma unroll
            for (int q = 0; q < TW; ++q) nb += __popc(words[i * TW + q]);
        }
    int incl = nb;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += o;
    }
    const int gbase = incl - nb;
    const int nbits = __shfl_sync(FULL, incl, 31);
    const bool staged = nbits <= L::NG;  // warp-uniform

    if (staged) {
        // first staging slot of each of the lane's tiles
        int32_t* spre = reinterpret_cast<int32_t*>(wsm + L::pre_off) + lane;
        int run = gbase;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            spre[i * 32] = run;
            if (i < ls.cnt) {
#pragma unroll
                for (int q = 0; q < TW; ++q) run += __popc(words[i * TW + q]);
            }
        }
#pragma unroll
        for (int q = 0; q < P * TW; ++q) swords[q * 32] = words[q];
#pragma unroll
        for (int i = 0; i < P; ++i) scol[i * 32] = col[i];
        int wi = 0;
        uint32_t cur = words[0];
        int ti = -1, qb = 0;
        const G* xt = nullptr;
        const float* wt = nullptr;
        for (int j = 0; j < nb; ++j) {
            while (cur == 0u) cur = swords[(++wi) * 32];
            const int bit = __ffs(cur) - 1;
            cur &= cur - 1;
            const int i = wi / TW;
            if (i != ti) {  // first set bit of tile i
                ti = i;
                qb = 0;
                xt = sem.src() + (int64_t)scol[i * 32] * K;
                if (sem.weighted) wt = sem.wts() + __ldg(sem.voffs() + ls.tl + i);
            }
            const int s = gbase + j;
            cp_async_gather<sizeof(G)>(sx + s, xt + bit % RB);
            if (sem.weighted) cp_async_gather<4>(sw + s, wt + qb);
            stag[s] = (uint8_t)(wi * RPW + bit / RB);  // = i * K + (wi % TW) * RPW + row in word
            ++qb;
        }
        cp_async_commit();
    }

    RegAcc<V, NV> idv;
#pragma unroll
    for (int v = 0; v < NV; ++v) idv.set(v, sem.ident());

    // ---- fast path: a staged chunk spanning at most four tile-rows.  Each
    // tile-row's staged values (contiguous slots, tile order) are dealt to
    // the lanes round-robin, summed in registers, and joined by a fixed
    // butterfly, so no lane waits on another's bit count.
    {
        const int32_t r0 = __ldg(g.chunk_row + c);
        const int32_t span = __ldg(g.chunk_row + c + 1) - r0;
        if (staged && span <= 3) {
            const int32_t win = lane <= span + 1 ? __ldg(g.rowptr + r0 + lane) : INT32_MAX;
            cp_async_wait_all();
            __syncwarp();  // values, tags and slot starts of every lane are visible
            const int32_t* pre = reinterpret_cast<const int32_t*>(wsm + L::pre_off);
            auto slot_of = [&](int32_t t) -> int {  // first slot of chunk tile t (nbits at the chunk end)
                if (t >= ls.ce) return nbits;
                const int32_t o = t - ls.cs;
                return pre[(o % P) * 32 + (o / P)];
            };
            const int32_t a0 = __shfl_sync(FULL, win, 0);
            if (lane == 0 && a0 == ls.cs && ls.cs > 0)  // empty rows just before the chunk's first tile-row
                for (int32_t R = r0 - 1; R >= 0 && __ldg(g.rowptr + R) == ls.cs; --R) sem.store(R, idv);
            for (int j = 0; j <= span; ++j) {
                const int32_t R = r0 + j;
                const int32_t a = __shfl_sync(FULL, win, j), b = __shfl_sync(FULL, win, j + 1);
                if (a == b) {  // empty tile-row inside the chunk's range
                    if (lane == 0 && a >= ls.cs && a < ls.ce && a > 0) sem.store(R, idv);
                    continue;
                }
                const int32_t ts = max(a, ls.cs), te = min(b, ls.ce);
                if (ts >= te) continue;  // its tiles lie outside this chunk
                const int s0 = slot_of(ts), s1 = slot_of(te);
                RegAcc<V, NV> acc;
#pragma unroll
                for (int v = 0; v < NV; ++v) acc.set(v, sem.ident());
                for (int sidx = s0 + lane; sidx < s1; sidx += 32) {
                    const int r = stag[sidx] % K;
                    const V cv = sem.contrib(sx[sidx], sem.weighted ? sw[sidx] : 1.0f);
#pragma unroll
                    for (int u = 0; u < K; ++u) acc.set(u, sem.comb(acc.get(u), r == u ? cv : sem.ident()));
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const V other = shfl_xor(acc.get(v), o);
                        acc.set(v, (lane & o) ? sem.comb(other, acc.get(v)) : sem.comb(acc.get(v), other));
                    }
                }
                if (lane < K) {  // every lane holds the totals: lane r writes row r
                    V v = acc.get(0);
#pragma unroll
                    for (int u = 1; u < K; ++u) v = lane == u ? acc.get(u) : v;
                    const bool started = a >= ls.cs, ended = b <= ls.ce;
                    if (started && ended) sem.store_row(R, lane, v);
                    else if (!started) part.val_first[c * NV + lane] = v;
                    else part.val_last[c * NV + lane] = v;
                }
            }
            return;
        }
    }

    const RowCursor rc = locate_row(g, c, ls, lane);
    RegAcc<V, NV> acc, F;
#pragma unroll
    for (int v = 0; v < NV; ++v) { acc.set(v, sem.ident()); F.set(v, sem.ident()); }
    Walk<SEM, RegAcc<V, NV>> wk;
    wk.row = rc.row;
    wk.next = rc.next;
    if (staged) cp_async_wait_all();  // each lane reads back only the slots it filled

    if (ls.cnt > 0) {
        // empty tile-rows just before a row that starts at this lane's first tile
        if (ls.tl > 0 && rc.row_start == ls.tl)
            for (int32_t R = rc.row - 1; R >= 0 && __ldg(g.rowptr + R) == ls.tl; --R) sem.store(R, idv);
        if (staged) {
            int i = 0;
            for (int j = 0; j < nb; ++j) {
                const int s = gbase + j;
                const int tag = stag[s];
                const int ti = tag / K;
                while (i < ti) {  // every tile has a set bit: the walk passes tile i
                    wk.end_tile(g, sem, acc, F, ls.tl + i, i, ls.cnt, idv);
                    ++i;
                }
                const int r = tag % K;
                const V cv = sem.contrib(sx[s], sem.weighted ? sw[s] : 1.0f);
                // branch-free row select: every row combines either the
                // contribution or the identity
#pragma unroll
                for (int u = 0; u < K; ++u) acc.set(u, sem.comb(acc.get(u), r == u ? cv : sem.ident()));
            }
            for (; i < ls.cnt; ++i) wk.end_tile(g, sem, acc, F, ls.tl + i, i, ls.cnt, idv);
        } else {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                if (i < ls.cnt) {
                    const int32_t t = ls.tl + i;
                    const G* xt = sem.src() + (int64_t)col[i] * K;
                    const float* wt = sem.weighted ? sem.wts() + __ldg(sem.voffs() + t) : nullptr;
                    int qb = 0;
#pragma unroll
                    for (int q = 0; q < TW; ++q) {
                        uint32_t b = words[i * TW + q];
                        while (b) {
                            const int bit = __ffs(b) - 1;
                            b &= b - 1;
                            const V cv = sem.contrib(__ldg(xt + bit % RB), sem.weighted ? __ldg(wt + qb) : 1.0f);
                            const int u = bit / RB;
#pragma unroll
                            for (int uu = 0; uu < RPW; ++uu)
                                acc.set(q * RPW + uu, sem.comb(acc.get(q * RPW + uu), u == uu ? cv : sem.ident()));
                            ++qb;
                        }
                    }
                    wk.end_tile(g, sem, acc, F, t, i, ls.cnt, idv);
                }
            }
        }
    }
    close_chunk(sem, part, c, ls, lane, rc.head_cs, rc.row, wk.has_end, wk.open, acc, F, P);
}

// Rows that span chunks, from the handle's split list of (row, first chunk,
// last chunk): the row's partials are the first chunk's val_last and every
// later chunk's val_first, joined in chunk order.  Blocks [0, short_blocks)
// give one thread to each row spanning at most kSplitShort chunks; the
// remaining blocks give a warp to each longer row (lane l folds every 32nd
// partial in order, then a fixed butterfly joins the lanes).
template <int K, class SEM>
__global__ void spmv_fixup_kernel(const int32_t* __restrict__ split, const int32_t* __restrict__ split_long,
                                  int64_t nshort, int64_t nlong, int64_t short_blocks, int64_t long_blocks,
                                  int32_t lead_end, int32_t trail_begin, int32_t ntr, SEM sem, Partials<typename SEM::V> part,
                                  const int32_t* gate) {
    using V = typename SEM::V;
    using J = typename SEM::J;
    constexpr int NV = SEM::NV;
    if (gated_off(gate)) return;
    if ((int64_t)blockIdx.x >= short_blocks + long_blocks) {  // rows outside the tiles: the identity
        RegAcc<V, NV> idv;
#pragma unroll
        for (int v = 0; v < NV; ++v) idv.set(v, sem.ident());
        const int64_t first = short_blocks + long_blocks;
        const int64_t stride = ((int64_t)gridDim.x - first) * blockDim.x;
        const int64_t tid = ((int64_t)blockIdx.x - first) * blockDim.x + threadIdx.x;
        for (int64_t R = tid; R < lead_end; R += stride) sem.store((int32_t)R, idv);
        for (int64_t R = trail_begin + tid; R < ntr; R += stride) sem.store((int32_t)R, idv);
        return;
    }
    if ((int64_t)blockIdx.x < short_blocks) {
        if constexpr (SEM::kGather) {
            // value schemes: a thread per (row, value); the NV threads of a
            // row read each partial's NV values side by side
            const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
            const int64_t e = tid / NV;
            const int v = (int)(tid % NV);
            if (e >= nshort) return;
            const int32_t R = split[3 * e], ca = split[3 * e + 1], cb = split[3 * e + 2];
            J acc = (J)part.val_last[(int64_t)ca * NV + v];
            for (int64_t q = ca + 1; q <= cb; ++q) acc = sem.jcomb(acc, (J)part.val_first[q * NV + v]);
            sem.store_row(R, v, (V)acc);
            return;
        }
        const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (e >= nshort) return;
        const int32_t R = split[3 * e], ca = split[3 * e + 1], cb = split[3 * e + 2];
        J acc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = (J)part.val_last[(int64_t)ca * NV + v];
        for (int64_t q = ca + 1; q <= cb; ++q) {
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = sem.jcomb(acc[v], (J)part.val_first[q * NV + v]);
        }
        RegAcc<V, NV> out;
#pragma unroll
        for (int v = 0; v < NV; ++v) out.set(v, (V)acc[v]);
        sem.store(R, out);
        return;
    }
    const int lane = (int)lane_id();
    const int64_t e = ((int64_t)(blockIdx.x - short_blocks) * blockDim.x + threadIdx.x) / 32;
    if (e >= nlong) return;  // whole warps leave together
    const int32_t R = split_long[3 * e], ca = split_long[3 * e + 1], cb = split_long[3 * e + 2];
    const int64_t np = (int64_t)cb - ca + 1;
    J acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = (J)sem.ident();
    for (int64_t p = lane; p < np; p += 32) {
        const V* src = p == 0 ? part.val_last + (int64_t)ca * NV : part.val_first + (ca + p) * NV;
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = sem.jcomb(acc[v], (J)src[v]);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const J other = shfl_xor(acc[v], o);
            acc[v] = (lane & o) ? sem.jcomb(other, acc[v]) : sem.jcomb(acc[v], other);
        }
    }
    if (lane == 0) {
        RegAcc<V, NV> out;
#pragma unroll
        for (int v = 0; v < NV; ++v) out.set(v, (V)acc[v]);
        sem.store(R, out);
    }
}

// The join, and with `edges` the tile-rows before the first tile and after the
// last one (every row when the matrix has no tiles), which get the identity.
template <int K, class SEM>
static b2sr_status launch_fixup(const b2sr_matrix* h, const SEM& sem, Partials<typename SEM::V> part,
                                cudaStream_t s, const int32_t* gate, bool edges) {
    const int32_t lead_end = h->T == 0 ? h->ntr : h->first_row;
    const int32_t trail_begin = h->T == 0 ? h->ntr : h->last_row + 1;
    const int64_t outside = edges ? (int64_t)lead_end + (h->ntr - trail_begin) : 0;
    const int64_t short_blocks = ceil_div(h->nsplit_short * (SEM::kGather ? SEM::NV : 1), 256);
    const int64_t long_blocks = ceil_div(h->nsplit_long, 8);
    const int64_t edge_blocks = std::min<int64_t>(ceil_div(outside, 256), (int64_t)sm_count() * 4);
    if (short_blocks + long_blocks + edge_blocks == 0) return B2SR_OK;
    spmv_fixup_kernel<K, SEM><<<(unsigned)(short_blocks + long_blocks + edge_blocks), 256, 0, s>>>(
        h->split, h->split + 3 * (h->nchunks - h->nsplit_long), h->nsplit_short, h->nsplit_long, short_blocks,
        long_blocks, lead_end, trail_begin, h->ntr, sem, part, gate);
    B2SR_LAUNCH_CHECK("spmv_fixup_kernel");
    return B2SR_OK;
}

// semirings whose result includes the diagonal's self term (min-plus)
template <class S, class = void>
struct HasSelfTerm : std::false_type {};
template <class S>
struct HasSelfTerm<S, std::void_t<decltype(S::kSelfTerm)>> : std::bool_constant<S::kSelfTerm> {};

template <class T>
__device__ __forceinline__ T min_self(T a, T b) {
    if constexpr (std::is_same<T, float>::value) return fminf(a, b);
    else return min(a, b);
}

// y_i = min(x_i, y_i) on the rows the mask keeps (the min-plus self term)
template <class SEM>
__global__ void spmv_self_kernel(SEM sem, const int32_t* gate) {
    if (gated_off(gate)) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < sem.n; i += (int64_t)gridDim.x * blockDim.x)
        if (mask_allows(sem.mask, sem.comp, i)) sem.y[i] = min_self(sem.y[i], __ldg(sem.x + i));
}

__global__ void clear_words_kernel(uint32_t* w, int64_t count, const int32_t* gate) {
    if (gated_off(gate)) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        w[i] = 0u;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Bitset outputs: bits past the last tile-row (>= nTileRow*k) are never
// stored by a row, so the words holding them are cleared first.
template <int K>
static b2sr_status clear_bitset_tail(const b2sr_matrix* h, uint32_t* bits, cudaStream_t s, const int32_t* gate) {
    int64_t words = ceil_div(h->n, 32);
    int64_t first = ((int64_t)h->ntr * K) / 32;
    if (first >= words) return B2SR_OK;
    if (!gate) {
        B2SR_CUDA_TRY(cudaMemsetAsync(bits + first, 0, (words - first) * sizeof(uint32_t), s));
        return B2SR_OK;
    }
    // gated: a closed gate must leave the output alone (the caller may have filled it another way)
    clear_words_kernel<<<1, 32, 0, s>>>(bits + first, words - first, gate);
    B2SR_LAUNCH_CHECK("clear_words_kernel");
    return B2SR_OK;
}

// Clears the whole bitset (schemes that OR into it).
static b2sr_status clear_bitset(const b2sr_matrix* h, uint32_t* bits, cudaStream_t s, const int32_t* gate) {
    const int64_t words = ceil_div(h->n, 32);
    if (words == 0) return B2SR_OK;
    if (!gate) {
        B2SR_CUDA_TRY(cudaMemsetAsync(bits, 0, words * sizeof(uint32_t), s));
        return B2SR_OK;
    }
    clear_words_kernel<<<grid_for(words), 256, 0, s>>>(bits, words, gate);
    B2SR_LAUNCH_CHECK("clear_words_kernel");
    return B2SR_OK;
}

template <class V, int NV>
static b2sr_status alloc_partials(DevBuf& pbuf, int64_t nchunks, void* scratch, Partials<V>* part) {
    const size_t vbytes = round_up((size_t)nchunks * NV * sizeof(V), 16);
    if (!scratch) B2SR_TRY(pbuf.alloc(2 * vbytes));
    uint8_t* base = scratch ? static_cast<uint8_t*>(scratch) : pbuf.as<uint8_t>();
    part->val_first = reinterpret_cast<V*>(base);
    part->val_last = reinterpret_cast<V*>(base + vbytes);
    return B2SR_OK;
}

// Algorithmic bytes of one SpMV: the three B2SR arrays once, plus the
// vectors each scheme reads and writes once.
static double spmv_bytes(const b2sr_matrix* h, double vec_bytes) {
    return 4.0 * ((double)h->ntr + 1.0) + (double)h->T * (4.0 + tile_bytes(h->k)) + vec_bytes;
}

// The small-tile kernel serves the bit-vector schemes at k = 4 and 8 and the
// unweighted value schemes with 4- and 8-byte values at k = 4.
template <int K, class SEM>
constexpr bool use_small() {
    if constexpr (!SEM::kGather) return K <= 8;
    else return K == 4 && !SEM::kMayWeight;
}

// The row-lane kernel serves the value schemes at k = 32, the unweighted ones
// at k = 16 and the 64-lane OR at k = 8.  us, the better of the staged and the
// general direct kernel / this one:
//   R-MAT 20 and its permutation   k = 8       k = 16                k = 32
//   plus-times               298, 230 / 285, 322   654, 622 / 439, 601     2034, 2516 / 661, 1147
//   64-lane OR               454, 390 / 328, 355   937, 815 / 482, 641     2853, 3696 / 729, 1239
//   four columns             650, 576 / 764, 935   1520, 1393 / 689, 911   5742, 6941 / 1257, 1968
//   weighted min-plus        377, 294 / 592, 657   860, 748 / 895, 1250    2358, 2873 / 1360, 2459
// The bits before a row, which a weight's place needs, cost a scan of the
// tile; at k = 8 a step of four tiles mostly holds fewer set bits than lanes.
// A tile-row that holds a quarter of the matrix and more keeps the other kernels:
// its tiles are full rows of one vertex, which one lane walks alone while 31
// wait (star of 2^20 leaves, k = 32 / 16 / 64-lane OR at k = 8: 177 / 97 / 73 us,
// 65 / 51 / 54 in the others).
enum { kRowLanesNever, kRowLanesUnweighted, kRowLanesAlways };
template <int K, class SEM>
constexpr int row_lanes() {
    if constexpr (!SEM::kGather || K < 8) return kRowLanesNever;
    else if constexpr (K == 8) return LaneWords<SEM>::value && sizeof(typename SEM::V) == 8 ? kRowLanesAlways : kRowLanesNever;
    else return K == 16 && SEM::kMayWeight ? kRowLanesUnweighted : kRowLanesAlways;
}
template <int K, class SEM>
static bool use_row_lanes(const b2sr_matrix* h, const SEM& sem) {
    if (4 * h->most_tiles > h->T) return false;
    if constexpr (row_lanes<K, SEM>() == kRowLanesUnweighted) return !sem.weighted;
    else return row_lanes<K, SEM>() == kRowLanesAlways;
}

template <int K, class SEM, int MODE>
static b2sr_status launch_small(const b2sr_matrix* h, const SEM& sem, Partials<typename SEM::V> part, cudaStream_t s,
                                const SpmvGeom& g) {
    // persistent: the resident blocks, each warp looping over chunks
    constexpr int threads = small_threads<K, SEM, MODE>();
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(h->nchunks, threads / 32),
                                                      (int64_t)sm_count() * small_min_blocks<K, SEM, MODE>());
    const int smem = threads / 32 * small_warp_smem<SEM>() +
                     (MODE == kSmBitsShared ? (int)ceil_div(h->n, 32) * 4
                                            : (MODE == kSmSegsLive ? (int)ceil_div(h->ntr, 32) * 4 : 0));
    void (*kernel)(SpmvGeom, SEM, Partials<typename SEM::V>);
    if constexpr (K == 4 && sizeof(typename SEM::V) == 4) kernel = spmv_k4_kernel<SEM, MODE>;
    else kernel = spmv_chunks_kernel<K, SEM, MODE>;
    // A size that goes with the graph is allowed up to the most a block can have,
    // not up to this call's: the limit belongs to the kernel, and another thread's
    // call with a smaller graph must not lower it before a launch.
    constexpr bool sized = MODE == kSmBitsShared || MODE == kSmSegsLive;
    if (sized || smem > 48 * 1024)
        B2SR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           sized ? (int)kMaxBlockSmem : smem));
    kernel<<<grid, threads, smem, s>>>(g, sem, part);
    B2SR_LAUNCH_CHECK("small-tile SpMV kernel");
    return B2SR_OK;
}

// The direct chunk kernel: the small-tile one where it serves, else the
// general one.
template <int K, class SEM>
static b2sr_status launch_direct(const b2sr_matrix* h, const SEM& sem, Partials<typename SEM::V> part,
                                 cudaStream_t s, const SpmvGeom& g) {
    if constexpr (use_small<K, SEM>()) {
        if constexpr (!SEM::kGather) {
            // The bitset of x in shared memory (x gathers at one distinct 128-byte
            // line a cycle were what bound the kernel) when it fits and a warp has a
            // few chunks to spread the copy over: R-MAT 20, k = 4 / k = 8, Boolean:
            // 75 / 74.7 us without, 68 / 72.5 with it; permuted ids 76 / 89 and 67 / 82.
            constexpr int threads = small_threads<K, SEM, kSmBitsShared>();
            // Counts at k = 8 of a large matrix without a chunk inside one tile-row:
            // the eight counts a row cost the walk more than the shared bitset saves
            // (uniform random graph of 2^20 vertices, 127 tiles a row: 118 us, 108 in the
            // general kernel; R-MAT 20: 142, 161).
            if constexpr (K == 8 && SEM::NV == 8 && !NoInput<SEM>::value)
                if (h->most_tiles <= chunk_tiles(K) && h->T >= h->ntr && h->nchunks >= 2048) {
                    spmv_chunks_kernel<K, SEM>
                        <<<(unsigned)ceil_div(h->nchunks, kSpmvWarps), kSpmvThreads, 0, s>>>(g, sem, part);
                    B2SR_LAUNCH_CHECK("spmv_chunks_kernel");
                    return B2SR_OK;
                }
            if constexpr (!NoInput<SEM>::value)
                if (h->nchunks >= (int64_t)sm_count() * (threads / 32) * 4 &&
                    ceil_div(h->n, 32) * 4 + threads / 32 * small_warp_smem<SEM>() <= kMaxBlockSmem)
                    return launch_small<K, SEM, kSmBitsShared>(h, sem, part, s, g);
            return launch_small<K, SEM, kSmBits>(h, sem, part, s, g);
        } else {
            using G = typename SEM::G;
            if constexpr (sizeof(G) == 16) {
                // R-MAT 20 (1.15 set bits a tile), its permutation (1.01), R-MAT 16
                // (1.3), us: by column 224 / 241 / 27, by bit 237 / 195 / 47
                if (8 * h->nnz > 9 * h->T) return launch_small<K, SEM, kSmVals>(h, sem, part, s, g);
                return launch_small<K, SEM, kSmEach>(h, sem, part, s, g);
            } else {
                // A batched BFS's frontier: zero segments are not loaded, and chunks
                // without a live one not walked.  R-MAT 20, 16 sources, us a level: the
                // first 66, the dense ones 131 to 164, the last four 53 to 93 (about 130
                // all with every segment loaded); R-MAT 22, 64 sources: 283, 703 to 865,
                // 233 to 354.
                if constexpr (LaneWords<SEM>::value) {
                    constexpr int threads = small_threads<K, SEM, kSmSegsLive>();
                    if (sem.live && h->n % 4 == 0 && reinterpret_cast<uintptr_t>(sem.x) % (4 * sizeof(G)) == 0 &&
                        h->nchunks >= (int64_t)sm_count() * (threads / 32) * 4 &&
                        ceil_div(h->ntr, 32) * 4 + threads / 32 * small_warp_smem<SEM>() <= kMaxBlockSmem)
                        return launch_small<K, SEM, kSmSegsLive>(h, sem, part, s, g);
                }
                // 8-byte values where hardly a tile holds two bits: by bit (64-lane OR,
                // us, segment / bit: permuted R-MAT 20, 1.006 bits a tile, 199 / 182;
                // R-MAT 22, 1.08 bits, 665 / 816)
                if constexpr (sizeof(G) == 8)
                    if (32 * h->nnz <= 33 * h->T) return launch_small<K, SEM, kSmEach>(h, sem, part, s, g);
                // whole segments need an aligned input without a ragged last one
                if (h->n % 4 == 0 && reinterpret_cast<uintptr_t>(sem.x) % (4 * sizeof(G)) == 0)
                    return launch_small<K, SEM, kSmSegs>(h, sem, part, s, g);
                return launch_small<K, SEM, kSmVals>(h, sem, part, s, g);
            }
        }
    } else {
        if constexpr (row_lanes<K, SEM>() != kRowLanesNever) {
            if (use_row_lanes<K>(h, sem)) {
                const unsigned grid =
                    (unsigned)std::min<int64_t>(ceil_div(h->nchunks, kSpmvWarps),
                                                (int64_t)sm_count() * small_min_blocks<K, SEM, kRowLanes>());
                spmv_chunks_kernel<K, SEM, kRowLanes><<<grid, kSpmvThreads, 0, s>>>(g, sem, part);
                B2SR_LAUNCH_CHECK("row-lane SpMV kernel");
                return B2SR_OK;
            }
        }
        spmv_chunks_kernel<K, SEM><<<(unsigned)ceil_div(h->nchunks, kSpmvWarps), kSpmvThreads, 0, s>>>(g, sem, part);
        B2SR_LAUNCH_CHECK("spmv_chunks_kernel");
    }
    return B2SR_OK;
}

// the chunk kernel (staged or direct) and the cross-chunk join
template <int K, class SEM>
static b2sr_status run_chunks(const b2sr_matrix* h, const SEM& sem, cudaStream_t s, const char* family,
                              double vec_bytes, const int32_t* gate, const SpmvGeom& g, void* scratch, bool edges) {
    using V = typename SEM::V;
    DevBuf pbuf(s);
    Partials<V> part{nullptr, nullptr};
    if (!OrsInto<SEM>::value) B2SR_TRY((alloc_partials<V, SEM::NV>(pbuf, h->nchunks, scratch, &part)));
    const unsigned blocks = (unsigned)ceil_div(h->nchunks, kSpmvWarps);
    bool staged = false;
    // AUTO: the small-tile and row-lane kernels where they serve
    if constexpr (SEM::kGather && K <= 16)
        staged = h->schedule == B2SR_SCHED_STAGED ||
                 (h->schedule == B2SR_SCHED_AUTO && !(use_small<K, SEM>() || use_row_lanes<K>(h, sem)));
    if constexpr (SEM::kGather && K <= 16) if (staged) {
        const int smem = kSpmvWarps * GatherLayout<K, SEM>::bytes;
        if (smem > 48 * 1024)
            B2SR_CUDA_TRY(cudaFuncSetAttribute(spmv_gather_kernel<K, SEM>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        void* tok = gate ? nullptr : timing_begin(s);  // a gated launch may do nothing
        spmv_gather_kernel<K, SEM><<<blocks, kSpmvThreads, smem, s>>>(g, sem, part);
        timing_end(tok, family, spmv_bytes(h, vec_bytes), s);
        B2SR_LAUNCH_CHECK("spmv_gather_kernel");
    }
    if (!staged) {
        void* tok = gate ? nullptr : timing_begin(s);  // a gated launch may do nothing
        const b2sr_status st = launch_direct<K, SEM>(h, sem, part, s, g);
        timing_end(tok, family, spmv_bytes(h, vec_bytes), s);
        B2SR_TRY(st);
    }
    if constexpr (OrsInto<SEM>::value) return B2SR_OK;
    else return launch_fixup<K, SEM>(h, sem, part, s, gate, edges);
}

template <int K, class SEM>
static b2sr_status run_spmv(const b2sr_matrix* h, const SEM& sem, uint32_t* bits_out, cudaStream_t s,
                            const char* family, double vec_bytes, const int32_t* gate, bool edges = true,
                            void* scratch = nullptr) {
    SpmvGeom g{h->rowptr, h->colind, h->tiles, h->chunk_row, h->T, h->nchunks, h->ntr, gate};
    if (OrsInto<SEM>::value) {
        if (edges) B2SR_TRY(clear_bitset(h, bits_out, s, gate));
    } else if (edges && bits_out) {
        B2SR_TRY(clear_bitset_tail<K>(h, bits_out, s, gate));
    }
    if (h->nchunks > 0) {
        B2SR_TRY((run_chunks<K, SEM>(h, sem, s, family, vec_bytes, gate, g, scratch, edges)));
    } else if constexpr (!OrsInto<SEM>::value) {
        B2SR_TRY((launch_fixup<K, SEM>(h, sem, Partials<typename SEM::V>{nullptr, nullptr}, s, gate, edges)));
    }
    if constexpr (HasSelfTerm<SEM>::value) {
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(h->n, 256), (int64_t)sm_count() * 8));
        spmv_self_kernel<SEM><<<grid, 256, 0, s>>>(sem, gate);
        B2SR_LAUNCH_CHECK("spmv_self_kernel");
    }
    return B2SR_OK;
}


// Ones per row, and the partial counts of the tile-rows that cross chunks
// (first, last: nchunks * k each): last[c] holds what chunk c has of a row
// continued from it, first[c] what it has of a row begun before it.  cnt is zero
// where a row has no tiles.  chunks_done: all but the join is done.
b2sr_status row_counts(const b2sr_matrix* h, int32_t* cnt, int32_t* first, int32_t* last, bool chunks_done,
                       cudaStream_t s) {
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        using SEM = SemOnes<K>;
        SEM sem;
        sem.x = nullptr;
        sem.y = cnt;
        sem.mask = nullptr;
        sem.comp = 0;
        sem.n = h->n;
        SpmvGeom g{h->rowptr, h->colind, h->tiles, h->chunk_row, h->T, h->nchunks, h->ntr, nullptr};
        const Partials<int32_t> part{first, last};
        if (!chunks_done && h->nchunks > 0) B2SR_TRY((launch_direct<K, SEM>(h, sem, part, s, g)));
        return launch_fixup<K, SEM>(h, sem, part, s, nullptr, false);
    });
}

b2sr_status spmv_dispatch(b2sr_matrix* h, b2sr_semiring sr, b2sr_vec in_kind, const void* x, b2sr_vec out_kind,
                          void* y, const uint32_t* mask, int comp, const float* weights, cudaStream_t s,
                          const int32_t* gate, bool edges) {
    comp = comp ? 1 : 0;
    if (sr == B2SR_BOOL_OR_AND && in_kind == B2SR_VEC_BITS && out_kind == B2SR_VEC_BITS) {
        if (weights) return fail(B2SR_ERR_INVALID_ARG, "weights apply to MIN_PLUS only");
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemBool<K> sem{static_cast<const uint32_t*>(x), static_cast<uint32_t*>(y), mask, comp, h->n};
            return run_spmv<K>(h, sem, static_cast<uint32_t*>(y), s, "spmv_bool", (mask ? 3.0 : 2.0) * h->n / 8.0, gate,
                               edges);
        });
    }
    if (sr == B2SR_PLUS_TIMES && in_kind == B2SR_VEC_BITS && out_kind == B2SR_VEC_I32) {
        if (weights) return fail(B2SR_ERR_INVALID_ARG, "weights apply to MIN_PLUS only");
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemCount<K> sem{static_cast<const uint32_t*>(x), static_cast<int32_t*>(y), mask, comp, h->n};
            return run_spmv<K>(h, sem, nullptr, s, "spmv_count", (mask ? 2.0 : 1.0) * h->n / 8.0 + 4.0 * h->n, gate);
        });
    }
    if (sr == B2SR_PLUS_TIMES && in_kind == B2SR_VEC_F32 && out_kind == B2SR_VEC_F32) {
        if (weights) return fail(B2SR_ERR_INVALID_ARG, "weights apply to MIN_PLUS only");
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemPlus<K> sem{static_cast<const float*>(x), static_cast<float*>(y), mask, comp, h->n};
            return run_spmv<K>(h, sem, nullptr, s, "spmv_plus", 8.0 * h->n + (mask ? h->n / 8.0 : 0.0), gate);
        });
    }
    if (sr == B2SR_MIN_PLUS && in_kind == B2SR_VEC_F32 && out_kind == B2SR_VEC_F32) {
        if (weights) B2SR_TRY(ensure_voff(h, s));
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemMinPlus<K> sem{static_cast<const float*>(x), static_cast<float*>(y), mask, comp, h->n, weights,
                              h->voff, weights != nullptr};
            return run_spmv<K>(h, sem, nullptr, s, "spmv_minplus",
                               8.0 * h->n + (mask ? h->n / 8.0 : 0.0) +
                                   (weights ? 4.0 * (double)h->nnz + 4.0 * (double)h->T : 0.0), gate);
        });
    }
    if (sr == B2SR_MIN_PLUS && in_kind == B2SR_VEC_I32 && out_kind == B2SR_VEC_I32) {
        if (weights) return fail(B2SR_ERR_INVALID_ARG, "int32 MIN_PLUS takes no weights (all weights are 0)");
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemMinI32<K> sem{static_cast<const int32_t*>(x), static_cast<int32_t*>(y), mask, comp, h->n};
            return run_spmv<K>(h, sem, nullptr, s, "spmv_min_i32", 8.0 * h->n + (mask ? h->n / 8.0 : 0.0), gate);
        });
    }
    if (sr == B2SR_MAX_TIMES && in_kind == B2SR_VEC_F32 && out_kind == B2SR_VEC_F32) {
        if (weights) return fail(B2SR_ERR_INVALID_ARG, "weights apply to MIN_PLUS only");
        return with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            SemMaxF32<K> sem{static_cast<const float*>(x), static_cast<float*>(y), mask, comp, h->n};
            return run_spmv<K>(h, sem, nullptr, s, "spmv_max", 8.0 * h->n + (mask ? h->n / 8.0 : 0.0), gate);
        });
    }
    return fail(B2SR_ERR_INVALID_ARG, "unsupported semiring / vector kind combination");
}

b2sr_status spmm64_dispatch(b2sr_matrix* h, const uint64_t* X, uint64_t* Y, const uint64_t* M, int comp,
                            cudaStream_t s, const int32_t* gate, bool edges, void* scratch, LiveColumns live) {
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        SemOr64<K> sem{reinterpret_cast<const unsigned long long*>(X), reinterpret_cast<unsigned long long*>(Y),
                       reinterpret_cast<const unsigned long long*>(M), comp ? 1 : 0, h->n, live.bits, live.dense};
        return run_spmv<K>(h, sem, nullptr, s, "spmm_or64", (M ? 24.0 : 16.0) * h->n, gate, edges, scratch);
    });
}

// The same over 32-lane words (at most 32 frontiers): half the bytes per
// gather and 4-byte accumulators, which the tile_dim-4 kernel takes.
b2sr_status spmm32_dispatch(b2sr_matrix* h, const uint32_t* X, uint32_t* Y, const uint32_t* M, int comp,
                            cudaStream_t s, const int32_t* gate, bool edges, LiveColumns live) {
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        SemOr32<K> sem{X, Y, M, comp ? 1 : 0, h->n, live.bits, live.dense};
        return run_spmv<K>(h, sem, nullptr, s, "spmm_or32", (M ? 12.0 : 8.0) * h->n, gate, edges);
    });
}

b2sr_status spmv_maxkey_dispatch(b2sr_matrix* h, const uint64_t* x, uint64_t* y, const uint32_t* mask, int comp,
                                 cudaStream_t s, const int32_t* gate) {
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        SemMaxKey<K> sem{reinterpret_cast<const unsigned long long*>(x), reinterpret_cast<unsigned long long*>(y), mask,
                         comp ? 1 : 0, h->n};
        return run_spmv<K>(h, sem, nullptr, s, "spmv_maxkey", 16.0 * h->n + (mask ? h->n / 8.0 : 0.0), gate);
    });
}

b2sr_status spmm4_dispatch(b2sr_matrix* h, const float* X, float* Y, const uint32_t* M, int comp, cudaStream_t s,
                           const int32_t* gate, bool edges, void* scratch) {
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        SemPlus4<K> sem{reinterpret_cast<const float4*>(X), reinterpret_cast<float4*>(Y), M, comp ? 1 : 0, h->n};
        return run_spmv<K>(h, sem, nullptr, s, "spmm_plus4", 32.0 * h->n + (M ? h->n / 8.0 : 0.0), gate, edges,
                           scratch);
    });
}

}  // namespace b2sr

using namespace b2sr;

extern "C" b2sr_status b2sr_spmm_f32x4(b2sr_handle h, const float* X, float* Y, const uint32_t* mask,
                                       int mask_complement, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (h->n > 0 && (!X || !Y)) return fail(B2SR_ERR_INVALID_ARG, "X or Y is NULL");
    if (X == Y) return fail(B2SR_ERR_INVALID_ARG, "Y must not alias X");
    if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15u)
        return fail(B2SR_ERR_INVALID_ARG, "X and Y must be 16-byte aligned");
    return spmm4_dispatch(h, X, Y, mask, mask_complement, to_stream(stream), nullptr);
}

extern "C" b2sr_status b2sr_spmv(b2sr_handle h, b2sr_semiring semiring, b2sr_vec in_kind, const void* x,
                                 b2sr_vec out_kind, void* y, const uint32_t* mask, int mask_complement,
                                 const float* weights, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (h->n > 0 && (!x || !y)) return fail(B2SR_ERR_INVALID_ARG, "x or y is NULL");
    if (x == y) return fail(B2SR_ERR_INVALID_ARG, "y must not alias x");
    return spmv_dispatch(h, semiring, in_kind, x, out_kind, y, mask, mask_complement, weights, to_stream(stream),
                         nullptr);
}

extern "C" b2sr_status b2sr_spmm_bits64(b2sr_handle h, const uint64_t* X, uint64_t* Y, const uint64_t* M,
                                        int complement, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (h->n > 0 && (!X || !Y)) return fail(B2SR_ERR_INVALID_ARG, "X or Y is NULL");
    if (X == Y) return fail(B2SR_ERR_INVALID_ARG, "Y must not alias X");
    return spmm64_dispatch(h, X, Y, M, complement, to_stream(stream), nullptr);
}

// ---------------------------------------------------------------------------
// Boolean SpMV without device allocation.
//
// Some callers cannot allocate device memory when they call into the library:
// a host whose own allocator has already reserved the device's free memory,
// or a deployment that must not allocate once it is running (fixed-memory or
// real-time services).  For them b2sr_spmv_bool_noalloc keeps the only scratch
// the Boolean SpMV needs -- the per-chunk partial rows joined by the fixup
// kernel at k = 16 and 32; k = 4 and 8 OR into the output and need none -- in a
// fixed array compiled into this file.  A device holds its copy
// from the moment the runtime loads this file's device code on it (the first
// SpMV launch or symbol lookup there, under lazy module loading) until the
// process exits or the device is reset.
// ---------------------------------------------------------------------------
namespace b2sr {

constexpr size_t kNoallocScratchBytes = size_t(4) << 20;  // 4 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

// Device address of g_noalloc_scratch, looked up once per device (host code
// cannot use the symbol itself as a device pointer).
static void* noalloc_scratch_ptr(int dev, b2sr_status* st) {
    static std::mutex mu;
    static void* ptrs[64] = {nullptr};
    if (dev < 0 || dev >= 64) {
        *st = fail(B2SR_ERR_INVALID_ARG, "device index out of range for the fixed scratch");
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (!ptrs[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) {
            *st = cuda_fail(e, "cudaGetSymbolAddress(fixed scratch)");
            return nullptr;
        }
        ptrs[dev] = p;
    }
    *st = B2SR_OK;
    return ptrs[dev];
}

template <int K>
static b2sr_status run_spmv_bool_fixed(const b2sr_matrix* h, const SemBool<K>& sem, uint32_t* y, void* scratch,
                                       cudaStream_t s) {
    using SEM = SemBool<K>;
    constexpr int NV = SEM::NV;
    const size_t half = round_up((size_t)h->nchunks * NV * sizeof(uint32_t), 256);
    if (2 * half > kNoallocScratchBytes)
        return fail(B2SR_ERR_INVALID_ARG, "matrix too large for b2sr_spmv_bool_noalloc: " +
                                              std::to_string(h->nchunks) + " chunks need " +
                                              std::to_string(2 * half) + " scratch bytes, the fixed array holds " +
                                              std::to_string(kNoallocScratchBytes));
    SpmvGeom g{h->rowptr, h->colind, h->tiles, h->chunk_row, h->T, h->nchunks, h->ntr, nullptr};
    if constexpr (OrsInto<SEM>::value) {  // needs no scratch; the entry point's limit stays what it was
        B2SR_TRY(clear_bitset(h, y, s, nullptr));
        if (h->nchunks == 0) return B2SR_OK;
        return launch_direct<K, SEM>(h, sem, Partials<uint32_t>{nullptr, nullptr}, s, g);
    } else {
        B2SR_TRY(clear_bitset_tail<K>(h, y, s, nullptr));
        // every partial the fixup reads is written by the chunk kernel of the
        // same call, so the scratch needs no clearing between calls
        Partials<uint32_t> part;
        part.val_first = static_cast<uint32_t*>(scratch);
        part.val_last = reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(scratch) + half);
        if (h->nchunks > 0) B2SR_TRY((launch_direct<K, SEM>(h, sem, part, s, g)));
        return launch_fixup<K, SEM>(h, sem, part, s, nullptr, true);
    }
}

}  // namespace b2sr

extern "C" b2sr_status b2sr_spmv_bool_noalloc(b2sr_handle h, const uint32_t* x, uint32_t* y, const uint32_t* mask,
                                              int mask_complement, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (h->n > 0 && (!x || !y)) return fail(B2SR_ERR_INVALID_ARG, "x or y is NULL");
    if (x == y) return fail(B2SR_ERR_INVALID_ARG, "y must not alias x");
    int dev = 0;
    B2SR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != h->device)
        return fail(B2SR_ERR_INVALID_ARG, "the handle belongs to device " + std::to_string(h->device) +
                                              ", the current device is " + std::to_string(dev));
    b2sr_status st = B2SR_OK;
    void* scratch = noalloc_scratch_ptr(dev, &st);
    if (!scratch) return st;
    const int comp = mask_complement ? 1 : 0;
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        SemBool<K> sem{x, y, mask, comp, h->n};
        return run_spmv_bool_fixed<K>(h, sem, y, scratch, to_stream(stream));
    });
}
