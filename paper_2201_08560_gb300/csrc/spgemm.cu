// B2SR SpGEMM: bmm_bin_bin_sum_masked (Table 3, Listing 2; the fused-sum
// triangle-counting kernel of Sec. V) and the Boolean product C = A (x) B.
//
// Masked count, two forms with one result: over the operands' rows, extracted as
// column lists (further down), and over tiles, where those are full, the mask has
// few or the rows find no room.  Tile form: each warp takes a run of consecutive mask tiles (so their
// tile-rows come from one search, then a walk of the row pointers); for a mask
// tile (I, J) the tile-column lists of A's tile-row I and B's tile-row J are
// intersected (binary search of the shorter list's entries in the longer one,
// 32 lanes at a time); every common K adds
//   sum over bits (r, c) of M_IJ of popc(A_IK[r] & B_JK[c]),
// i.e. Listing 2's AND-popc of two bit-rows, restricted to the mask.  Lanes
// accumulate in registers, a warp sums with shuffles and one 64-bit atomic
// per warp joins the global count (integer, so the order does not matter).
//
// Boolean product: expand every tile product A_IK (x) B_KJ, whose row r is
// the OR of B_KJ's rows selected by the bits of A_IK[r]; sort the non-zero
// products by (I, J) with the library's radix sort; OR equal keys into the
// output tiles.
#include <algorithm>

#include "b2sr_internal.cuh"

namespace b2sr {

template <int K>
__device__ __forceinline__ uint32_t gword(const uint8_t* __restrict__ tiles, int64_t t, int r) {
    if (K == 32) return __ldg(reinterpret_cast<const uint32_t*>(tiles) + t * 32 + r);
    if (K == 16) return __ldg(reinterpret_cast<const uint16_t*>(tiles) + t * 16 + r);
    return __ldg(tiles + t * K + r);
}

// a k <= 8 tile as one word: byte r is row r
template <int K>
__device__ __forceinline__ uint64_t tile_word64(const uint8_t* __restrict__ tiles, int64_t t) {
    if (K == 8) return __ldg(reinterpret_cast<const unsigned long long*>(tiles) + t);
    return __ldg(reinterpret_cast<const uint32_t*>(tiles) + t);
}

// Tile positions fit int32 (a handle holds fewer than 2^31 tiles), which keeps
// the searches' arithmetic 32-bit.
__device__ __forceinline__ int32_t lower_bound_i32(const int32_t* __restrict__ a, int32_t lo, int32_t hi, int32_t v) {
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(a + mid) < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

struct MatView {
    const int32_t* rowptr;
    const int32_t* colind;
    const uint8_t* tiles;
    int64_t T;
    int32_t ntr;
};

template <int K>
__global__ void masked_count_kernel(MatView A, MatView B, MatView M, unsigned long long* __restrict__ out,
                                    unsigned long long* __restrict__ pairs) {
    const int lane = (int)lane_id();
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long acc = 0, npairs = 0;
    // each warp takes a run of consecutive mask tiles: their tile-row is found
    // once by a binary search and then advanced as the run crosses rows
    const int64_t per = (M.T + nw - 1) / nw;
    const int64_t t0 = gw * per, t1 = min(M.T, t0 + per);
    int32_t I = 0;
    if (t0 < t1) {
        int32_t lo = 0, hi = M.ntr - 1;  // largest I with M.rowptr[I] <= t0
        while (lo < hi) {
            int32_t mid = lo + (hi - lo + 1) / 2;
            if ((int64_t)__ldg(M.rowptr + mid) <= t0) lo = mid; else hi = mid - 1;
        }
        I = lo;
    }
    int64_t row_end = t0 < t1 ? __ldg(M.rowptr + I + 1) : 0;
    for (int64_t mt = t0; mt < t1; ++mt) {
        while (mt >= row_end) row_end = __ldg(M.rowptr + (++I) + 1);
        const int32_t J = __ldg(M.colind + mt);
        // k <= 8: a tile is one 32/64-bit word whose bytes are its rows, so a
        // row is picked by a shift; larger tiles keep their rows in registers
        constexpr int MR = K <= 8 ? 1 : K;
        uint32_t mrow[MR];
        uint64_t mw = 0;
        (void)mrow;
        if constexpr (K <= 8) {
            mw = tile_word64<K>(M.tiles, mt);
        } else {
#pragma unroll
            for (int r = 0; r < K; ++r) mrow[r] = gword<K>(M.tiles, mt, r);
        }
        const int32_t a0 = __ldg(A.rowptr + I), a1 = __ldg(A.rowptr + I + 1);
        const int32_t b0 = __ldg(B.rowptr + J), b1 = __ldg(B.rowptr + J + 1);
        const bool a_short = (a1 - a0) <= (b1 - b0);
        const int32_t s0 = a_short ? a0 : b0, s1 = a_short ? a1 : b1;
        const int32_t l0 = a_short ? b0 : a0, l1 = a_short ? b1 : a1;
        const int32_t* scol = a_short ? A.colind : B.colind;
        const int32_t* lcol = a_short ? B.colind : A.colind;
        int32_t from = l0;  // a lane's entries rise, so each search starts where its last one ended
        for (int32_t p = s0 + lane; p < s1; p += 32) {
            const int32_t Kc = __ldg(scol + p);
            const int32_t q = lower_bound_i32(lcol, from, l1, Kc);
            from = q;
            if (q >= l1 || __ldg(lcol + q) != Kc) continue;
            const int32_t ta = a_short ? p : q;  // tile A_IK
            const int32_t tb = a_short ? q : p;  // tile B_JK
            if constexpr (K <= 8) {
                const uint64_t aw = tile_word64<K>(A.tiles, ta), bw = tile_word64<K>(B.tiles, tb);
                uint64_t m = mw;
                while (m) {
                    const int bit = __ffsll((long long)m) - 1;  // row bit >> 3, column bit & 7
                    m &= m - 1;
                    acc += (unsigned long long)__popc((uint32_t)((aw >> (bit & ~7)) & (bw >> (8 * (bit & 7))) & 0xFFu));
                    ++npairs;
                }
            } else {
                uint32_t brow[K];
#pragma unroll
                for (int c = 0; c < K; ++c) brow[c] = gword<K>(B.tiles, tb, c);
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    uint32_t bits = mrow[r];
                    if (!bits) continue;
                    const uint32_t ar = gword<K>(A.tiles, ta, r);
                    while (bits) {
                        const int c = __ffs(bits) - 1;
                        bits &= bits - 1;
                        uint32_t bc = 0;
#pragma unroll
                        for (int q2 = 0; q2 < K; ++q2) bc = (q2 == c) ? brow[q2] : bc;
                        acc += (unsigned long long)__popc(ar & bc);
                        ++npairs;
                    }
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        npairs += __shfl_xor_sync(0xffffffffu, npairs, o);
    }
    if (lane == 0) {
        if (acc) atomicAdd(out, acc);
        if (pairs && npairs) atomicAdd(pairs, npairs);
    }
}

// ---------------------------------------------------------------------------
// masked count over rows
// ---------------------------------------------------------------------------
// For every mask entry (i, j): the columns common to row i of A and row j of
// B.  The three operands' rows are extracted as column lists first (one
// balanced pass over their tiles).  The shorter of the two rows is walked and
// tested in the longer one: a first launch takes the entries whose row of A is
// at least as long, by rows of the mask, a second one the others, by columns
// (walking row j of B always: 3.5 G columns for the triangles of R-MAT 18, ef
// 32; the shorter row: 1.2 G).  A block takes kRunEntries consecutive mask
// entries, row by row:
//   * a row with more than 32 columns becomes a bitmap in the block's shared
//     memory; the warps fetch the row's mask entries one by one, and the lanes
//     walk the entry's other row, testing each column in the bitmap: a
//     coalesced load and one shared load per column, no searches;
//   * a shorter row stays a list: eight lanes a mask entry search its columns
//     in the entry's other row;
//   * a long row whose entries in the run have few columns to test for the
//     row's length, and an entry whose other row is many times longer, are
//     searched: a warp an entry walks the shorter row and looks its columns up
//     in the longer one.
// Where a bitmap of n bits does not fit in shared memory every long row is
// searched, in one launch; where it leaves an SM few blocks, rows of up to
// kApartRow columns are.
constexpr int kRunEntries = 256;
constexpr int64_t kMaxBitmapBytes = 200 * 1024;
// Fewer mask entries than this take one launch: grouping the others by column
// (five launches and a scan, 60 us) costs more than the shorter walks save
// (R-MAT 16, 1.8M entries, half of them below the diagonal: about as much).
constexpr int64_t kSplitEntries = 1 << 21;
// Up to this size a run's bitmaps are made where its lists are; larger ones
// leave few blocks on an SM, so a second launch makes them, for the runs that
// have rows for them, and the lists go first without.
constexpr int kOneLaunchBitmap = 32 * 1024;
constexpr int32_t kApartRow = 512;
// A looked-up column costs a chain of loads where a tested one costs one, and a
// bitmap costs two passes over its row.
constexpr int kSearchLonger = 8;  // an entry is searched if its other row is longer by this factor
constexpr int kSearchFewer = 4;   // a row is if it has this many columns for each one to test

// Row i: colind[begin[i] .. end[i]) (end = begin + 1 for a plain CSR).  Rows
// lie one after another, with gaps where end[i] < begin[i + 1].
struct RowLists {
    const int32_t* begin;
    const int32_t* end;
    const int32_t* colind;
};

// Columns of the list acol[0..d) in the row [b0, b1) of B, by a group of WIDTH
// lanes.
template <int WIDTH>
__device__ __forceinline__ uint32_t count_listed(const int32_t* __restrict__ acol, int32_t d,
                                                 const int32_t* __restrict__ bcol, int32_t b0, int32_t b1, int sub) {
    uint32_t acc = 0;
    for (int32_t p = sub; p < d; p += WIDTH) {
        const int32_t v = __ldg(acol + p);
        const int32_t q = lower_bound_i32(bcol, b0, b1, v);
        acc += q < b1 && __ldg(bcol + q) == v;
    }
    return acc;
}

__global__ void column_starts_kernel(const int64_t* __restrict__ off, int64_t len, int32_t* __restrict__ colptr,
                                     int32_t* __restrict__ cursor) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        colptr[i] = cursor[i] = (int32_t)off[i];
}

// Mask entries whose row of B is longer than their row of A.  First pass: the
// entry's row in row_of (-1 for the others), counted by column; second: the
// rows written by column.  A thread an entry, so that a hub's row is shared
// (a warp a row took 520 us a pass on R-MAT 18, ef 32).
__global__ void count_by_column_kernel(int32_t n, RowLists A, RowLists B, RowLists M, int32_t mnnz,
                                       int32_t* __restrict__ row_of, int32_t* __restrict__ count) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < mnnz; e += (int64_t)gridDim.x * blockDim.x) {
        int32_t lo = 0, hi = n - 1;  // the last row starting at or before e
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo + 1) >> 1);
            if (__ldg(M.begin + mid) <= e) lo = mid; else hi = mid - 1;
        }
        const int32_t d = __ldg(A.end + lo) - __ldg(A.begin + lo);
        const int32_t j = __ldg(M.colind + e);
        const bool other = d > 0 && e < __ldg(M.end + lo) && __ldg(B.end + j) - __ldg(B.begin + j) > d;
        row_of[e] = other ? lo : -1;
        if (other) atomicAdd(count + j, 1);
    }
}

__global__ void place_by_column_kernel(const int32_t* __restrict__ row_of, const int32_t* __restrict__ mcol,
                                       int32_t mnnz, int32_t* __restrict__ cursor, int32_t* __restrict__ rows) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < mnnz; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = __ldg(row_of + e);
        if (i >= 0) rows[atomicAdd(cursor + __ldg(mcol + e), 1)] = i;
    }
}

// What a launch does of its runs: all; all but the rows that take bitmaps, and
// lists the runs that have some; those rows, of the listed runs.
enum { kRunsWhole, kRunsLists, kRunsBitmaps };

template <int PART>
__global__ void __launch_bounds__(256) masked_rows_kernel(int32_t n, RowLists A, RowLists B, RowLists M,
                                                          const int32_t* __restrict__ mnnz, int longer, int32_t bitmap_from,
                                                          int bitmap_words, int32_t* __restrict__ pending,
                                                          unsigned long long* __restrict__ out) {
    extern __shared__ __align__(16) uint32_t bitmap[];
    __shared__ unsigned long long warp_sum[8];
    // the run's entries: where row i of A begins, row j of B as a range (compact:
    // six blocks an SM beside bitmaps of 2^18 bits)
    __shared__ int32_t row_a[kRunEntries];      // at a long row's first entry: columns to test for the row
    __shared__ int2 row_b[kRunEntries];
    __shared__ int32_t long_row[kRunEntries];   // rows with more than bitmap_from columns
    __shared__ uint8_t short_len[kRunEntries];  // row i's length, up to 32; of a longer row: 1 where the entry is searched
    __shared__ uint8_t listed[kRunEntries];     // entries of rows with up to 32 columns; from the back, searched entries
    __shared__ uint8_t other[kRunEntries];      // entries of one long row
    __shared__ int nlong, nlisted, nsearched, nother;
    __shared__ int32_t row_range[2];
    const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
    const int32_t nruns = PART == kRunsBitmaps ? __ldg(pending) : (int32_t)gridDim.x;  // pending[0]: how many are listed
    unsigned long long sum = 0;
    if (PART != kRunsLists) {
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);  // the bitmap is padded to whole 16 bytes
        for (int w = threadIdx.x; w < (bitmap_words + 3) / 4; w += 256) reinterpret_cast<uint4*>(bitmap)[w] = zero;
    }
    for (int32_t run = blockIdx.x; run < nruns; run += gridDim.x) {
        const int32_t e0 = (PART == kRunsBitmaps ? __ldg(pending + 1 + run) : run) * kRunEntries;
        const int32_t e1 = min(e0 + kRunEntries, __ldg(mnnz));
        if (e0 >= e1) continue;  // the same for every thread
        // the last row starting at or before entry e, between lo and hi
        auto row_at = [&](int32_t e, int32_t lo, int32_t hi) {
            while (lo < hi) {
                const int32_t mid = lo + ((hi - lo + 1) >> 1);
                if (__ldg(M.begin + mid) <= e) lo = mid; else hi = mid - 1;
            }
            return lo;
        };
        if (PART == kRunsBitmaps) __syncthreads();  // the run before is done with
        if (warp < 2) {  // rows of the first and the last entry of the run
            const int32_t i = row_at(warp == 0 ? e0 : e1 - 1, 0, n - 1);
            if (lane == 0) row_range[warp] = i;
        }
        if (threadIdx.x == 0) nlong = nlisted = nsearched = nother = 0;
        row_a[threadIdx.x] = 0;
        __syncthreads();
        const int32_t i0 = row_range[0], i1 = row_range[1];
        if (i0 == i1 && __ldg(M.end + i0) <= e0) continue;  // the run lies in a gap
        {
            const int t = threadIdx.x;
            const int32_t e = e0 + t;
            int2 rb = make_int2(0, 0);
            if (e < e1) {
                const int32_t i = row_at(e, i0, i1);
                if (e < __ldg(M.end + i)) {
                    const int32_t j = __ldg(M.colind + e);
                    const int32_t a0 = __ldg(A.begin + i), d = __ldg(A.end + i) - a0;
                    rb = make_int2(__ldg(B.begin + j), __ldg(B.end + j));
                    if (d > bitmap_from && (t == 0 || e == __ldg(M.begin + i))) long_row[atomicAdd(&nlong, 1)] = i;
                    const int32_t len = rb.y - rb.x;
                    if (d <= 0 || len <= 0 || (longer && len > d)) {
                        rb.y = rb.x;  // nothing to count here
                    } else if (d <= 32) {
                        row_a[t] = a0;
                        short_len[t] = (uint8_t)d;
                        listed[atomicAdd(&nlisted, 1)] = (uint8_t)t;
                    } else if (d <= bitmap_from || len / kSearchLonger > d) {
                        short_len[t] = 1;
                        listed[kRunEntries - 1 - atomicAdd(&nsearched, 1)] = (uint8_t)t;
                    } else {
                        short_len[t] = 0;
                        atomicAdd(row_a + max(__ldg(M.begin + i) - e0, 0), min(len, 1 << 22));
                    }
                }
            }
            row_b[t] = rb;
        }
        __syncthreads();
        uint32_t acc = 0;
        // the columns that row i of A, [a0, a1), and row [b.x, b.y) of B share, by a warp
        auto search = [&](int32_t a0, int32_t a1, int2 b) {
            return b.y - b.x <= a1 - a0 ? count_listed<32>(B.colind + b.x, b.y - b.x, A.colind, a0, a1, lane)
                                        : count_listed<32>(A.colind + a0, a1 - a0, B.colind, b.x, b.y, lane);
        };
        if (PART != kRunsBitmaps) {
            for (int q = threadIdx.x >> 3; q < nlisted; q += 32) {
                const int t = listed[q];
                acc += count_listed<8>(A.colind + row_a[t], short_len[t], B.colind, row_b[t].x, row_b[t].y, lane & 7);
            }
            for (int q = warp; q < nsearched; q += 8) {
                const int t = listed[kRunEntries - 1 - q];
                const int32_t i = row_at(e0 + t, i0, i1);
                acc += search(__ldg(A.begin + i), __ldg(A.end + i), row_b[t]);
            }
        }
        int bitmaps = 0;
        for (int r = 0; r < nlong; ++r) {
            const int32_t i = long_row[r];
            const int32_t a0 = __ldg(A.begin + i), a1 = __ldg(A.end + i);
            const int32_t m0 = max(e0, __ldg(M.begin + i)), m1 = min(e1, __ldg(M.end + i));
            const int32_t tests = row_a[m0 - e0];
            if (tests < (a1 - a0) / kSearchFewer) {  // the same for every thread
                if (PART != kRunsBitmaps)
                    for (int t = m0 - e0 + warp; t < m1 - e0; t += 8)
                        if (row_b[t].y > row_b[t].x && !short_len[t]) acc += search(a0, a1, row_b[t]);
                continue;
            }
            ++bitmaps;
            if (PART == kRunsLists) continue;
            if (threadIdx.x < m1 - m0) {
                const int t = m0 - e0 + threadIdx.x;
                if (row_b[t].y > row_b[t].x && !short_len[t]) other[atomicAdd(&nother, 1)] = (uint8_t)t;
            }
            for (int32_t p = a0 + threadIdx.x; p < a1; p += 256) {
                const int32_t v = __ldg(A.colind + p);
                atomicOr(bitmap + (v >> 5), 1u << (v & 31));
            }
            __syncthreads();
            const int todo = nother;
            // the next entry's first columns are loaded before this one's are used
            auto test = [&](int32_t v) { return (bitmap[v >> 5] >> (v & 31)) & 1u; };
            int2 o = warp < todo ? row_b[other[warp]] : make_int2(0, 0);
            int32_t v = o.x + lane < o.y ? __ldg(B.colind + o.x + lane) : -1;
            for (int q = warp; q < todo; q += 8) {
                const int2 o2 = q + 8 < todo ? row_b[other[q + 8]] : make_int2(0, 0);
                const int32_t v2 = o2.x + lane < o2.y ? __ldg(B.colind + o2.x + lane) : -1;
                if (v >= 0) acc += test(v);
#pragma unroll 4
                for (int32_t p = o.x + 32 + lane; p < o.y; p += 32) acc += test(__ldg(B.colind + p));
                o = o2;
                v = v2;
            }
            __syncthreads();
            for (int32_t p = a0 + threadIdx.x; p < a1; p += 256) bitmap[__ldg(A.colind + p) >> 5] = 0u;
            if (threadIdx.x == 0) nother = 0;
            __syncthreads();
        }
        if (PART == kRunsLists && bitmaps > 0 && threadIdx.x == 0) pending[1 + atomicAdd(pending, 1)] = run;
        sum += acc;
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) warp_sum[warp] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) total += warp_sum[w];
        if (total) atomicAdd(out, total);
    }
}

// ---------------------------------------------------------------------------
// Boolean SpGEMM (expand, sort, merge)
// ---------------------------------------------------------------------------
__global__ void row_of_tiles_kernel(const int32_t* __restrict__ rowptr, int32_t ntr, int64_t T,
                                    int32_t* __restrict__ tilerow) {
    for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < ntr;
         I += (int64_t)gridDim.x * blockDim.x)
        for (int64_t t = rowptr[I]; t < rowptr[I + 1]; ++t) tilerow[t] = (int32_t)I;
}

__global__ void product_counts_kernel(const int32_t* __restrict__ a_colind, int64_t TA,
                                      const int32_t* __restrict__ b_rowptr, int32_t* __restrict__ cnt) {
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < TA;
         a += (int64_t)gridDim.x * blockDim.x) {
        int32_t Kc = a_colind[a];
        cnt[a] = b_rowptr[Kc + 1] - b_rowptr[Kc];
    }
}

template <int K>
__global__ void expand_kernel(const int32_t* __restrict__ a_tilerow, const int32_t* __restrict__ a_colind,
                              const uint8_t* __restrict__ a_tiles, int64_t TA, const int64_t* __restrict__ off,
                              const int32_t* __restrict__ b_rowptr, const int32_t* __restrict__ b_colind,
                              const uint8_t* __restrict__ b_tiles, int64_t P, int sbits,
                              uint64_t* __restrict__ keys, uint32_t* __restrict__ idx,
                              uint32_t* __restrict__ prod) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P;
         p += (int64_t)gridDim.x * blockDim.x) {
        // A tile a with off[a] <= p < off[a+1]
        int64_t lo = 0, hi = TA - 1;
        while (lo < hi) {
            int64_t mid = (lo + hi + 1) >> 1;
            if (off[mid] <= p) lo = mid; else hi = mid - 1;
        }
        const int64_t a = lo;
        const int32_t Kc = a_colind[a];
        const int64_t b = b_rowptr[Kc] + (p - off[a]);
        const int32_t I = a_tilerow[a];
        const int32_t J = b_colind[b];
        uint32_t any = 0;
#pragma unroll
        for (int r = 0; r < K; ++r) {
            uint32_t ar = gword<K>(a_tiles, a, r);
            uint32_t row = 0;
            while (ar) {
                int m = __ffs(ar) - 1;
                ar &= ar - 1;
                row |= gword<K>(b_tiles, b, m);
            }
            prod[p * K + r] = row;
            any |= row;
        }
        keys[p] = any ? (((uint64_t)I << sbits) | (uint64_t)J) : ~0ull;
        idx[p] = (uint32_t)p;
    }
}

__global__ void spgemm_heads_kernel(const uint64_t* __restrict__ keys, int64_t N, int32_t* __restrict__ flag) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N;
         e += (int64_t)gridDim.x * blockDim.x)
        flag[e] = (keys[e] != ~0ull && (e == 0 || keys[e] != keys[e - 1])) ? 1 : 0;
}

template <int K>
__global__ void spgemm_merge_kernel(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ idx,
                                    const int32_t* __restrict__ flag, const int64_t* __restrict__ tidx, int64_t N,
                                    const uint32_t* __restrict__ prod, int sbits, int32_t* __restrict__ c_colind,
                                    int32_t* __restrict__ c_tilerow, uint32_t* __restrict__ c_tiles32) {
    constexpr int WB = K <= 8 ? 1 : (K == 16 ? 2 : 4);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N;
         e += (int64_t)gridDim.x * blockDim.x) {
        uint64_t key = keys[e];
        if (key == ~0ull) continue;
        int64_t t = tidx[e] + flag[e] - 1;  // tile of this run
        if (flag[e]) {
            c_colind[t] = (int32_t)(key & ((1ull << sbits) - 1ull));
            c_tilerow[t] = (int32_t)(key >> sbits);
        }
        const uint32_t* pr = prod + (int64_t)idx[e] * K;
#pragma unroll
        for (int r = 0; r < K; ++r) {
            uint32_t v = pr[r];
            if (!v) continue;
            int64_t byte = (t * K + r) * WB;
            atomicOr(c_tiles32 + (byte >> 2), v << ((int)(byte & 3) * 8));
        }
    }
}

__global__ void build_rowptr_from_rows(const int32_t* __restrict__ tilerow, int64_t T, int32_t ntr,
                                       int32_t* __restrict__ rowptr) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= T;
         t += (int64_t)gridDim.x * blockDim.x) {
        int32_t prev = t == 0 ? -1 : tilerow[t - 1];
        int32_t cur = t == T ? ntr : tilerow[t];
        for (int32_t R = prev + 1; R <= cur; ++R) rowptr[R] = (int32_t)t;
    }
}

static MatView view(const b2sr_matrix* h) { return MatView{h->rowptr, h->colind, h->tiles, h->T, h->ntr}; }

// Tiles a third full or more: the tile form counts such a mask faster than the
// row form, whose work goes with the entries; at k = 32 where bitmaps leave an SM
// few blocks.  us, tiles / rows, triangles of 64-vertex cliques, n = 2^20: k = 4
// 1,798 / 12,817, k = 8 1,461 / 12,951, k = 16 2,327 / 12,724, k = 32 4,783 /
// 6,948; of 256-vertex cliques, n = 2^15: k = 8 365 / 722, k = 32 1,432 / 777.
static bool full_tiles(const b2sr_matrix* h, int64_t nnz, int64_t T) {
    return (h->k <= 16 || ceil_div(h->n, 32) * 4 > kOneLaunchBitmap) && 3 * nnz >= (int64_t)h->k * h->k * T;
}

// Row lists of a handle, owned by `buf`.
static b2sr_status row_lists(const b2sr_matrix* h, DevBuf& buf, RowLists* out, cudaStream_t s) {
    DevBuf off(s);
    const size_t rp = round_up(((int64_t)h->n + 1) * sizeof(int32_t), 256);
    B2SR_TRY(off.alloc(((size_t)h->n + 1) * sizeof(int64_t)));
    B2SR_TRY(buf.alloc(rp + (size_t)h->nnz * sizeof(int32_t) + 4));
    int32_t* rowptr = buf.as<int32_t>();
    int32_t* colind = reinterpret_cast<int32_t*>(buf.as<char>() + rp);
    B2SR_TRY(extract_csr(h, off.as<int64_t>(), rowptr, colind, s));
    *out = RowLists{rowptr, rowptr + 1, colind};
    return B2SR_OK;
}

// The count over extracted rows; `slots` entries of m.colind, gaps included,
// hold the mask.
static b2sr_status count_rows(int32_t n, RowLists a, RowLists b, RowLists m, int64_t slots, unsigned long long* out,
                              cudaStream_t s, double bytes) {
    const int64_t words = ceil_div(n, 32);
    const bool use_bitmap = words * 4 <= kMaxBitmapBytes;
    const int smem = use_bitmap ? (int)round_up(words, 4) * 4 : 0;
    const int64_t runs = ceil_div(slots, kRunEntries);
    const bool split = use_bitmap && slots >= kSplitEntries;
    const bool apart = use_bitmap && smem > kOneLaunchBitmap;
    const int32_t bitmap_from = !use_bitmap ? INT32_MAX : (apart ? kApartRow : 32);
    DevBuf listed(s);
    if (apart) B2SR_TRY(listed.alloc((size_t)(runs + 1) * sizeof(int32_t)));
    // the largest bitmap, not this call's: the limit belongs to the kernel, and
    // another thread's call with a smaller graph must not lower it before a launch
    for (auto kernel : {masked_rows_kernel<kRunsWhole>, masked_rows_kernel<kRunsBitmaps>})
        B2SR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxBitmapBytes));
    // the entries of mask mm, the rows of x against those of y; mm.begin[n] (the row
    // pointer of a CSR) ends the slots
    auto count_runs = [&](RowLists x, RowLists y, RowLists mm, int longer) -> b2sr_status {
        if (!apart) {
            masked_rows_kernel<kRunsWhole><<<(unsigned)runs, 256, smem, s>>>(n, x, y, mm, mm.begin + n, longer, bitmap_from,
                                                                            use_bitmap ? (int)words : 0, nullptr, out);
            B2SR_LAUNCH_CHECK("masked_rows_kernel");
            return B2SR_OK;
        }
        int32_t* pending = listed.as<int32_t>();
        B2SR_CUDA_TRY(cudaMemsetAsync(pending, 0, sizeof(int32_t), s));
        masked_rows_kernel<kRunsLists><<<(unsigned)runs, 256, 0, s>>>(n, x, y, mm, mm.begin + n, longer, bitmap_from,
                                                                     (int)words, pending, out);
        B2SR_LAUNCH_CHECK("masked_rows_kernel");
        const int64_t resident = (int64_t)sm_count() * std::max<int64_t>(1, kMaxBitmapBytes / smem);
        masked_rows_kernel<kRunsBitmaps><<<(unsigned)std::min<int64_t>(runs, resident), 256, smem, s>>>(
            n, x, y, mm, mm.begin + n, longer, bitmap_from, (int)words, pending, out);
        B2SR_LAUNCH_CHECK("masked_rows_kernel");
        return B2SR_OK;
    };
    // the other entries by column: cnt, off, colptr and cursor a column, row_of and
    // the rows a slot
    DevBuf cnt(s), off(s), cur(s), rows(s);
    if (split) {
        B2SR_TRY(cnt.alloc(((size_t)n + 1) * sizeof(int32_t)));
        B2SR_TRY(off.alloc(((size_t)n + 1) * sizeof(int64_t)));
        B2SR_TRY(cur.alloc(2 * ((size_t)n + 1) * sizeof(int32_t)));
        B2SR_TRY(rows.alloc(2 * (size_t)slots * sizeof(int32_t)));
    }
    void* tok = timing_begin(s);
    auto count_all = [&]() -> b2sr_status {
        B2SR_TRY(count_runs(a, b, m, split));
        if (!split) return B2SR_OK;
        int32_t* colptr = cur.as<int32_t>();
        int32_t* cursor = colptr + n + 1;
        int32_t* row_of = rows.as<int32_t>() + slots;
        B2SR_CUDA_TRY(cudaMemsetAsync(cnt.p, 0, ((size_t)n + 1) * sizeof(int32_t), s));
        count_by_column_kernel<<<grid_wide(slots), 256, 0, s>>>(n, a, b, m, (int32_t)slots, row_of, cnt.as<int32_t>());
        B2SR_LAUNCH_CHECK("count_by_column_kernel");
        B2SR_TRY(exclusive_scan_i32_to_i64(cnt.as<int32_t>(), off.as<int64_t>(), (int64_t)n + 1, s));
        column_starts_kernel<<<grid_wide((int64_t)n + 1), 256, 0, s>>>(off.as<int64_t>(), (int64_t)n + 1, colptr, cursor);
        B2SR_LAUNCH_CHECK("column_starts_kernel");
        place_by_column_kernel<<<grid_wide(slots), 256, 0, s>>>(row_of, m.colind, (int32_t)slots, cursor,
                                                               rows.as<int32_t>());
        B2SR_LAUNCH_CHECK("place_by_column_kernel");
        return count_runs(b, a, RowLists{colptr, colptr + 1, rows.as<int32_t>()}, 0);
    };
    const b2sr_status st = count_all();
    timing_end(tok, "spgemm_masked", bytes, s);
    return st;
}

static b2sr_status masked_count_rows(const b2sr_matrix* A, const b2sr_matrix* B, const b2sr_matrix* M,
                                     unsigned long long* out, cudaStream_t s, double bytes) {
    DevBuf abuf(s), bbuf(s), mbuf(s);
    RowLists a, b, m;
    B2SR_TRY(row_lists(A, abuf, &a, s));
    if (B == A) b = a; else B2SR_TRY(row_lists(B, bbuf, &b, s));
    if (M == A) m = a; else if (M == B) m = b; else B2SR_TRY(row_lists(M, mbuf, &m, s));
    return count_rows(A->n, a, b, m, M->nnz, out, s, bytes);
}

// Row i's columns below i are a prefix of the row.
__global__ void lower_ends_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind, int32_t n,
                                  int32_t* __restrict__ end) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        end[i] = lower_bound_i32(colind, rowptr[i], rowptr[i + 1], (int32_t)i);
}

// Whether lower_count is the form for the triangles of h: rows of 2^31 entries
// or more and full tiles keep the tile form over the lower triangle.
bool counts_by_rows(const b2sr_matrix* h) {
    return h->nnz < (int64_t(1) << 31) - 1024 && !full_tiles(h, h->nnz, h->T);
}

// Triangles: L the strictly lower triangle of h, sum over its entries (i, j)
// of the columns common to rows i and j of L, without building L.
b2sr_status lower_count(const b2sr_matrix* h, int64_t* count, cudaStream_t s) {
    B2SR_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(int64_t), s));
    if (h->T == 0) return B2SR_OK;
    DevBuf buf(s), ends(s);
    RowLists a;
    B2SR_TRY(row_lists(h, buf, &a, s));
    B2SR_TRY(ends.alloc((size_t)h->n * sizeof(int32_t)));
    lower_ends_kernel<<<grid_wide(h->n), 256, 0, s>>>(a.begin, a.colind, h->n, ends.as<int32_t>());
    B2SR_LAUNCH_CHECK("lower_ends_kernel");
    a.end = ends.as<int32_t>();
    const double bytes = 4.0 * ((double)h->ntr + 1.0) + (double)h->T * (4.0 + tile_bytes(h->k));
    return count_rows(h->n, a, a, a, h->nnz, reinterpret_cast<unsigned long long*>(count), s, bytes);
}

// The masked count; `pairs` (device int64, optional) receives the number of
// AND-popc word operations of the tile form (one per mask bit per common
// tile-column).  The row form extracts all of A's and B's rows, so a mask of
// far fewer tiles than they have takes the tile form, and so do full tiles.
b2sr_status masked_count(const b2sr_matrix* A, const b2sr_matrix* B, const b2sr_matrix* M, int64_t* count,
                         cudaStream_t s, int64_t* pairs) {
    B2SR_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(int64_t), s));
    if (pairs) B2SR_CUDA_TRY(cudaMemsetAsync(pairs, 0, sizeof(int64_t), s));
    if (M->T == 0) return B2SR_OK;
    auto* out = reinterpret_cast<unsigned long long*>(count);
    auto* prs = reinterpret_cast<unsigned long long*>(pairs);
    const double bytes = 3.0 * (4.0 * ((double)A->ntr + 1.0)) + ((double)A->T + B->T + M->T) * (4.0 + tile_bytes(A->k));
    const int64_t most = std::max(A->nnz, std::max(B->nnz, M->nnz));
    if (!pairs && most < (int64_t(1) << 31) - kRunEntries && 16 * M->T >= A->T + B->T &&
        !full_tiles(A, A->nnz + B->nnz + M->nnz, A->T + B->T + M->T)) {
        const b2sr_status st = masked_count_rows(A, B, M, out, s, bytes);
        if (st != B2SR_ERR_OOM) return st;
        clear_error();  // the tile form needs no memory
        B2SR_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(int64_t), s));
    }
    return with_tile(A->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        // runs of eight mask tiles a warp; the blocks are scheduled as SMs free
        // up, which balances runs of long (hub) rows against short ones
        const int64_t warps = ceil_div(M->T, 8);
        const int grid = (int)std::max<int64_t>(1, ceil_div(warps, 8));
        void* tok = timing_begin(s);
        masked_count_kernel<K><<<grid, 256, 0, s>>>(view(A), view(B), view(M), out, prs);
        timing_end(tok, "spgemm_masked", bytes, s);
        B2SR_LAUNCH_CHECK("masked_count_kernel");
        return B2SR_OK;
    });
}

b2sr_status spgemm_bool(const b2sr_matrix* A, const b2sr_matrix* B, cudaStream_t s, b2sr_matrix** out) {
    const int k = A->k;
    const int32_t ntr = A->ntr;
    const int sbits = bits_for((int64_t)ntr + 1);  // all-ones key stays invalid
    int64_t P = 0;
    DevBuf a_tilerow(s), cnt(s), off(s);
    if (A->T > 0) {
        B2SR_TRY(a_tilerow.alloc(A->T * sizeof(int32_t)));
        B2SR_TRY(cnt.alloc((A->T + 1) * sizeof(int32_t)));
        B2SR_TRY(off.alloc((A->T + 1) * sizeof(int64_t)));
        row_of_tiles_kernel<<<grid_wide(ntr), 256, 0, s>>>(A->rowptr, ntr, A->T, a_tilerow.as<int32_t>());
        B2SR_LAUNCH_CHECK("row_of_tiles_kernel");
        product_counts_kernel<<<grid_wide(A->T), 256, 0, s>>>(A->colind, A->T, B->rowptr, cnt.as<int32_t>());
        B2SR_LAUNCH_CHECK("product_counts_kernel");
        B2SR_CUDA_TRY(cudaMemsetAsync(cnt.as<int32_t>() + A->T, 0, sizeof(int32_t), s));
        B2SR_TRY(exclusive_scan_i32_to_i64(cnt.as<int32_t>(), off.as<int64_t>(), A->T + 1, s));
        B2SR_CUDA_TRY(cudaMemcpyAsync(&P, off.as<int64_t>() + A->T, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    }
    if (P >= (int64_t(1) << 32)) return fail(B2SR_ERR_OOM, "Boolean SpGEMM: too many tile products");
    DevBuf keys(s), ktmp(s), idx(s), itmp(s), prod(s), flag(s), tidx(s);
    uint64_t* skeys = nullptr;
    uint32_t* sidx = nullptr;
    int64_t TC = 0;
    if (P > 0) {
        B2SR_TRY(keys.alloc(P * sizeof(uint64_t)));
        B2SR_TRY(ktmp.alloc(P * sizeof(uint64_t)));
        B2SR_TRY(idx.alloc(P * sizeof(uint32_t)));
        B2SR_TRY(itmp.alloc(P * sizeof(uint32_t)));
        B2SR_TRY(prod.alloc(P * k * sizeof(uint32_t)));
        B2SR_TRY(with_tile(k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            expand_kernel<K><<<grid_wide(P), 256, 0, s>>>(a_tilerow.as<int32_t>(), A->colind, A->tiles, A->T,
                                                         off.as<int64_t>(), B->rowptr, B->colind, B->tiles, P,
                                                         sbits, keys.as<uint64_t>(), idx.as<uint32_t>(),
                                                         prod.as<uint32_t>());
            B2SR_LAUNCH_CHECK("expand_kernel");
            return B2SR_OK;
        }));
        B2SR_TRY(radix_sort_u64_pairs(keys.as<uint64_t>(), ktmp.as<uint64_t>(), idx.as<uint32_t>(),
                                      itmp.as<uint32_t>(), P, 0, 2 * sbits, s, &skeys, &sidx));
        B2SR_TRY(flag.alloc(P * sizeof(int32_t)));
        B2SR_TRY(tidx.alloc(P * sizeof(int64_t)));
        spgemm_heads_kernel<<<grid_wide(P), 256, 0, s>>>(skeys, P, flag.as<int32_t>());
        B2SR_LAUNCH_CHECK("spgemm_heads_kernel");
        B2SR_TRY(exclusive_scan_i32_to_i64(flag.as<int32_t>(), tidx.as<int64_t>(), P, s));
        int64_t last = 0;
        int32_t lastf = 0;
        B2SR_CUDA_TRY(cudaMemcpyAsync(&last, tidx.as<int64_t>() + P - 1, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaMemcpyAsync(&lastf, flag.as<int32_t>() + P - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        TC = last + lastf;
    }
    const int64_t cap = std::max<int64_t>(round_up(TC, kTilePad), kTilePad);
    int32_t* crp = nullptr;
    int32_t* cci = nullptr;
    uint8_t* ct = nullptr;
    auto release = [&](b2sr_status st) {
        dfree(crp, s); dfree(cci, s); dfree(ct, s);
        return st;
    };
    b2sr_status st = dalloc(&crp, (size_t)ntr + 1, s);
    if (st == B2SR_OK) st = dalloc(&cci, (size_t)cap, s);
    if (st == B2SR_OK) st = dalloc(&ct, (size_t)cap * tile_bytes(k), s);
    if (st != B2SR_OK) return release(st);
    cudaError_t e = cudaMemsetAsync(cci, 0, (size_t)cap * sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(ct, 0, (size_t)cap * tile_bytes(k), s);
    if (e != cudaSuccess) return release(cuda_fail(e, "memset spgemm output"));
    DevBuf ctilerow(s);
    st = ctilerow.alloc(std::max<int64_t>(TC, 1) * sizeof(int32_t));
    if (st != B2SR_OK) return release(st);
    if (P > 0) {
        st = with_tile(k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            spgemm_merge_kernel<K><<<grid_wide(P), 256, 0, s>>>(skeys, sidx, flag.as<int32_t>(), tidx.as<int64_t>(), P,
                                                               prod.as<uint32_t>(), sbits, cci, ctilerow.as<int32_t>(),
                                                               reinterpret_cast<uint32_t*>(ct));
            B2SR_LAUNCH_CHECK("spgemm_merge_kernel");
            return B2SR_OK;
        });
        if (st != B2SR_OK) return release(st);
    }
    build_rowptr_from_rows<<<grid_wide(TC + 1), 256, 0, s>>>(ctilerow.as<int32_t>(), TC, ntr, crp);
    note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return release(cuda_fail(e, "build_rowptr_from_rows"));
    return new_handle_from_tiles(A->n, k, TC, crp, cci, ct, cap, s, out);
}

}  // namespace b2sr

using namespace b2sr;

extern "C" b2sr_status b2sr_spgemm_masked_count(b2sr_handle A, b2sr_handle B, b2sr_handle M, int64_t* count,
                                                void* stream) {
    clear_error();
    B2SR_TRY(check_handle(A));
    B2SR_TRY(check_handle(B));
    B2SR_TRY(check_handle(M));
    if (!count) return fail(B2SR_ERR_INVALID_ARG, "count is NULL");
    if (A->n != B->n || A->n != M->n || A->k != B->k || A->k != M->k)
        return fail(B2SR_ERR_INVALID_ARG, "A, B and M need the same n and tile_dim");
    return masked_count(A, B, M, count, to_stream(stream), nullptr);
}

extern "C" b2sr_status b2sr_spgemm_masked_count_work(b2sr_handle A, b2sr_handle B, b2sr_handle M, int64_t* count,
                                                     int64_t* pairs, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(A));
    B2SR_TRY(check_handle(B));
    B2SR_TRY(check_handle(M));
    if (!count || !pairs) return fail(B2SR_ERR_INVALID_ARG, "count or pairs is NULL");
    if (A->n != B->n || A->n != M->n || A->k != B->k || A->k != M->k)
        return fail(B2SR_ERR_INVALID_ARG, "A, B and M need the same n and tile_dim");
    return masked_count(A, B, M, count, to_stream(stream), pairs);
}

extern "C" b2sr_status b2sr_spgemm_bool(b2sr_handle A, b2sr_handle B, void* stream, b2sr_handle* C) {
    clear_error();
    if (!C) return fail(B2SR_ERR_INVALID_ARG, "C is NULL");
    *C = nullptr;
    B2SR_TRY(check_handle(A));
    B2SR_TRY(check_handle(B));
    if (A->n != B->n || A->k != B->k) return fail(B2SR_ERR_INVALID_ARG, "A and B need the same n and tile_dim");
    b2sr_matrix* out = nullptr;
    B2SR_TRY(spgemm_bool(A, B, to_stream(stream), &out));
    *C = out;
    return B2SR_OK;
}
