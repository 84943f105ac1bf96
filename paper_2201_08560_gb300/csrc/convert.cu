// CSR <-> B2SR conversion (Sec. III-A "Bit-tile Indexing System", Sec. III-B
// "Bit Packing", Table 1), the strictly-lower-triangle extraction used by
// triangle counting (Sec. V, TC), the weight side array, and the per-handle
// derived arrays (SpMV chunk schedule, set-bit offsets, column counts).
//
// Conversion: every entry (i, j) becomes the 64-bit key
//   (i/k) << (S+10) | (j/k) << 10 | ((j%k)*k + i%k)
// with S the bit width of a tile index.  Once the keys are in order, equal
// tiles are runs in (tile-row, tile-column) order, run heads become the tiles,
// and each entry ORs its bit into its tile.  When every CSR row is already in
// column order (the usual case) the k rows of a tile-row are k sorted runs.  At
// k = 4 and 8, without repeated entries, blocks merge them and build the tiles
// in shared memory, piece by piece; otherwise the keys are put in order by
// ranking each entry among its tile-row's rows (binary searches) and, at k =
// 16 and 32, merging groups of eight rows pairwise.  Rows in no order go
// through a radix sort on the tile part.  All replace the paper's cusparseXcsr2bsrNnz / cusparseScsr2bsr + packing kernels
// (Sec. III-B) and give the same three arrays.
#include <algorithm>
#include <mutex>

#include "b2sr_internal.cuh"

namespace b2sr {
b2sr_status row_counts(const b2sr_matrix* h, int32_t* cnt, int32_t* first, int32_t* last, bool chunks_done,
                       cudaStream_t s);

// ---------------------------------------------------------------------------
// input validation
// ---------------------------------------------------------------------------
__global__ void validate_csr_kernel(int32_t n, const int32_t* __restrict__ rowptr,
                                    const int32_t* __restrict__ colind, int64_t nnz,
                                    int* __restrict__ bad) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0 && (rowptr[0] != 0 || (int64_t)rowptr[n] != nnz)) atomicOr(bad, 1);
    for (int64_t i = tid; i < n; i += stride)
        if (rowptr[i + 1] < rowptr[i]) atomicOr(bad, 2);
    for (int64_t e = tid; e < nnz; e += stride) {
        int32_t c = colind[e];
        if (c < 0 || c >= n) atomicOr(bad, 4);
    }
}

// The validation b2sr_from_csr runs, which also finds whether every row is
// in column order.  Row pass: the rowptr checks of validate_csr_kernel, and
// in `starts` (one bit per entry) the entries that begin a row.
__global__ void validate_rows_kernel(int32_t n, const int32_t* __restrict__ rowptr, int64_t nnz,
                                     int* __restrict__ bad, uint32_t* __restrict__ starts) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0 && (rowptr[0] != 0 || (int64_t)rowptr[n] != nnz)) atomicOr(bad, 1);
    for (int64_t i = tid; i < n; i += stride) {
        const int32_t a = rowptr[i], b = rowptr[i + 1];
        if (b < a) atomicOr(bad, 2);
        if (a >= 0 && a < nnz) atomicOr(starts + (a >> 5), 1u << (a & 31));
    }
}

// Entry pass, four entries a step: every column in [0, n) (else bit 4 of
// *bad); bit 1 of *unsorted set if an entry that does not begin a row has a
// smaller column than the entry before it, bit 2 if it has the same.
__global__ void validate_entries_kernel(int32_t n, const int32_t* __restrict__ colind, int64_t nnz,
                                        const uint32_t* __restrict__ starts, int* __restrict__ bad,
                                        int* __restrict__ unsorted) {
    const int64_t groups = (nnz + 3) / 4;
    const bool vec = (reinterpret_cast<uintptr_t>(colind) & 15u) == 0;
    bool out = false, down = false, same = false;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e0 = g * 4;
        int32_t c[4];
        if (vec && e0 + 4 <= nnz) {
            const int4 v = __ldg(reinterpret_cast<const int4*>(colind) + g);
            c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] = e0 + q < nnz ? __ldg(colind + e0 + q) : 0;
        }
        const uint32_t sw = __ldg(starts + (e0 >> 5)) >> (e0 & 31);  // e0 % 4 == 0: one word holds all four
        int32_t prev = e0 > 0 ? __ldg(colind + e0 - 1) : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (e0 + q >= nnz) break;
            out |= c[q] < 0 || c[q] >= n;
            const bool inner = e0 + q > 0 && !((sw >> q) & 1u);
            down |= inner && prev > c[q];
            same |= inner && prev == c[q];
            prev = c[q];
        }
    }
    if (out) atomicOr(bad, 4);
    if (down) atomicOr(unsorted, 1);
    if (same) atomicOr(unsorted, 2);
}

// Sets *bad (device) non-zero if the CSR is malformed; stream-ordered, no sync.
b2sr_status validate_csr_async(int32_t n, const int32_t* rowptr, const int32_t* colind, int64_t nnz, int* bad,
                               cudaStream_t s) {
    validate_csr_kernel<<<grid_wide(std::max<int64_t>(n, nnz)), 256, 0, s>>>(n, rowptr, colind, nnz, bad);
    B2SR_LAUNCH_CHECK("validate_csr_kernel");
    return B2SR_OK;
}

// ---------------------------------------------------------------------------
// keys
// ---------------------------------------------------------------------------
// largest r in [lo, hi] with rowptr[r] <= e
__device__ __forceinline__ int32_t row_of(const int32_t* __restrict__ rowptr, int32_t lo, int32_t hi,
                                          int64_t e) {
    while (lo < hi) {
        int32_t mid = lo + (hi - lo + 1) / 2;
        if ((int64_t)__ldg(rowptr + mid) <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The entry-parallel kernels below give each thread kRankPer consecutive CSR
// entries.  A thread finds the row of its first entry by a binary search
// between the rows of its block's first and last entries (brow), then walks
// forward through rows as its entries cross them.
constexpr int kRankThreads = 256;
constexpr int kRankPer = 8;
constexpr int kRankEntries = kRankThreads * kRankPer;

// brow[b] = row of entry b * kRankEntries for every block b < nblocks, and
// brow[nblocks] = row of the last entry: one independent search per block, so
// that no block starts with a chain of dependent global loads.  The entries of
// block b lie in rows brow[b] .. brow[b+1].
__global__ void block_rows_kernel(int32_t n, const int32_t* __restrict__ rowptr, int64_t nnz, int64_t nblocks,
                                  int32_t* __restrict__ brow) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= nblocks;
         b += (int64_t)gridDim.x * blockDim.x)
        brow[b] = row_of(rowptr, 0, n - 1, b < nblocks ? b * kRankEntries : nnz - 1);
}

// The thread's entries [e0, e1) and the row holding e0: rows i with
// rowptr[i] <= e < rowptr[i+1] = re.  Returns false for a thread with none.
struct EntryRun {  // positions fit int32: the conversion takes nnz < 2^31
    int32_t e0, e1;
    int32_t i;
    int32_t rs, re;  // rowptr[i], rowptr[i+1]
};

// largest r in [lo, hi] with rowptr[r] <= e (int32 positions)
__device__ __forceinline__ int32_t row_of32(const int32_t* __restrict__ rowptr, int32_t lo, int32_t hi, int32_t e) {
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (__ldg(rowptr + mid) <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ bool entry_run(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ brow,
                                          int32_t n, int64_t nnz, EntryRun& u) {
    const int64_t e0 = ((int64_t)blockIdx.x * kRankThreads + threadIdx.x) * kRankPer;
    if (e0 >= nnz) return false;
    u.e0 = (int32_t)e0;
    u.e1 = (int32_t)min(e0 + kRankPer, nnz);
    u.i = row_of32(rowptr, __ldg(brow + blockIdx.x), __ldg(brow + blockIdx.x + 1), u.e0);
    u.rs = __ldg(rowptr + u.i);
    u.re = __ldg(rowptr + u.i + 1);
    return true;
}

// Moves u to the row holding entry e (e >= u.rs); true if the row changed.
// Never passes row n-1 (for a valid CSR, e < nnz lies in a row below n).
__device__ __forceinline__ bool advance_row(const int32_t* __restrict__ rowptr, int32_t n, int32_t e, EntryRun& u) {
    bool moved = false;
    while (e >= u.re && u.i + 1 < n) {
        ++u.i;
        u.rs = u.re;
        u.re = __ldg(rowptr + u.i + 1);
        moved = true;
    }
    return moved;
}

// k is a power of two: shifts and masks instead of divisions by a runtime k.
__device__ __forceinline__ uint64_t entry_key(int32_t i, int32_t j, int k, int sbits) {
    const int lk = __ffs(k) - 1;
    return ((uint64_t)(i >> lk) << (sbits + 10)) | ((uint64_t)(j >> lk) << 10) |
           (uint64_t)(((j & (k - 1)) << lk) | (i & (k - 1)));
}

__global__ void __launch_bounds__(kRankThreads) make_keys_kernel(int32_t n, const int32_t* __restrict__ rowptr,
                                                                 const int32_t* __restrict__ brow,
                                                                 const int32_t* __restrict__ colind,
                                                                 int64_t nnz, int k, int sbits,
                                                                 uint64_t* __restrict__ keys) {
    EntryRun u;
    if (!entry_run(rowptr, brow, n, nnz, u)) return;
    for (int32_t e = u.e0; e < u.e1; ++e) {
        advance_row(rowptr, n, e, u);
        keys[e] = entry_key(u.i, __ldg(colind + e), k, sbits);
    }
}

// Sorted rows: writes every entry's key straight to its place in the order of
// its group of G rows (G divides k, groups start at multiples of G).  The
// place is the group's first CSR position, plus the entry's offset in its own
// row, plus, for every other row q of the group, the entries of q ahead of it
// in (column, row) order: those with a smaller column, and those with the same
// column when q is an earlier row.  A thread's first entry in a row finds
// those counts by binary searches (advancing side by side, so that their loads
// overlap); its later entries in the row have columns no smaller, so each
// count moves forward from the last one by a galloping search.
template <int G>
__global__ void __launch_bounds__(kRankThreads) rank_keys_kernel(int32_t n, const int32_t* __restrict__ rowptr,
                                                                 const int32_t* __restrict__ brow,
                                                                 const int32_t* __restrict__ colind,
                                                                 int64_t nnz, int k, int sbits,
                                                                 uint64_t* __restrict__ keys) {
    EntryRun u;
    if (!entry_run(rowptr, brow, n, nnz, u)) return;
    // pos[q]: entries of row q of the group ahead of the current entry (from
    // base[q]); end[q]: the row's end.  The entry's own row keeps an empty
    // range.  An entry x of row q is ahead of column j when x < j + tie[q]:
    // the same column counts as ahead in an earlier row.
    int32_t pos[G], end[G], base[G];
    int tie[G];
    int32_t gstart = 0;
    bool fresh = true;
    for (int32_t e = u.e0; e < u.e1; ++e) {
        fresh |= advance_row(rowptr, n, e, u);
        const int32_t j = __ldg(colind + e);
        if (fresh) {
            const int rg = u.i % G;
            const int32_t g0 = u.i - rg;
            gstart = __ldg(rowptr + g0);
            int32_t hi[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int32_t iq = g0 + q;
                const bool live = q != rg && iq < n;
                pos[q] = live ? __ldg(rowptr + iq) : 0;
                end[q] = live ? __ldg(rowptr + iq + 1) : 0;
                base[q] = pos[q];
                hi[q] = end[q];
                tie[q] = q < rg ? 1 : 0;
            }
            // binary searches, side by side
            for (;;) {
                bool more = false;
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    if (pos[q] < hi[q]) {
                        const int32_t mid = pos[q] + ((hi[q] - pos[q]) >> 1);
                        if (__ldg(colind + mid) < j + tie[q]) pos[q] = mid + 1; else hi[q] = mid;
                        more = true;
                    }
                }
                if (!more) break;
            }
            fresh = false;
        } else {
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int32_t jq = j + tie[q];
                int32_t lo = pos[q], hi = end[q];
                if (lo >= hi || __ldg(colind + lo) >= jq) continue;  // nothing more of row q is ahead
                // gallop: entry lo is ahead; double the step until an entry is not
                int32_t step = 1, last = lo;
                while (hi - last > step) {
                    const int32_t probe = last + step;
                    if (__ldg(colind + probe) >= jq) { hi = probe; break; }
                    last = probe;
                    step <<= 1;
                }
                lo = last + 1;
                while (lo < hi) {
                    const int32_t mid = lo + ((hi - lo) >> 1);
                    if (__ldg(colind + mid) < jq) lo = mid + 1; else hi = mid;
                }
                pos[q] = lo;
            }
        }
        int32_t dest = gstart + (e - u.rs);
#pragma unroll
        for (int q = 0; q < G; ++q) dest += pos[q] - base[q];
        keys[dest] = entry_key(u.i, j, k, sbits);
    }
}

// One pairwise merge of sorted runs of `run` rows inside every tile-row (the
// runs a sorted-row conversion leaves when k > 8): each key moves to its
// offset in its own run plus the partner run's keys ahead of it (the left
// run wins ties).
__global__ void merge_runs_kernel(const uint64_t* __restrict__ src, uint64_t* __restrict__ dst, int64_t nnz,
                                  const int32_t* __restrict__ rowptr, int32_t n, int k, int run, int sbits) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = src[e];
        const int r = (int)(x & 1023u) & (k - 1);
        const int64_t rowL = (int64_t)(x >> (sbits + 10)) * k + (r & ~(2 * run - 1));
        const int64_t a0 = __ldg(rowptr + min(rowL, (int64_t)n));
        const int64_t m = __ldg(rowptr + min(rowL + run, (int64_t)n));
        const int64_t b1 = __ldg(rowptr + min(rowL + 2 * run, (int64_t)n));
        const bool right = (r & run) != 0;
        int64_t lo = right ? a0 : m, hi = right ? m : b1;
        const int64_t base = lo;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            uint64_t y = src[mid];
            if (y < x || (right && y == x)) lo = mid + 1; else hi = mid;
        }
        dst[a0 + (e - (right ? m : a0)) + (lo - base)] = x;
    }
}

// Keys in order -> tiles, in two passes over the keys.  A key whose tile
// (its bits above the low 10) differs from the previous key's is a run head:
// the first entry of a new tile.  Pass 1 counts the heads of every block of
// kFillTile keys; after an exclusive scan of those counts, pass 2 gives each
// key its tile index (the block's offset plus the heads before it), writes
// the column index of every new tile, points rowptr at the first tile of
// every tile-row that begins there, and ORs the bits of each run of keys that
// fall in one 32-bit word of the tile array in one atomic.
constexpr int kFillThreads = 256;
constexpr int kFillItems = 8;  // consecutive keys per thread
constexpr int kFillTile = kFillThreads * kFillItems;

// Loads keys base .. base+kFillItems-1 (those below N) and the key before base.
__device__ __forceinline__ void load_run(const uint64_t* __restrict__ keys, int64_t N, int64_t base,
                                         uint64_t (&key)[kFillItems], uint64_t& before) {
    before = base > 0 && base <= N ? __ldg(keys + base - 1) : 0ull;
    if (base + kFillItems <= N) {
        const ulonglong2* v = reinterpret_cast<const ulonglong2*>(keys + base);  // base is a multiple of 8 keys
#pragma unroll
        for (int q = 0; q < kFillItems / 2; ++q) {
            const ulonglong2 x = __ldg(v + q);
            key[2 * q] = x.x;
            key[2 * q + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < kFillItems; ++q) key[q] = base + q < N ? __ldg(keys + base + q) : 0ull;
    }
}

// Bit q of the result: key q of the run is a head.
__device__ __forceinline__ uint32_t run_heads(const uint64_t (&key)[kFillItems], uint64_t before, int64_t base,
                                              int64_t N) {
    uint32_t h = 0;
#pragma unroll
    for (int q = 0; q < kFillItems; ++q) {
        const uint64_t prev = q == 0 ? before : key[q - 1];
        if (base + q < N && (base + q == 0 || (key[q] >> 10) != (prev >> 10))) h |= 1u << q;
    }
    return h;
}

// Sum of v over the block; every thread gets it.  Also returns, in *excl,
// the sum over the threads before this one.
template <int THREADS>
__device__ __forceinline__ int block_scan(int v, int* excl) {
    __shared__ int warp_tot[THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        const int x = warp_tot[w];
        before += w < wid ? x : 0;
        total += x;
    }
    *excl = before + inc - v;
    return total;
}

__global__ void __launch_bounds__(kFillThreads) count_heads_kernel(const uint64_t* __restrict__ keys, int64_t N,
                                                                   int64_t* __restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kFillTile + (int64_t)threadIdx.x * kFillItems;
    uint64_t key[kFillItems], before;
    load_run(keys, N, base, key, before);
    int excl;
    const int total = block_scan<kFillThreads>(__popc(run_heads(key, before, base, N)), &excl);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Pass 2 for k <= 8, where a tile (one byte per row) is one 64-bit word:
// the block's keys come in coalesced through shared memory, its tiles and
// their column indices are built in shared memory and leave in coalesced
// stores.  Only a tile whose run of keys crosses a block boundary is ORed
// into global memory by atomics (from both sides).
__device__ __forceinline__ int fill_slot(int i) { return i + (i >> 4); }  // padding: no bank conflicts

__global__ void __launch_bounds__(kFillThreads) fill_small_tiles_kernel(const uint64_t* __restrict__ keys, int64_t N,
                                                                        const int64_t* __restrict__ block_off,
                                                                        int k, int sbits, int32_t ntr, int64_t T,
                                                                        int32_t* __restrict__ colind,
                                                                        int32_t* __restrict__ rowptr,
                                                                        uint32_t* __restrict__ tiles32) {
    __shared__ uint64_t s_key[kFillTile + kFillTile / 16];
    __shared__ unsigned long long s_tile[kFillTile];
    __shared__ int32_t s_col[kFillTile];
    const int64_t b0 = (int64_t)blockIdx.x * kFillTile;
    const int cnt = (int)min((int64_t)kFillTile, N - b0);
    {
        uint64_t v[kFillItems];  // all loads in flight before the first store
#pragma unroll
        for (int q = 0; q < kFillItems; ++q) {
            const int i = q * kFillThreads + threadIdx.x;
            v[q] = i < cnt ? __ldg(keys + b0 + i) : 0ull;
        }
#pragma unroll
        for (int q = 0; q < kFillItems; ++q) {
            const int i = q * kFillThreads + threadIdx.x;
            s_key[fill_slot(i)] = v[q];
            s_tile[i] = 0ull;
        }
    }
    __syncthreads();
    const int q0 = threadIdx.x * kFillItems;
    uint64_t key[kFillItems];
#pragma unroll
    for (int q = 0; q < kFillItems; ++q) key[q] = s_key[fill_slot(q0 + q)];
    const uint64_t before = threadIdx.x > 0 ? s_key[fill_slot(q0 - 1)] : (b0 > 0 ? __ldg(keys + b0 - 1) : 0ull);
    const uint32_t h = run_heads(key, before, b0 + q0, N);
    int excl;
    const int heads = block_scan<kFillThreads>(__popc(h), &excl);
    const int64_t boff = block_off[blockIdx.x];
    const uint64_t jmask = (1ull << sbits) - 1ull;
    const bool wide = k == 8;
    int lt = excl - 1;  // block-local tile of the run in progress (-1: a tile begun in an earlier block)
    uint64_t acc = 0;
    // A run that begins and ends among this thread's keys owns its tile: a
    // plain shared-memory store.  Runs cut by a thread boundary are ORed in.
    bool owned = false;
    uint64_t lastkey = 0;
    auto flush = [&](bool cut) {
        if (!acc) return;
        if (lt >= 0) {
            if (owned && !cut) s_tile[lt] = acc;
            else atomicOr(&s_tile[lt], (unsigned long long)acc);
        } else if (wide) {
            atomicOr(reinterpret_cast<unsigned long long*>(tiles32) + (boff - 1), (unsigned long long)acc);
        } else {
            atomicOr(tiles32 + (boff - 1), (uint32_t)acc);
        }
        acc = 0;
    };
#pragma unroll
    for (int q = 0; q < kFillItems; ++q) {
        if (q0 + q >= cnt) break;
        const uint64_t x = key[q];
        lastkey = x;
        if ((h >> q) & 1u) {
            flush(false);
            ++lt;
            owned = true;
            s_col[lt] = (int32_t)((x >> 10) & jmask);
            const int64_t I = (int64_t)(x >> (sbits + 10));
            const int64_t Ip = b0 + q0 + q == 0 ? -1 : (int64_t)((q == 0 ? before : key[q - 1]) >> (sbits + 10));
            for (int64_t R = Ip + 1; R <= I; ++R) rowptr[R] = (int32_t)(boff + lt);
        }
        const int p = (int)(x & 1023u);
        acc |= 1ull << ((p & (k - 1)) * 8 + (p >> (__ffs(k) - 1)));
        if (b0 + q0 + q == N - 1)  // tile-rows after the last entry's start at T
            for (int64_t R = (int64_t)(x >> (sbits + 10)) + 1; R <= ntr; ++R) rowptr[R] = (int32_t)T;
    }
    {
        // the last run goes on past this thread unless the next key starts a tile
        const int nq = q0 + kFillItems;
        const int last = min(kFillItems, cnt - q0) - 1;
        bool cut = false;
        if (last >= 0 && b0 + q0 + last + 1 < N) {
            const uint64_t nk = nq < cnt ? s_key[fill_slot(nq)] : __ldg(keys + b0 + q0 + last + 1);
            cut = (nk >> 10) == (lastkey >> 10);
        }
        flush(cut);
    }
    __syncthreads();
    // the block's last tile goes on into the next block unless the next key starts a tile
    const bool cut = b0 + cnt < N && (__ldg(keys + b0 + cnt) >> 10) == (s_key[fill_slot(cnt - 1)] >> 10);
    for (int i = threadIdx.x; i < heads; i += kFillThreads) {
        const int64_t t = boff + i;
        colind[t] = s_col[i];
        const unsigned long long v = s_tile[i];
        const bool shared_tile = cut && i == heads - 1;
        if (wide) {
            unsigned long long* t64 = reinterpret_cast<unsigned long long*>(tiles32);
            if (shared_tile) atomicOr(t64 + t, v); else t64[t] = v;
        } else {
            if (shared_tile) atomicOr(tiles32 + t, (uint32_t)v); else tiles32[t] = (uint32_t)v;
        }
    }
}

__global__ void __launch_bounds__(kFillThreads, 4) fill_tiles_kernel(const uint64_t* __restrict__ keys, int64_t N,
                                                                  const int64_t* __restrict__ block_off, int k,
                                                                  int sbits, int32_t ntr, int64_t T,
                                                                  int32_t* __restrict__ colind,
                                                                  int32_t* __restrict__ rowptr,
                                                                  uint32_t* __restrict__ tiles32) {
    const int64_t base = (int64_t)blockIdx.x * kFillTile + (int64_t)threadIdx.x * kFillItems;
    uint64_t key[kFillItems], before;
    load_run(keys, N, base, key, before);
    const uint32_t h = run_heads(key, before, base, N);
    int excl;
    block_scan<kFillThreads>(__popc(h), &excl);
    const int wb = word_bytes(k);
    const uint64_t jmask = (1ull << sbits) - 1ull;
    int64_t t = block_off[blockIdx.x] + excl - 1;  // the tile of the run in progress
    // k <= 8: a whole tile (one byte per row) fits one 64-bit register.  A tile
    // whose run of keys begins and ends in this thread is stored outright;
    // only the runs cut by a thread boundary need atomics.
    const bool whole = k <= 8;
    bool owned = false;  // the run in progress began in this thread
    uint64_t tacc = 0;
    int64_t accw = -1;
    uint32_t acc = 0;
    auto flush_tile = [&](bool cut) {
        if (k == 4) {
            if (owned && !cut) tiles32[t] = (uint32_t)tacc;
            else atomicOr(tiles32 + t, (uint32_t)tacc);
        } else {
            unsigned long long* t64 = reinterpret_cast<unsigned long long*>(tiles32);
            if (owned && !cut) t64[t] = tacc;
            else atomicOr(t64 + t, (unsigned long long)tacc);
        }
    };
    int last = -1;
    uint64_t lastkey = 0;
#pragma unroll
    for (int q = 0; q < kFillItems; ++q) {
        if (base + q >= N) break;
        last = q;
        const uint64_t x = key[q];
        lastkey = x;
        if ((h >> q) & 1u) {
            if (whole && q > 0) flush_tile(false);
            ++t;
            owned = true;
            tacc = 0;
            colind[t] = (int32_t)((x >> 10) & jmask);
            const int64_t I = (int64_t)(x >> (sbits + 10));
            const int64_t Ip = base + q == 0 ? -1 : (int64_t)((q == 0 ? before : key[q - 1]) >> (sbits + 10));
            for (int64_t R = Ip + 1; R <= I; ++R) rowptr[R] = (int32_t)t;
        }
        const int p = (int)(x & 1023u);
        const int r = p & (k - 1), c = p >> (__ffs(k) - 1);
        if (whole) {
            tacc |= 1ull << (r * 8 + c);
        } else {
            const int64_t byte = (t * k + r) * wb + (c >> 3);
            if ((byte >> 2) != accw) {
                if (accw >= 0) atomicOr(tiles32 + accw, acc);
                accw = byte >> 2;
                acc = 0;
            }
            acc |= 1u << ((int)(byte & 3) * 8 + (c & 7));
        }
        if (base + q == N - 1)  // tile-rows after the last entry's start at T
            for (int64_t R = (int64_t)(x >> (sbits + 10)) + 1; R <= ntr; ++R) rowptr[R] = (int32_t)T;
    }
    if (last < 0) return;
    if (whole) {
        // the last run goes on into the next thread unless the next key starts a tile
        const int64_t nx = base + last + 1;
        const bool cut = nx < N && (__ldg(keys + nx) >> 10) == (lastkey >> 10);
        flush_tile(cut);
    } else if (accw >= 0) {
        atomicOr(tiles32 + accw, acc);
    }
}

// ---------------------------------------------------------------------------
// rows in column order without repeats, k = 4 and 8: pieces merged in shared
// memory
// ---------------------------------------------------------------------------
// A piece is at most kPieceCap entries of whole tile-rows, or of one long
// tile-row's range of tile-columns.  The CSR entries are cut into windows of
// kWindow; a window's pieces are the tile-rows that begin in it, at most
// kPieceRows to a piece (a stretch of empty rows is shared by many blocks), and
// if the last of those is longer than kWindow (a long tile-row; its end lies
// past the window, so it is the last), its slices of about kSliceTarget entries.
// A block loads a piece, merges the k rows of each of its tile-rows pairwise in
// shared memory (log2 k levels; a thread finds where its eight outputs begin
// in the two runs by a binary search along their diagonal and merges from
// there), counts the run heads, and builds the tiles and their column indices
// there.  They leave in coalesced stores to the piece's place
// among the entries (a piece has at most as many tiles as entries); once the
// counts are scanned a second kernel moves them together.  Ranking every entry
// in global memory instead cost 393M warp instructions and 504 us on R-MAT 20
// at k = 4, and the 8-byte keys it wrote were read twice to build the tiles
// (187 us).  Merging and building takes 470 us there (300M instructions; the
// block's barriers and the merge's dependent shared loads bound it: 48 warps
// an SM, of which a piece of 1,100 entries keeps five in eight busy), finding
// the pieces 75 and moving the tiles together 80.
constexpr int kWindow = 1024;
constexpr int kPieceCap = 2048;
constexpr int kPieceRows = 4096;
constexpr int kSliceTarget = 1920;  // a slice is cut at a tile-column: up to k * k <= 64 entries more
constexpr int kPieceThreads = 256;
constexpr int kPieceItems = kPieceCap / kPieceThreads;

// First tile-row beginning at entry e or later (ntr if none).
__device__ __forceinline__ int32_t tile_row_from(const int32_t* __restrict__ rowptr, int32_t n, int32_t ntr, int k,
                                                 int64_t e) {
    int32_t lo = 0, hi = ntr;
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if ((int64_t)__ldg(rowptr + min((int64_t)mid * k, (int64_t)n)) < e) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Window b: first[b] = its first tile-row, slices[b] = the slices of its long
// tile-row (0: none), cnt[b] = its pieces.  Runs beside the validation: a malformed rowptr gives meaningless numbers, never an
// access out of range.
__global__ void windows_kernel(const int32_t* __restrict__ rowptr, int32_t n, int32_t ntr, int k, int64_t nwin,
                               int32_t* __restrict__ first, int32_t* __restrict__ slices,
                               int32_t* __restrict__ cnt) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= nwin;
         b += (int64_t)gridDim.x * blockDim.x) {
        if (b == nwin) {
            first[b] = ntr;
            slices[b] = 0;
            cnt[b] = 0;
            continue;
        }
        const int32_t f = tile_row_from(rowptr, n, ntr, k, b * kWindow);
        const int32_t g = b + 1 == nwin ? ntr : tile_row_from(rowptr, n, ntr, k, (b + 1) * kWindow);
        int32_t parts = 0;
        if (g > f) {
            const int64_t last = (int64_t)(g - 1) * k;
            const int32_t len = __ldg(rowptr + min(last + k, (int64_t)n)) - __ldg(rowptr + last);
            if (len > kWindow) parts = (len + kSliceTarget - 1) / kSliceTarget;
        }
        first[b] = f;
        slices[b] = parts;
        const int32_t rows = g - (parts > 0 ? 1 : 0) - f;
        cnt[b] = parts + (rows > 0 ? (rows + kPieceRows - 1) / kPieceRows : 0);
    }
}

// What a block needs of piece p: its window, and for a slice the position in
// each of the k rows where it begins (the next slice's, or the rows' ends, are
// where it ends).  A warp a piece: the cut is a search over tile-columns with a
// search of every row inside, a chain of loads, so 32/k tile-columns are tried
// side by side (R-MAT 20, k = 4: 74 us with one at a time, 48 so).
__global__ void pieces_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind, int32_t n,
                              int32_t ntr, int k, int64_t nwin, const int32_t* __restrict__ first,
                              const int32_t* __restrict__ parts, const int64_t* __restrict__ poff, int64_t npieces, int32_t* __restrict__ window,
                              int32_t* __restrict__ cut) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = (int)lane_id();
    const int q = lane & (k - 1), g = lane / k, tries = 32 / k;  // lane q of group g: row q, g-th tile-column
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < npieces; p += stride) {
        int64_t lo = 0, hi = nwin - 1;  // the last window whose pieces begin at or before p
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (__ldg(poff + mid) <= p) lo = mid; else hi = mid - 1;
        }
        if (lane == 0) window[p] = (int32_t)lo;
        const int64_t slices = __ldg(parts + lo);
        const int64_t slice = p - (__ldg(poff + lo + 1) - slices);
        if (slice < 0) continue;
        const int64_t row0 = (int64_t)(__ldg(first + lo + 1) - 1) * k;
        int32_t plo = __ldg(rowptr + min(row0 + q, (int64_t)n));
        if (slice > 0) {
            const int32_t start = __ldg(rowptr + row0);
            const int64_t len = __ldg(rowptr + min(row0 + k, (int64_t)n)) - start;
            const int64_t target = slice * len / slices;
            const int32_t r0 = plo;
            int32_t phi = __ldg(rowptr + min(row0 + q + 1, (int64_t)n));
            // the tile-column J with at most `target` entries before it, at most k * k short of it
            int32_t jlo = 0, jhi = ntr;
            while (jhi - jlo > 1) {
                const int32_t mid = jlo + (int32_t)((int64_t)(jhi - jlo) * (g + 1) / (tries + 1));
                int32_t a = plo, b = phi;
                while (a < b) {
                    const int32_t m = a + ((b - a) >> 1);
                    if ((int64_t)__ldg(colind + m) < (int64_t)mid * k) a = m + 1; else b = m;
                }
                __syncwarp();
                int32_t before = a - r0;
                for (int o = 1; o < k; o <<= 1) before += __shfl_xor_sync(FULL, before, o);
                const int below = __popc(__ballot_sync(FULL, before <= target)) / k;  // groups at or before the cut
                const int32_t a_lo = __shfl_sync(FULL, a, max(below - 1, 0) * k + q);
                const int32_t a_hi = __shfl_sync(FULL, a, min(below, tries - 1) * k + q);
                const int32_t j_lo = __shfl_sync(FULL, mid, max(below - 1, 0) * k);
                const int32_t j_hi = __shfl_sync(FULL, mid, min(below, tries - 1) * k);
                const int32_t at = __shfl_sync(FULL, before, max(below - 1, 0) * k);
                if (below < tries) {
                    jhi = j_hi;
                    phi = a_hi;
                }
                if (below > 0) {
                    jlo = j_lo;
                    plo = a_lo;
                    if (at >= target - k * k) break;
                }
            }
        }
        if (g == 0) cut[p * k + q] = plo;
    }
}

template <int K>
struct PieceTile {
    using type = typename std::conditional<K == 4, uint32_t, unsigned long long>::type;
};

template <int K>
__global__ void __launch_bounds__(kPieceThreads, K == 4 ? 6 : 5) merge_piece_kernel(
    const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind, int32_t n, const int32_t* __restrict__ first,
    const int32_t* __restrict__ parts, const int64_t* __restrict__ poff, const int32_t* __restrict__ window,
    const int32_t* __restrict__ cut,
    int32_t* __restrict__ trow_at, int32_t* __restrict__ count, int32_t* __restrict__ place, int32_t* __restrict__ col,
    typename PieceTile<K>::type* __restrict__ tile) {
    using Tile = typename PieceTile<K>::type;
    constexpr int LK = K == 4 ? 2 : 3;
    __shared__ __align__(16) uint32_t s_key[2][kPieceCap];  // column * K + row in tile
    __shared__ __align__(16) int32_t s_row[kPieceCap];      // row at the position, from the piece's first
    __shared__ __align__(16) Tile s_tile[kPieceCap];
    __shared__ int32_t s_off[K + 1];  // a slice's rows
    const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
    const int64_t p = blockIdx.x;
    const int32_t b = __ldg(window + p);
    const int32_t slices = __ldg(parts + b);
    const int64_t p0 = __ldg(poff + b + 1) - slices;  // the first slice
    const bool slice = p >= p0;
    const int32_t I0 = slice ? __ldg(first + b + 1) - 1
                             : __ldg(first + b) + (int32_t)(p - __ldg(poff + b)) * kPieceRows;
    const int32_t I1 = slice ? I0 + 1 : min(I0 + kPieceRows, __ldg(first + b + 1) - (slices > 0 ? 1 : 0));
    const int64_t row0 = (int64_t)I0 * K;
    const int32_t nrows = (int32_t)(min((int64_t)I1 * K, (int64_t)n) - row0);
    int32_t e0, cnt;
    if (slice) {
        if (threadIdx.x == 0) {
            const bool final = p == p0 + slices - 1;
            int32_t at = 0;
            int64_t before = 0;
            for (int q = 0; q < K; ++q) {
                const int32_t lo = __ldg(cut + p * K + q);
                const int32_t hi = final ? __ldg(rowptr + min(row0 + q + 1, (int64_t)n)) : __ldg(cut + (p + 1) * K + q);
                before += lo - __ldg(rowptr + min(row0 + q, (int64_t)n));
                s_off[q] = at;
                at += hi - lo;
            }
            s_off[K] = at;
            place[p] = __ldg(rowptr + row0) + (int32_t)before;
        }
        __syncthreads();
        cnt = s_off[K];
        e0 = 0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const int32_t lo = __ldg(cut + p * K + q), at = s_off[q], len = s_off[q + 1] - at;
            for (int32_t i = threadIdx.x; i < len; i += kPieceThreads) {
                s_key[0][at + i] = (uint32_t)__ldg(colind + lo + i) * K + q;
                s_row[at + i] = q;
            }
        }
    } else {
        e0 = __ldg(rowptr + min(row0, (int64_t)n));
        cnt = __ldg(rowptr + row0 + nrows) - e0;
        if (threadIdx.x == 0) place[p] = e0;
        uint32_t v[kPieceItems];  // all loads in flight before the rows are known
#pragma unroll
        for (int i = 0; i < kPieceItems; ++i) {
            const int32_t at = i * kPieceThreads + threadIdx.x;
            v[i] = at < cnt ? (uint32_t)__ldg(colind + e0 + at) * K : 0u;
        }
        constexpr int W = kPieceThreads / 32;  // neighbouring rows go to different warps
        for (int32_t r0 = warp; r0 < nrows; r0 += kPieceThreads) {
            const int32_t r = r0 + W * lane;
            int32_t a = 0, z = 0;
            if (r < nrows) {
                a = __ldg(rowptr + row0 + r) - e0;
                z = __ldg(rowptr + row0 + r + 1) - e0;
            }
            for (unsigned todo = __ballot_sync(0xffffffffu, z > a); todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const int32_t ra = __shfl_sync(0xffffffffu, a, src), rz = __shfl_sync(0xffffffffu, z, src);
                for (int32_t i = ra + lane; i < rz; i += 32) s_row[i] = r0 + W * src;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPieceItems; ++i) {
            const int32_t at = i * kPieceThreads + threadIdx.x;
            if (at < cnt) s_key[0][at] = v[i] + (uint32_t)(s_row[at] & (K - 1));
        }
    }
    for (int i = threadIdx.x; i < cnt; i += kPieceThreads) s_tile[i] = 0;
    __syncthreads();
    // merge level l: runs of 2^l rows, two by two; a thread makes the eight
    // outputs at its positions.  A position stays inside its tile-row (and its
    // pair of runs), so s_row says which pair it belongs to.
    const int32_t q0 = threadIdx.x * kPieceItems;
#pragma unroll
    for (int l = 0; l < LK; ++l) {
        const uint32_t* src = s_key[l & 1];
        uint32_t* dst = s_key[(l & 1) ^ 1];
        const int32_t q1 = min(q0 + kPieceItems, cnt);
        // the pair of runs [st, m) and [m, e) that holds position `at`
        int32_t st = 0, m = 0, e = 0;
        auto pair_of = [&](int32_t at) {
            const int32_t r = (s_row[at] >> (l + 1)) << (l + 1);
            if (slice) {
                st = s_off[r];
                m = s_off[r + (1 << l)];
                e = s_off[r + (2 << l)];
            } else {
                st = __ldg(rowptr + row0 + r) - e0;
                m = __ldg(rowptr + min(row0 + r + (1 << l), (int64_t)n)) - e0;
                e = __ldg(rowptr + min(row0 + r + (2 << l), (int64_t)n)) - e0;
            }
        };
        int32_t ia = 0, ib = 0;
        uint32_t ka = 0u, kb = 0u;
        auto heads_of = [&]() {
            ka = ia < m ? src[ia] : 0xFFFFFFFFu;  // above every key
            kb = ib < e ? src[ib] : 0xFFFFFFFFu;
        };
        if (q0 < q1) {
            pair_of(q0);
            const int32_t d = q0 - st;  // outputs before: how many of them from the first run?
            int32_t lo = max(0, d - (e - m)), hi = min(d, m - st);
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if (src[st + mid] < src[m + d - 1 - mid]) lo = mid + 1; else hi = mid;
            }
            ia = st + lo;
            ib = m + d - lo;
            heads_of();
        }
#pragma unroll
        for (int i = 0; i < kPieceItems; ++i) {
            const int32_t at = q0 + i;
            if (at < q1) {
                if (at == e) {  // the next pair begins here
                    pair_of(at);
                    ia = st;
                    ib = m;
                    heads_of();
                }
                const bool first_run = ka < kb;
                dst[at] = first_run ? ka : kb;
                const int32_t next = first_run ? ++ia : ++ib;
                const uint32_t k2 = next < (first_run ? m : e) ? src[next] : 0xFFFFFFFFu;
                if (first_run) ka = k2; else kb = k2;
            }
        }
        __syncthreads();
    }
    const uint32_t* keys = s_key[LK & 1];
    int32_t* s_col = reinterpret_cast<int32_t*>(s_key[(LK & 1) ^ 1]);
    // run heads, then tiles
    uint32_t key[kPieceItems];
    int32_t trow[kPieceItems];
    {
        const uint4 a = *reinterpret_cast<const uint4*>(keys + q0), c = *reinterpret_cast<const uint4*>(keys + q0 + 4);
        key[0] = a.x; key[1] = a.y; key[2] = a.z; key[3] = a.w;
        key[4] = c.x; key[5] = c.y; key[6] = c.z; key[7] = c.w;
        const int4 r = *reinterpret_cast<const int4*>(s_row + q0), t = *reinterpret_cast<const int4*>(s_row + q0 + 4);
        trow[0] = r.x >> LK; trow[1] = r.y >> LK; trow[2] = r.z >> LK; trow[3] = r.w >> LK;
        trow[4] = t.x >> LK; trow[5] = t.y >> LK; trow[6] = t.z >> LK; trow[7] = t.w >> LK;
    }
    const uint32_t key_before = q0 > 0 ? keys[q0 - 1] : 0u;
    const int32_t trow_before = q0 > 0 ? s_row[q0 - 1] >> LK : -1;
    uint32_t h = 0u;
#pragma unroll
    for (int q = 0; q < kPieceItems; ++q) {
        const uint32_t kp = q == 0 ? key_before : key[q - 1];
        const int32_t rp = q == 0 ? trow_before : trow[q - 1];
        if (q0 + q < cnt && (rp != trow[q] || (kp >> (2 * LK)) != (key[q] >> (2 * LK)))) h |= 1u << q;
    }
    int excl;
    const int heads = block_scan<kPieceThreads>(__popc(h), &excl);
    {
        int t = excl - 1;  // tile of the run in progress
        Tile acc = 0;
        bool owned = false;  // the run began in this thread
        auto flush = [&](bool ended) {
            if (!acc) return;
            if (owned && ended) s_tile[t] = acc;
            else atomicOr(&s_tile[t], acc);
            acc = 0;
        };
#pragma unroll
        for (int q = 0; q < kPieceItems; ++q) {
            if (q0 + q < cnt) {
                if ((h >> q) & 1u) {
                    flush(true);
                    ++t;
                    owned = true;
                    s_col[t] = (int32_t)(key[q] >> (2 * LK));
                    const int32_t rp = q == 0 ? trow_before : trow[q - 1];
                    if (!slice)
                        for (int32_t r = rp + 1; r <= trow[q]; ++r) trow_at[I0 + r] = t;
                }
                acc |= (Tile)1 << ((key[q] & (K - 1)) * 8 + ((key[q] >> LK) & (K - 1)));
            }
        }
        flush(false);
    }
    __syncthreads();
    if (!slice) {  // tile-rows after the last entry, or all of an empty piece
        const int32_t from = cnt > 0 ? (s_row[cnt - 1] >> LK) + 1 : 0;
        for (int32_t r = from + threadIdx.x; r < I1 - I0; r += kPieceThreads) trow_at[I0 + r] = heads;
    } else if (threadIdx.x == 0 && p == p0) {
        trow_at[I0] = 0;
    }
    if (threadIdx.x == 0) count[p] = heads;
    const int64_t to = slice ? place[p] : e0;
    for (int i = threadIdx.x; i < heads; i += kPieceThreads) {
        col[to + i] = s_col[i];
        tile[to + i] = s_tile[i];
    }
}

// Moves every piece's tiles to their final place and completes TileRowPtr
// (trow_at holds a tile-row's first tile counted from its piece's first).
template <int K>
__global__ void __launch_bounds__(kPieceThreads) gather_pieces_kernel(
    int32_t ntr, int64_t npieces, const int32_t* __restrict__ first, const int32_t* __restrict__ parts,
    const int64_t* __restrict__ poff, const int32_t* __restrict__ window, const int32_t* __restrict__ place, const int64_t* __restrict__ toff,
    const int32_t* __restrict__ col, const typename PieceTile<K>::type* __restrict__ tile, int32_t* __restrict__ rowptr,
    int32_t* __restrict__ colind, typename PieceTile<K>::type* __restrict__ tiles) {
    const int64_t p = blockIdx.x;
    const int32_t b = __ldg(window + p);
    const int32_t slices = __ldg(parts + b);
    const int64_t p0 = __ldg(poff + b + 1) - slices;  // the first slice
    const int64_t t0 = __ldg(toff + p);
    const int64_t cnt = __ldg(toff + p + 1) - t0, from = __ldg(place + p);
    const int32_t f1 = __ldg(first + b + 1);
    if (p < p0) {
        const int32_t I0 = __ldg(first + b) + (int32_t)(p - __ldg(poff + b)) * kPieceRows;
        const int32_t I1 = min(I0 + kPieceRows, f1 - (slices > 0 ? 1 : 0));
        for (int32_t I = I0 + threadIdx.x; I < I1; I += kPieceThreads) rowptr[I] += (int32_t)t0;
    } else if (p == p0 && threadIdx.x == 0) {
        rowptr[f1 - 1] += (int32_t)t0;
    }
    if (p == npieces - 1 && threadIdx.x == 0) rowptr[ntr] = (int32_t)(t0 + cnt);
    // four tiles a thread and step, all loads before the stores
    for (int64_t i0 = threadIdx.x; i0 < cnt; i0 += 4 * kPieceThreads) {
        int32_t c[4];
        typename PieceTile<K>::type w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * kPieceThreads;
            if (i < cnt) {
                c[q] = __ldg(col + from + i);
                w[q] = __ldg(tile + from + i);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * kPieceThreads;
            if (i < cnt) {
                colind[t0 + i] = c[q];
                tiles[t0 + i] = w[q];
            }
        }
    }
}

// Output arrays for T tiles; the padding after T is zeroed.
struct TileArrays {
    int32_t* rowptr = nullptr;
    int32_t* colind = nullptr;
    uint8_t* tiles = nullptr;
    int64_t cap = 0;
};

static b2sr_status merge_pieces(int32_t n, const int32_t* rowptr, const int32_t* colind, int64_t nnz, int k,
                                int32_t ntr, int64_t nwin, const int32_t* first, const int32_t* parts,
                                const int64_t* poff, int64_t npieces, cudaStream_t s, TileArrays* out, int64_t* T) {
    const int tb = tile_bytes(k);
    DevBuf info(s), tmp(s), toff(s);
    B2SR_TRY(info.alloc((size_t)npieces * (3 + k) * sizeof(int32_t) + sizeof(int32_t)));
    int32_t* window = info.as<int32_t>();
    int32_t* place = window + npieces;
    int32_t* count = place + npieces;           // npieces + 1
    int32_t* cut = count + npieces + 1;         // npieces * k
    B2SR_TRY(tmp.alloc((size_t)nnz * (tb + sizeof(int32_t))));
    uint8_t* tile = tmp.as<uint8_t>();          // 8-byte tiles first: aligned
    int32_t* col = reinterpret_cast<int32_t*>(tile + (size_t)nnz * tb);
    B2SR_TRY(toff.alloc((size_t)(npieces + 1) * sizeof(int64_t)));
    B2SR_TRY(dalloc(&out->rowptr, (size_t)ntr + 1, s));
    pieces_kernel<<<grid_wide(npieces * 32), 256, 0, s>>>(rowptr, colind, n, ntr, k, nwin, first, parts, poff, npieces, window,
                                                        cut);
    B2SR_LAUNCH_CHECK("pieces_kernel");
    B2SR_CUDA_TRY(cudaMemsetAsync(count + npieces, 0, sizeof(int32_t), s));
    if (k == 4)
        merge_piece_kernel<4><<<(unsigned)npieces, kPieceThreads, 0, s>>>(rowptr, colind, n, first, parts, poff, window, cut,
                                                                        out->rowptr, count, place, col,
                                                                        reinterpret_cast<uint32_t*>(tile));
    else
        merge_piece_kernel<8><<<(unsigned)npieces, kPieceThreads, 0, s>>>(rowptr, colind, n, first, parts, poff, window, cut,
                                                                        out->rowptr, count, place, col,
                                                                        reinterpret_cast<unsigned long long*>(tile));
    B2SR_LAUNCH_CHECK("merge_piece_kernel");
    B2SR_TRY(exclusive_scan_i32_to_i64(count, toff.as<int64_t>(), npieces + 1, s));
    B2SR_CUDA_TRY(cudaMemcpyAsync(T, toff.as<int64_t>() + npieces, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    out->cap = std::max<int64_t>(round_up(*T, kTilePad), kTilePad);
    B2SR_TRY(dalloc(&out->colind, (size_t)out->cap, s));
    B2SR_TRY(dalloc(&out->tiles, (size_t)out->cap * tb, s));
    B2SR_CUDA_TRY(cudaMemsetAsync(out->colind + *T, 0, (size_t)(out->cap - *T) * sizeof(int32_t), s));
    B2SR_CUDA_TRY(cudaMemsetAsync(out->tiles + *T * tb, 0, (size_t)(out->cap - *T) * tb, s));
    if (k == 4)
        gather_pieces_kernel<4><<<(unsigned)npieces, kPieceThreads, 0, s>>>(
            ntr, npieces, first, parts, poff, window, place, toff.as<int64_t>(), col, reinterpret_cast<const uint32_t*>(tile),
            out->rowptr, out->colind, reinterpret_cast<uint32_t*>(out->tiles));
    else
        gather_pieces_kernel<8><<<(unsigned)npieces, kPieceThreads, 0, s>>>(
            ntr, npieces, first, parts, poff, window, place, toff.as<int64_t>(), col,
            reinterpret_cast<const unsigned long long*>(tile), out->rowptr, out->colind,
            reinterpret_cast<unsigned long long*>(out->tiles));
    B2SR_LAUNCH_CHECK("gather_pieces_kernel");
    return B2SR_OK;
}

// ---------------------------------------------------------------------------
// schedule: tile-row of the first tile of every SpMV chunk, and the tile-rows
// that cross chunks
// ---------------------------------------------------------------------------
// The row R that chunk c begins inside, when R started in an earlier chunk
// and ends in c, goes to the split list: rows over at most kSplitShort chunks
// from the front, longer ones from the back (in no order: each is joined by
// itself).  meta: first and last tile-row with tiles, short and long rows, tiles
// of the longest of them.
__global__ void schedule_kernel(const int32_t* __restrict__ rowptr, int32_t ntr, int64_t T, int64_t CT,
                                int64_t nchunks, int32_t* __restrict__ chunk_row, int32_t* __restrict__ split,
                                int32_t* __restrict__ meta) {
    int32_t most = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= nchunks;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cs = min(c * CT, T - 1);
        const int32_t R = row_of(rowptr, 0, ntr - 1, cs);
        chunk_row[c] = R;
        if (c == 0) meta[0] = R;
        if (c == nchunks) meta[1] = R;
        if (c == 0 || c == nchunks) continue;
        const int64_t ce = min(cs + CT, T);
        const int64_t rs = rowptr[R], re = rowptr[R + 1];
        if (rs >= cs || re > ce) continue;
        most = max(most, (int32_t)(re - rs));
        const int64_t ca = rs / CT;
        const int64_t at = c - ca + 1 <= kSplitShort ? atomicAdd(meta + 2, 1) : nchunks - 1 - atomicAdd(meta + 3, 1);
        split[3 * at] = R;
        split[3 * at + 1] = (int32_t)ca;
        split[3 * at + 2] = (int32_t)c;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane_id() == 0 && most > 0) atomicMax(meta + 4, most);
}

b2sr_status build_schedule(b2sr_matrix* h, cudaStream_t s) {
    if (h->T == 0) {
        h->nchunks = 0;
        h->first_row = h->ntr;
        h->last_row = -1;
        return B2SR_OK;
    }
    const int64_t CT = chunk_tiles(h->k);
    h->nchunks = ceil_div(h->T, CT);
    B2SR_TRY(dalloc(&h->chunk_row, h->nchunks + 1, s));
    B2SR_TRY(dalloc(&h->split, 3 * h->nchunks, s));
    DevBuf meta(s);
    B2SR_TRY(meta.alloc(5 * sizeof(int32_t)));
    B2SR_CUDA_TRY(cudaMemsetAsync(meta.p, 0, 5 * sizeof(int32_t), s));
    schedule_kernel<<<grid_for(h->nchunks + 1), 256, 0, s>>>(h->rowptr, h->ntr, h->T, CT, h->nchunks, h->chunk_row,
                                                            h->split, meta.as<int32_t>());
    B2SR_LAUNCH_CHECK("schedule_kernel");
    int32_t got[5] = {0, 0, 0, 0, 0};
    B2SR_CUDA_TRY(cudaMemcpyAsync(got, meta.p, sizeof(got), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    h->first_row = got[0];
    h->last_row = got[1];
    h->nsplit_short = got[2];
    h->nsplit_long = got[3];
    h->most_tiles = got[4];
    return B2SR_OK;
}

b2sr_status new_handle_from_tiles(int32_t n, int k, int64_t T, int32_t* rowptr, int32_t* colind,
                                  uint8_t* tiles, int64_t cap, cudaStream_t s, b2sr_matrix** out, int64_t known_nnz) {
    b2sr_matrix* h = new b2sr_matrix();
    h->n = n;
    h->k = k;
    h->ntr = (int32_t)ceil_div(n, k);
    h->T = T;
    h->cap = cap;
    h->rowptr = rowptr;
    h->colind = colind;
    h->tiles = tiles;
    h->mtx = new std::mutex();
    cudaGetDevice(&h->device);
    auto cleanup = [&](b2sr_status st) {
        b2sr_destroy(h);
        return st;
    };
    // the SpMV and driver kernels index tiles with int32
    if (T >= (int64_t(1) << 31)) return cleanup(fail(B2SR_ERR_OOM, "more than 2^31 - 1 tiles"));
    DevBuf cnt(s);
    b2sr_status st = B2SR_OK;
    int64_t nnz = known_nnz;
    if (known_nnz < 0) {
        st = cnt.alloc(sizeof(int64_t));
        if (st != B2SR_OK) return cleanup(st);
        st = popcount_bytes(tiles, cap * tile_bytes(k), cnt.as<int64_t>(), s);
        if (st != B2SR_OK) return cleanup(st);
        cudaError_t e = cudaMemcpyAsync(&nnz, cnt.p, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return cleanup(cuda_fail(e, "copy nnz"));
        if (T == 0) {  // build_schedule does not wait for the copy then
            e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return cleanup(cuda_fail(e, "copy nnz"));
        }
    }
    st = build_schedule(h, s);  // synchronises s when there are tiles
    if (st != B2SR_OK) return cleanup(st);
    h->nnz = nnz;
    *out = h;
    return B2SR_OK;
}

// ---------------------------------------------------------------------------
// set-bit offsets and column counts (cached on the handle)
// ---------------------------------------------------------------------------
template <int K>
__device__ __forceinline__ uint32_t tile_word(const uint8_t* __restrict__ tiles, int64_t t, int r) {
    if (K == 32) return __ldg(reinterpret_cast<const uint32_t*>(tiles) + t * 32 + r);
    if (K == 16) return __ldg(reinterpret_cast<const uint16_t*>(tiles) + t * 16 + r);
    return __ldg(tiles + t * K + r);
}

template <int K>
__global__ void tile_popc_kernel(const uint8_t* __restrict__ tiles, int64_t T, int32_t* __restrict__ cnt) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T;
         t += (int64_t)gridDim.x * blockDim.x) {
        int c = 0;
#pragma unroll
        for (int r = 0; r < K; ++r) c += __popc(tile_word<K>(tiles, t, r));
        cnt[t] = c;
    }
}

__global__ void i64_to_i32_kernel(const int64_t* __restrict__ in, int64_t n, int32_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (int32_t)in[i];
}

// Column counts go to `copies` copies of the count array (warp w adds into
// copy w % copies), summed at the end: the hub columns' atomics spread over
// several addresses, and so over several L2 slices, instead of queueing on one.
constexpr int kDegCopies = 8;

__global__ void deg_sum_kernel(const int32_t* __restrict__ sub, int64_t stride, int copies, int64_t len,
                               int32_t* __restrict__ deg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t v = 0;
        for (int c = 0; c < copies; ++c) v += __ldg(sub + c * stride + i);
        deg[i] = v;
    }
}

// k = 4: four tiles (16 bytes of words, 16 of column indices) per thread and
// step; the padding after T is zero, so whole groups of four can be read.
// Column c of a tile word (row r in byte r) counts popc(w & (0x01010101 << c)).
__global__ void col_count4_kernel(const int32_t* __restrict__ colind, const uint8_t* __restrict__ tiles,
                                  int64_t groups, int32_t* __restrict__ sub, int64_t stride, int copies) {
    int32_t* __restrict__ deg = sub + (int64_t)((threadIdx.x >> 5) % copies) * stride;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups;
         g += (int64_t)gridDim.x * blockDim.x) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(tiles) + g);
        const int4 J = __ldg(reinterpret_cast<const int4*>(colind) + g);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
        const int32_t js[4] = {J.x, J.y, J.z, J.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int v = __popc(ws[q] & (0x01010101u << c));
                if (v) atomicAdd(deg + (int64_t)js[q] * 4 + c, v);
            }
        }
    }
}

template <int K>
__global__ void col_count_kernel(const int32_t* __restrict__ colind, const uint8_t* __restrict__ tiles,
                                 int64_t T, int32_t* __restrict__ sub, int64_t stride, int copies) {
    int32_t* __restrict__ deg = sub + (int64_t)((threadIdx.x >> 5) % copies) * stride;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t J = colind[t];
        uint32_t cols = 0;
        int per[K];
#pragma unroll
        for (int c = 0; c < K; ++c) per[c] = 0;
#pragma unroll
        for (int r = 0; r < K; ++r) {
            uint32_t w = tile_word<K>(tiles, t, r);
            cols |= w;
#pragma unroll
            for (int c = 0; c < K; ++c) per[c] += (w >> c) & 1u;
        }
        while (cols) {
            int c = __ffs(cols) - 1;
            cols &= cols - 1;
            int v = 0;
#pragma unroll
            for (int q = 0; q < K; ++q) v = (q == c) ? per[q] : v;
            atomicAdd(deg + J * K + c, v);
        }
    }
}

b2sr_status ensure_voff(b2sr_matrix* h, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(*static_cast<std::mutex*>(h->mtx));
    if (h->voff) return B2SR_OK;
    int32_t* voff = nullptr;
    B2SR_TRY(dalloc(&voff, h->T + 1, s));
    DevBuf cnt(s), scan(s);
    b2sr_status st = cnt.alloc((h->T + 1) * sizeof(int32_t));
    if (st == B2SR_OK) st = scan.alloc((h->T + 1) * sizeof(int64_t));
    if (st == B2SR_OK) {
        st = with_tile(h->k, [&](auto kc) -> b2sr_status {
            constexpr int K = decltype(kc)::value;
            if (h->T > 0) tile_popc_kernel<K><<<grid_wide(h->T), 256, 0, s>>>(h->tiles, h->T, cnt.as<int32_t>());
            B2SR_LAUNCH_CHECK("tile_popc_kernel");
            return B2SR_OK;
        });
    }
    if (st == B2SR_OK) {
        cudaMemsetAsync(cnt.as<int32_t>() + h->T, 0, sizeof(int32_t), s);
        st = exclusive_scan_i32_to_i64(cnt.as<int32_t>(), scan.as<int64_t>(), h->T + 1, s);
    }
    if (st == B2SR_OK) {
        i64_to_i32_kernel<<<grid_wide(h->T + 1), 256, 0, s>>>(scan.as<int64_t>(), h->T + 1, voff);
        note_launch();
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_fail(e, "voff");
    }
    if (st != B2SR_OK) {
        dfree(voff, s);
        return st;
    }
    h->voff = voff;
    return B2SR_OK;
}

b2sr_status ensure_outdeg(b2sr_matrix* h, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(*static_cast<std::mutex*>(h->mtx));
    if (h->outdeg) return B2SR_OK;
    const int64_t len = (int64_t)h->ntr * h->k;
    int32_t* deg = nullptr;
    B2SR_TRY(dalloc(&deg, (size_t)len, s));
    // copies while they stay under 1 GiB in all
    const int copies = (int)std::max<int64_t>(1, std::min<int64_t>(kDegCopies, (int64_t(1) << 30) / (len * 4 + 1)));
    DevBuf sub(s);
    b2sr_status st = sub.alloc((size_t)copies * len * sizeof(int32_t));
    if (st != B2SR_OK) { dfree(deg, s); return st; }
    cudaError_t e = cudaMemsetAsync(sub.p, 0, (size_t)copies * len * sizeof(int32_t), s);
    if (e != cudaSuccess) { dfree(deg, s); return cuda_fail(e, "memset outdeg"); }
    st = with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        if (h->T > 0 && K == 4)  // cap is a multiple of 512 tiles: groups of four stay inside the arrays
            col_count4_kernel<<<grid_wide(ceil_div(h->T, 4)), 256, 0, s>>>(h->colind, h->tiles, ceil_div(h->T, 4),
                                                                          sub.as<int32_t>(), len, copies);
        else if (h->T > 0)
            col_count_kernel<K><<<grid_wide(h->T), 256, 0, s>>>(h->colind, h->tiles, h->T, sub.as<int32_t>(), len,
                                                                copies);
        B2SR_LAUNCH_CHECK("col_count_kernel");
        deg_sum_kernel<<<grid_wide(len), 256, 0, s>>>(sub.as<int32_t>(), len, copies, len, deg);
        B2SR_LAUNCH_CHECK("deg_sum_kernel");
        return B2SR_OK;
    });
    if (st == B2SR_OK) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_fail(e, "outdeg");
    }
    if (st != B2SR_OK) { dfree(deg, s); return st; }
    h->outdeg = deg;
    return B2SR_OK;
}

// ---------------------------------------------------------------------------
// B2SR -> CSR
// ---------------------------------------------------------------------------
// Ones per row come from the row-count SpMV (spmv.cu) or csr_rows_kernel, which
// also leaves the partial counts of the tile-rows that cross chunks; a scan makes
// them row pointers.  The columns are then written by a warp per chunk of tiles,
// so a hub's row of 10^5 tiles is shared by many warps.  An entry's place is its
// row's pointer, plus the row's ones in earlier chunks (the partials), plus those
// in earlier tiles of the chunk.  Here a lane takes a tile, 32 tiles a step, and
// those are a carry from earlier steps and a scan over the lanes that restarts at
// every tile-row.
template <int K>
__global__ void __launch_bounds__(256) csr_fill_kernel(const int32_t* __restrict__ trp,
                                                       const int32_t* __restrict__ tci,
                                                       const uint8_t* __restrict__ tiles, int64_t T, int64_t nchunks,
                                                       const int32_t* __restrict__ chunk_row,
                                                       const int64_t* __restrict__ off,
                                                       const int32_t* __restrict__ first,
                                                       const int32_t* __restrict__ last,
                                                       int32_t* __restrict__ colind) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int CT = chunk_tiles(K);
    constexpr int H = K / 2;  // 16-bit counters, two a word (a chunk holds at most 2,048 ones of a row)
    __shared__ int32_t s_base[8][K];
    const int lane = (int)lane_id(), warp = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * 8 + warp;
    if (c >= nchunks) return;  // whole warps leave together
    const int32_t cs = (int32_t)(c * CT), ce = (int32_t)min((int64_t)cs + CT, T);
    const int32_t ra = __ldg(chunk_row + c), rb = __ldg(chunk_row + c + 1);
    // ones of tile-row ra in earlier chunks
    const int32_t rs = __ldg(trp + ra);
    {
        constexpr int L = 32 / K;  // lanes a row: lane l takes row l % K of every L-th chunk
        const int64_t ca = rs / CT;
        int32_t v = 0;
        if (rs < cs)
            for (int64_t q = ca + lane / K; q < c; q += L) v += __ldg((q == ca ? last : first) + q * K + lane % K);
#pragma unroll
        for (int o = K; o < 32; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane < K) s_base[warp][lane] = v;
    }
    __syncwarp();
    uint32_t carry[H];  // ones of tile-row crow in earlier steps
    int32_t crow = ra;
#pragma unroll
    for (int h = 0; h < H; ++h) carry[h] = 0u;
    for (int32_t g0 = cs; g0 < ce; g0 += 32) {
        const int32_t t = g0 + lane;
        const bool live = t < ce;
        int32_t lo = ra, hi = rb;  // the tile's row: the last one starting at or before t
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo + 1) >> 1);
            if (__ldg(trp + mid) <= t) lo = mid; else hi = mid - 1;
        }
        const int32_t I = lo;
        uint32_t row[K], inc[H];
#pragma unroll
        for (int r = 0; r < K; ++r) row[r] = live ? tile_word<K>(tiles, t, r) : 0u;
#pragma unroll
        for (int h = 0; h < H; ++h) inc[h] = __popc(row[2 * h]) | (__popc(row[2 * h + 1]) << 16);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t Io = __shfl_up_sync(FULL, I, d);
            const bool same = lane >= d && Io == I;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t o = __shfl_up_sync(FULL, inc[h], d);
                if (same) inc[h] += o;
            }
        }
        if (I == crow) {
#pragma unroll
            for (int h = 0; h < H; ++h) inc[h] += carry[h];
        }
        if (live) {
            const int32_t j0 = __ldg(tci + t) * K;
#pragma unroll
            for (int r = 0; r < K; ++r) {
                uint32_t b = row[r];
                if (!b) continue;
                const int32_t before = (int32_t)((inc[r / 2] >> (16 * (r & 1))) & 0xFFFFu) - __popc(b);
                int64_t at = __ldg(off + (int64_t)I * K + r) + before + (I == ra ? s_base[warp][r] : 0);
                do {
                    colind[at++] = j0 + __ffs(b) - 1;
                    b &= b - 1;
                } while (b);
            }
        }
        crow = __shfl_sync(FULL, I, 31);
#pragma unroll
        for (int h = 0; h < H; ++h) carry[h] = __shfl_sync(FULL, inc[h], 31);
    }
}

// k = 16 and 32: the lanes are the rows of a tile (two tiles a step at k = 16),
// so that the ones in earlier tiles are a running count in a register; a lane a
// tile scanned k counters a step over the lanes instead (16.6 M tiles of one
// entry, k = 32: 3.97 ms a call, 1.72 so; a thread a row 2.07).  FILL: writes the
// columns, of full tiles 32 neighbours at a time; else: counts the ones of the
// rows that begin and end in the chunk, and the partials of the others.
template <int K, bool FILL>
__global__ void __launch_bounds__(256) csr_rows_kernel(const int32_t* __restrict__ trp,
                                                       const int32_t* __restrict__ tci,
                                                       const uint8_t* __restrict__ tiles, int32_t n, int64_t T,
                                                       int64_t nchunks, const int32_t* __restrict__ chunk_row,
                                                       const int64_t* __restrict__ off, int32_t* __restrict__ cnt,
                                                       int32_t* __restrict__ first, int32_t* __restrict__ last,
                                                       int32_t* __restrict__ colind) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int CT = chunk_tiles(K);
    constexpr int SUBS = 32 / K;  // tiles a step
    constexpr int STEPS = 8;      // whose words are in flight together
    static_assert(K == 16 || K == 32, "one or two tiles a step");
    const int lane = (int)lane_id(), r = lane % K, sub = lane / K;
    const int64_t c = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= nchunks) return;  // whole warps leave together
    const int32_t cs = (int32_t)(c * CT), ce = (int32_t)min((int64_t)cs + CT, T);
    const int32_t ra = __ldg(chunk_row + c), rb = __ldg(chunk_row + c + 1);
    const int32_t rs = __ldg(trp + ra);
    const bool head = rs >= cs;  // tile-row ra begins with this chunk
    // FILL: the rows of a tile that this warp writes (the grid's y shares them out)
    const int row0 = (int)blockIdx.y * K / (int)gridDim.y, row1 = ((int)blockIdx.y + 1) * K / (int)gridDim.y;
    int32_t acc = 0;             // ones of lane's row so far
    int64_t at = 0;              // or the place of its next entry
    if constexpr (FILL) {
        int32_t v = 0;  // ones of the row in earlier chunks, every SUBS-th a lane
        const int64_t ca = rs / CT;
        if (!head)
            for (int64_t q = ca + sub; q < c; q += SUBS) v += __ldg((q == ca ? last : first) + q * K + r);
        if constexpr (SUBS == 2) v += __shfl_xor_sync(FULL, v, 16);
        at = __ldg(off + min((int64_t)ra * K + r, (int64_t)n)) + v;
    }
    int32_t before = ra;  // tile-row of the tile before the step's
    bool open = true;     // the last tile's row goes on in the next chunk
    for (int32_t g0 = cs; g0 < ce; g0 += 32) {
        const int32_t t = g0 + lane;
        int32_t lo = ra, hi = rb;  // the tile's row: the last one starting at or before t
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo + 1) >> 1);
            if (__ldg(trp + mid) <= t) lo = mid; else hi = mid - 1;
        }
        const int32_t I = lo;
        int32_t Ip = __shfl_up_sync(FULL, I, 1);
        if (lane == 0) Ip = before;
        before = __shfl_sync(FULL, I, 31);
        // FILL: tiles whose row is not that of the tile before; else: the last of their rows
        const uint32_t marks = __ballot_sync(FULL, t < ce && (FILL ? I != Ip : __ldg(trp + I + 1) == t + 1));
        int32_t j0 = 0;
        if constexpr (FILL) j0 = t < ce ? __ldg(tci + t) * K : 0;
        if (g0 + 32 >= ce) open = !((marks >> (ce - 1 - g0)) & 1u);
#pragma unroll 1
        for (int u0 = 0; u0 < min(32, ce - g0); u0 += SUBS * STEPS) {
            uint32_t b[STEPS];
            int64_t start[STEPS];
#pragma unroll
            for (int q = 0; q < STEPS; ++q) {
                const int u = u0 + q * SUBS + sub;
                b[q] = g0 + u < ce ? tile_word<K>(tiles, g0 + u, r) : 0u;
                start[q] = 0;
                if constexpr (FILL) {
                    const int32_t Iu = __shfl_sync(FULL, I, u);
                    if ((marks >> u) & 1u) start[q] = __ldg(off + min((int64_t)Iu * K + r, (int64_t)n));
                }
            }
#pragma unroll
            for (int q = 0; q < STEPS; ++q) {
                const int ua = u0 + q * SUBS;
                if constexpr (FILL) {
                    int64_t p = at;
                    if constexpr (SUBS == 1) {
                        if ((marks >> ua) & 1u) p = start[q];
                        at = p + __popc(b[q]);
                    } else {  // both halves follow both tiles
                        const int mine = __popc(b[q]), theirs = __shfl_xor_sync(FULL, mine, 16);
                        const int64_t other = __shfl_xor_sync(FULL, start[q], 16);
                        const int64_t pa = (marks >> ua) & 1u ? (sub ? other : start[q]) : at;
                        const int64_t pb = (marks >> (ua + 1)) & 1u ? (sub ? start[q] : other) : pa + (sub ? theirs : mine);
                        p = sub ? pb : pa;
                        at = pb + (sub ? mine : theirs);
                    }
                    const int32_t j = __shfl_sync(FULL, j0, ua + sub);
                    // rows of many entries, if they are most of the tile's or there are few: row
                    // by row, a lane a column
                    const uint32_t many = __ballot_sync(FULL, __popc(b[q]) > 8);
                    uint32_t some = __ballot_sync(FULL, b[q] != 0u);  // rows with entries
                    if constexpr (SUBS == 2) some = (some | (some >> 16)) & 0xFFFFu;
                    if (many != 0u && (__popc(many) >= 8 || __popc(some) <= 4)) {
                        auto write_row = [&](int i) {
                            const int from = sub * K + i;
                            const uint32_t w = __shfl_sync(FULL, b[q], from);
                            const int64_t pw = __shfl_sync(FULL, p, from);
                            if ((w >> r) & 1u) colind[pw + __popc(w & ((1u << r) - 1u))] = j + r;
                        };
                        if (__popc(some) <= 4) {
                            for (; some; some &= some - 1u) {
                                const int i = __ffs(some) - 1;
                                if (i >= row0 && i < row1) write_row(i);
                            }
                        } else {
#pragma unroll 8
                            for (int i = row0; i < row1; ++i) write_row(i);
                        }
                    } else {
                        for (uint32_t w = r >= row0 && r < row1 ? b[q] : 0u; w; w &= w - 1)
                            colind[p++] = j + __ffs(w) - 1;
                    }
                } else {
                    const int mine = __popc(b[q]), theirs = SUBS == 2 ? __shfl_xor_sync(FULL, mine, 16) : 0;
#pragma unroll
                    for (int h = 0; h < SUBS; ++h) {
                        acc += sub == h ? mine : theirs;
                        const int32_t Iu = __shfl_sync(FULL, I, ua + h);
                        if ((marks >> (ua + h)) & 1u) {  // the row ends
                            if (sub == 0) {
                                if (Iu == ra && !head) first[c * K + r] = acc;
                                else if ((int64_t)Iu * K + r < n) cnt[(int64_t)Iu * K + r] = acc;
                            }
                            acc = 0;
                        }
                    }
                }
            }
        }
    }
    if (!FILL && open && sub == 0) (ra == rb && !head ? first : last)[c * K + r] = acc;
}

__global__ void rowptr_out_kernel(const int64_t* __restrict__ off, int64_t len, int32_t* __restrict__ rowptr) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        rowptr[i] = (int32_t)off[i];
}

b2sr_status extract_csr(const b2sr_matrix* h, int64_t* off, int32_t* rowptr, int32_t* colind, cudaStream_t s) {
    const int32_t n = h->n;
    DevBuf cnt(s), part(s);
    B2SR_TRY(cnt.alloc(((size_t)n + 1) * sizeof(int32_t)));
    const size_t np = (size_t)h->nchunks * h->k;
    B2SR_TRY(part.alloc(std::max<size_t>(2 * np, 1) * sizeof(int32_t)));
    int32_t* first = part.as<int32_t>();
    int32_t* last = first + np;
    B2SR_CUDA_TRY(cudaMemsetAsync(cnt.p, 0, ((size_t)n + 1) * sizeof(int32_t), s));  // rows without tiles stay 0
    // k = 16 and 32: a kernel over the chunks' rows where tiles are an eighth full,
    // hardly a tile-row has one, or, at k = 32, the chunks outnumber the warps.  us,
    // rows / tiles: k = 16, 1 entry a tile 1078 / 903, 2.2 529 / 438, 9.8 104 / 104,
    // 43 150 / 156, 171 195 / 297, 256 123 / 213; 2,000 entries in 2^26 rows 563 /
    // 26,784; k = 32, 4,000 chunks and fewer 152 / 126, 8,000 218 / 254, 130,000
    // 1,719 / 3,967.
    const bool full = 8 * h->nnz >= (int64_t)h->k * h->k * h->T;
    const bool wide = h->k >= 16 && h->nchunks > 0 &&
                      (full || h->ntr > 32 * h->T || (h->k == 32 && h->nchunks >= 4096));
    auto wide_rows = [&](auto fill, const int64_t* row_start) -> b2sr_status {
        constexpr bool FILL = decltype(fill)::value;
        auto kernel = h->k == 16 ? csr_rows_kernel<16, FILL> : csr_rows_kernel<32, FILL>;
        // few chunks of full tiles (64 full tiles are 65,536 entries) are shared by four warps each
        const unsigned share = FILL && full && h->nchunks <= (int64_t)sm_count() * 16 ? 4 : 1;
        kernel<<<dim3((unsigned)ceil_div(h->nchunks, 8), share), 256, 0, s>>>(
            h->rowptr, h->colind, h->tiles, n, h->T, h->nchunks, h->chunk_row, row_start, cnt.as<int32_t>(), first, last,
            colind);
        B2SR_LAUNCH_CHECK("csr_rows_kernel");
        return B2SR_OK;
    };
    if (wide) B2SR_TRY(wide_rows(std::false_type(), nullptr));
    B2SR_TRY(row_counts(h, cnt.as<int32_t>(), first, last, wide, s));
    B2SR_TRY(exclusive_scan_i32_to_i64(cnt.as<int32_t>(), off, (int64_t)n + 1, s));
    rowptr_out_kernel<<<grid_wide((int64_t)n + 1), 256, 0, s>>>(off, (int64_t)n + 1, rowptr);
    B2SR_LAUNCH_CHECK("rowptr_out_kernel");
    if (!colind || h->nchunks == 0) return B2SR_OK;
    if (wide) return wide_rows(std::true_type(), off);
    return with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        csr_fill_kernel<K><<<(unsigned)ceil_div(h->nchunks, 8), 256, 0, s>>>(
            h->rowptr, h->colind, h->tiles, h->T, h->nchunks, h->chunk_row, off, first, last, colind);
        B2SR_LAUNCH_CHECK("csr_fill_kernel");
        return B2SR_OK;
    });
}

// ---------------------------------------------------------------------------
// strictly lower triangle
// ---------------------------------------------------------------------------
template <int K>
__device__ __forceinline__ uint32_t strict_lower_mask(int r) {  // columns c < r
    return r == 0 ? 0u : ((r >= 32) ? 0xffffffffu : ((1u << r) - 1u));
}

// A tile-row's tiles are in column order, so those strictly left of the
// diagonal are a prefix, found by one binary search; the diagonal tile, if
// present, follows it and keeps only its bits below the diagonal.
template <int K>
__device__ __forceinline__ bool diag_has_lower(const uint8_t* __restrict__ tiles, int64_t t) {
    uint32_t any = 0;
#pragma unroll
    for (int r = 0; r < K; ++r) any |= tile_word<K>(tiles, t, r) & strict_lower_mask<K>(r);
    return any != 0;
}

template <int K>
__global__ void lower_count_kernel(const int32_t* __restrict__ trp, const int32_t* __restrict__ tci,
                                   const uint8_t* __restrict__ tiles, int32_t ntr, int32_t* __restrict__ cnt,
                                   int32_t* __restrict__ pre) {
    for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < ntr;
         I += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t0 = __ldg(trp + I), t1 = __ldg(trp + I + 1);
        int32_t lo = t0, hi = t1;  // first tile with column >= I
        while (lo < hi) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(tci + mid) < I) lo = mid + 1; else hi = mid;
        }
        pre[I] = lo - t0;
        cnt[I] = lo - t0 + ((lo < t1 && __ldg(tci + lo) == I && diag_has_lower<K>(tiles, lo)) ? 1 : 0);
    }
}

// A warp per tile-row: the lanes copy the prefix tile by tile (coalesced),
// then lane 0 writes the masked diagonal tile.
template <int K>
__global__ void lower_fill_kernel(const int32_t* __restrict__ trp, const int32_t* __restrict__ tci,
                                  const uint8_t* __restrict__ tiles, int32_t ntr, const int64_t* __restrict__ off,
                                  const int32_t* __restrict__ pre, int32_t* __restrict__ lrp,
                                  int32_t* __restrict__ lci, uint8_t* __restrict__ ltiles) {
    constexpr int TB = K * (K <= 8 ? 1 : (K == 16 ? 2 : 4));  // bytes per tile
    constexpr int TW = (TB + 3) / 4;                            // 32-bit words per tile
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t I = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; I <= ntr; I += warps) {
        const int64_t o = off[I];
        if (lane == 0) lrp[I] = (int32_t)o;
        if (I == ntr) continue;
        const int32_t t0 = __ldg(trp + I), t1 = __ldg(trp + I + 1), np = pre[I];
        for (int32_t q = lane; q < np; q += 32) {
            lci[o + q] = __ldg(tci + t0 + q);
            if (TB >= 4) {
                const uint32_t* src = reinterpret_cast<const uint32_t*>(tiles) + (int64_t)(t0 + q) * TW;
                uint32_t* dst = reinterpret_cast<uint32_t*>(ltiles) + (o + q) * TW;
#pragma unroll
                for (int w = 0; w < TW; ++w) dst[w] = __ldg(src + w);
            }
        }
        const int32_t d = t0 + np;
        if (lane == 0 && d < t1 && __ldg(tci + d) == I && diag_has_lower<K>(tiles, d)) {
            const int64_t w = o + np;
            lci[w] = (int32_t)I;
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const uint32_t v = tile_word<K>(tiles, d, r) & strict_lower_mask<K>(r);
                if (K <= 8) ltiles[w * K + r] = (uint8_t)v;
                else if (K == 16) reinterpret_cast<uint16_t*>(ltiles)[w * K + r] = (uint16_t)v;
                else reinterpret_cast<uint32_t*>(ltiles)[w * K + r] = v;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// weights: CSR order -> set-bit order
// ---------------------------------------------------------------------------
template <int K>
__global__ void weights_kernel(int32_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                               const float* __restrict__ w_csr, int64_t nnz, const int32_t* __restrict__ trp,
                               const int32_t* __restrict__ tci, const uint8_t* __restrict__ tiles,
                               const int32_t* __restrict__ voff, float* __restrict__ w_bits,
                               int* __restrict__ bad) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = row_of(rowptr, 0, n - 1, e);
        int32_t j = colind[e];
        int32_t I = i / K, J = j / K;
        int r = i % K, c = j % K;
        int32_t lo = trp[I], hi = trp[I + 1] - 1;
        while (lo < hi) {
            int32_t mid = (lo + hi) / 2;
            if (tci[mid] < J) lo = mid + 1; else hi = mid;
        }
        if (lo > hi || tci[lo] != J) { atomicOr(bad, 1); continue; }
        int64_t t = lo;
        int before = 0;
        for (int q = 0; q < r; ++q) before += __popc(tile_word<K>(tiles, t, q));
        uint32_t word = tile_word<K>(tiles, t, r);
        before += __popc(word & ((1u << c) - 1u));
        w_bits[(int64_t)voff[t] + before] = w_csr[e];
    }
}

}  // namespace b2sr

using namespace b2sr;

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" b2sr_status b2sr_from_csr(int32_t n, const int32_t* rowptr, const int32_t* colind, int64_t nnz,
                                     int tile_dim, void* stream, b2sr_handle* out) {
    clear_error();
    if (!out) return fail(B2SR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!valid_tile(tile_dim)) return fail(B2SR_ERR_UNSUPPORTED_TILE, "tile_dim must be 4, 8, 16 or 32");
    if (n < 0 || nnz < 0 || nnz >= (int64_t(1) << 31)) return fail(B2SR_ERR_INVALID_ARG, "bad n or nnz");
    if (!rowptr || (nnz > 0 && !colind)) return fail(B2SR_ERR_INVALID_ARG, "null CSR pointer");
    cudaStream_t s = to_stream(stream);
    const int k = tile_dim;
    const int32_t ntr = (int32_t)ceil_div(n, k);
    const int sbits = bits_for(std::max<int64_t>(ntr, 2));
    if (2 * sbits + 10 > 64) return fail(B2SR_ERR_INVALID_ARG, "matrix too large");

    // validate; note whether every row is in column order
    bool sorted_rows = false, repeats = false;
    const int64_t blocks = ceil_div(nnz, kRankEntries);
    // rows in column order without repeats at k <= 8: pieces (32-bit keys)
    const bool small = k <= 8 && nnz > 0 && (int64_t)n * k < (int64_t(1) << 32);
    const int64_t nwin = ceil_div(std::max<int64_t>(nnz, 1), kWindow);
    int64_t npieces = 0;
    DevBuf brow(s), wbuf(s), poff(s);
    {
        DevBuf bad(s), starts(s);
        const size_t start_words = (size_t)ceil_div(std::max<int64_t>(nnz, 1), 32);
        B2SR_TRY(bad.alloc(2 * sizeof(int)));
        B2SR_TRY(starts.alloc(start_words * sizeof(uint32_t)));
        B2SR_CUDA_TRY(cudaMemsetAsync(bad.p, 0, 2 * sizeof(int), s));
        B2SR_CUDA_TRY(cudaMemsetAsync(starts.p, 0, start_words * sizeof(uint32_t), s));
        validate_rows_kernel<<<grid_wide((int64_t)n + 1), 256, 0, s>>>(n, rowptr, nnz, bad.as<int>(),
                                                                      starts.as<uint32_t>());
        B2SR_LAUNCH_CHECK("validate_rows_kernel");
        if (nnz > 0) {
            validate_entries_kernel<<<grid_wide(ceil_div(nnz, 4)), 256, 0, s>>>(
                n, colind, nnz, starts.as<uint32_t>(), bad.as<int>(), bad.as<int>() + 1);
            B2SR_LAUNCH_CHECK("validate_entries_kernel");
        }
        if (small) {
            B2SR_TRY(wbuf.alloc(3 * (size_t)(nwin + 1) * sizeof(int32_t)));
            B2SR_TRY(poff.alloc((size_t)(nwin + 1) * sizeof(int64_t)));
            int32_t* first = wbuf.as<int32_t>();
            int32_t* counts = first + 2 * (nwin + 1);
            windows_kernel<<<grid_wide(nwin + 1), 256, 0, s>>>(rowptr, n, ntr, k, nwin, first, first + nwin + 1, counts);
            B2SR_LAUNCH_CHECK("windows_kernel");
            B2SR_TRY(exclusive_scan_i32_to_i64(counts, poff.as<int64_t>(), nwin + 1, s));
            B2SR_CUDA_TRY(cudaMemcpyAsync(&npieces, poff.as<int64_t>() + nwin, sizeof(int64_t), cudaMemcpyDeviceToHost,
                                          s));
        }
        int hbad[2] = {0, 0};
        B2SR_CUDA_TRY(cudaMemcpyAsync(hbad, bad.p, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        if (hbad[0]) return fail(B2SR_ERR_INVALID_ARG, "malformed CSR (rowptr/colind/nnz inconsistent)");
        sorted_rows = (hbad[1] & 1) == 0;
        repeats = (hbad[1] & 2) != 0;
    }
    if (small && sorted_rows && !repeats) {
        TileArrays a;
        int64_t tiles = 0;
        const b2sr_status st = merge_pieces(n, rowptr, colind, nnz, k, ntr, nwin, wbuf.as<int32_t>(),
                                            wbuf.as<int32_t>() + nwin + 1, poff.as<int64_t>(), npieces, s, &a, &tiles);
        if (st != B2SR_OK) {
            dfree(a.rowptr, s); dfree(a.colind, s); dfree(a.tiles, s);
            return st;
        }
        b2sr_matrix* h = nullptr;
        B2SR_TRY(new_handle_from_tiles(n, k, tiles, a.rowptr, a.colind, a.tiles, a.cap, s, &h, nnz));
        *out = h;
        return B2SR_OK;
    }
    if (nnz > 0) {
        B2SR_TRY(brow.alloc((size_t)(blocks + 1) * sizeof(int32_t)));
        block_rows_kernel<<<grid_for(blocks + 1), 256, 0, s>>>(n, rowptr, nnz, blocks, brow.as<int32_t>());
        B2SR_LAUNCH_CHECK("block_rows_kernel");
    }

    // keys in (tile-row, tile-column) order -> heads -> tile index
    int64_t T = 0;
    DevBuf keys(s), ktmp(s), hsum(s), hoff(s);
    const int64_t fill_blocks = ceil_div(nnz, kFillTile);
    uint64_t* sorted = nullptr;
    if (nnz > 0) {
        B2SR_TRY(keys.alloc(nnz * sizeof(uint64_t)));
        B2SR_TRY(ktmp.alloc(nnz * sizeof(uint64_t)));
        const int32_t* br = brow.as<int32_t>();
        if (sorted_rows) {
            const int G = std::min(k, 8);
            if (G == 4)
                rank_keys_kernel<4><<<(unsigned)blocks, kRankThreads, 0, s>>>(n, rowptr, br, colind, nnz, k, sbits,
                                                                            keys.as<uint64_t>());
            else
                rank_keys_kernel<8><<<(unsigned)blocks, kRankThreads, 0, s>>>(n, rowptr, br, colind, nnz, k, sbits,
                                                                            keys.as<uint64_t>());
            B2SR_LAUNCH_CHECK("rank_keys_kernel");
            uint64_t* cur = keys.as<uint64_t>();
            uint64_t* oth = ktmp.as<uint64_t>();
            for (int run = G; run < k; run *= 2) {
                merge_runs_kernel<<<grid_wide(nnz), 256, 0, s>>>(cur, oth, nnz, rowptr, n, k, run, sbits);
                B2SR_LAUNCH_CHECK("merge_runs_kernel");
                std::swap(cur, oth);
            }
            sorted = cur;
        } else {
            make_keys_kernel<<<(unsigned)blocks, kRankThreads, 0, s>>>(n, rowptr, br, colind, nnz, k, sbits,
                                                                     keys.as<uint64_t>());
            B2SR_LAUNCH_CHECK("make_keys_kernel");
            B2SR_TRY(radix_sort_u64(keys.as<uint64_t>(), ktmp.as<uint64_t>(), nnz, 10, 10 + 2 * sbits, s, &sorted));
        }
        B2SR_TRY(hsum.alloc(fill_blocks * sizeof(int64_t)));
        B2SR_TRY(hoff.alloc(fill_blocks * sizeof(int64_t)));
        count_heads_kernel<<<(unsigned)fill_blocks, kFillThreads, 0, s>>>(sorted, nnz, hsum.as<int64_t>());
        B2SR_LAUNCH_CHECK("count_heads_kernel");
        B2SR_TRY(exclusive_scan_i64(hsum.as<int64_t>(), hoff.as<int64_t>(), fill_blocks, s));
        int64_t last[2] = {0, 0};
        B2SR_CUDA_TRY(cudaMemcpyAsync(&last[0], hoff.as<int64_t>() + fill_blocks - 1, sizeof(int64_t),
                                      cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaMemcpyAsync(&last[1], hsum.as<int64_t>() + fill_blocks - 1, sizeof(int64_t),
                                      cudaMemcpyDeviceToHost, s));
        B2SR_CUDA_TRY(cudaStreamSynchronize(s));
        T = last[0] + last[1];
    }

    // outputs
    const int64_t cap = std::max<int64_t>(round_up(T, kTilePad), kTilePad);
    int32_t* o_rowptr = nullptr;
    int32_t* o_colind = nullptr;
    uint8_t* o_tiles = nullptr;
    auto release = [&](b2sr_status st) {
        dfree(o_rowptr, s); dfree(o_colind, s); dfree(o_tiles, s);
        return st;
    };
    b2sr_status st = dalloc(&o_rowptr, (size_t)ntr + 1, s);
    if (st == B2SR_OK) st = dalloc(&o_colind, (size_t)cap, s);
    if (st == B2SR_OK) st = dalloc(&o_tiles, (size_t)cap * tile_bytes(k), s);
    if (st != B2SR_OK) return release(st);
    cudaError_t e = cudaMemsetAsync(o_colind, 0, (size_t)cap * sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(o_tiles, 0, (size_t)cap * tile_bytes(k), s);
    if (e != cudaSuccess) return release(cuda_fail(e, "memset outputs"));
    if (nnz > 0) {
        if (k <= 8)
            fill_small_tiles_kernel<<<(unsigned)fill_blocks, kFillThreads, 0, s>>>(
                sorted, nnz, hoff.as<int64_t>(), k, sbits, ntr, T, o_colind, o_rowptr,
                reinterpret_cast<uint32_t*>(o_tiles));
        else
            fill_tiles_kernel<<<(unsigned)fill_blocks, kFillThreads, 0, s>>>(sorted, nnz, hoff.as<int64_t>(), k,
                                                                             sbits, ntr, T, o_colind, o_rowptr,
                                                                             reinterpret_cast<uint32_t*>(o_tiles));
        note_launch();
        e = cudaGetLastError();
        if (e != cudaSuccess) return release(cuda_fail(e, "fill_tiles_kernel"));
    } else {
        e = cudaMemsetAsync(o_rowptr, 0, ((size_t)ntr + 1) * sizeof(int32_t), s);
        if (e != cudaSuccess) return release(cuda_fail(e, "memset rowptr"));
    }
    b2sr_matrix* h = nullptr;
    st = new_handle_from_tiles(n, k, T, o_rowptr, o_colind, o_tiles, cap, s, &h);
    if (st != B2SR_OK) return st;  // arrays released by the failed handle
    *out = h;
    return B2SR_OK;
}

extern "C" b2sr_status b2sr_to_csr(b2sr_handle h, int32_t* rowptr, int32_t* colind, int64_t* nnz_host,
                                   void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (!rowptr) return fail(B2SR_ERR_INVALID_ARG, "rowptr is NULL");
    cudaStream_t s = to_stream(stream);
    DevBuf off(s);
    B2SR_TRY(off.alloc(((size_t)h->n + 1) * sizeof(int64_t)));
    B2SR_TRY(extract_csr(h, off.as<int64_t>(), rowptr, colind, s));
    int64_t nnz = 0;
    B2SR_CUDA_TRY(cudaMemcpyAsync(&nnz, off.as<int64_t>() + h->n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    if (nnz_host) *nnz_host = nnz;
    return B2SR_OK;
}

extern "C" b2sr_status b2sr_lower(b2sr_handle h, void* stream, b2sr_handle* out) {
    clear_error();
    if (!out) return fail(B2SR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    B2SR_TRY(check_handle(h));
    cudaStream_t s = to_stream(stream);
    const int k = h->k;
    const int32_t ntr = h->ntr;
    DevBuf cnt(s), off(s), pre(s);
    B2SR_TRY(cnt.alloc(((size_t)ntr + 1) * sizeof(int32_t)));
    B2SR_TRY(off.alloc(((size_t)ntr + 1) * sizeof(int64_t)));
    B2SR_TRY(pre.alloc(((size_t)ntr + 1) * sizeof(int32_t)));
    B2SR_CUDA_TRY(cudaMemsetAsync(cnt.as<int32_t>() + ntr, 0, sizeof(int32_t), s));
    int64_t T = 0;
    B2SR_TRY(with_tile(k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        if (ntr > 0)
            lower_count_kernel<K><<<grid_wide(ntr), 256, 0, s>>>(h->rowptr, h->colind, h->tiles, ntr, cnt.as<int32_t>(),
                                                                 pre.as<int32_t>());
        B2SR_LAUNCH_CHECK("lower_count_kernel");
        return B2SR_OK;
    }));
    B2SR_TRY(exclusive_scan_i32_to_i64(cnt.as<int32_t>(), off.as<int64_t>(), (int64_t)ntr + 1, s));
    B2SR_CUDA_TRY(cudaMemcpyAsync(&T, off.as<int64_t>() + ntr, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    const int64_t cap = std::max<int64_t>(round_up(T, kTilePad), kTilePad);
    int32_t* lrp = nullptr;
    int32_t* lci = nullptr;
    uint8_t* lt = nullptr;
    auto release = [&](b2sr_status st) {
        dfree(lrp, s); dfree(lci, s); dfree(lt, s);
        return st;
    };
    b2sr_status st = dalloc(&lrp, (size_t)ntr + 1, s);
    if (st == B2SR_OK) st = dalloc(&lci, (size_t)cap, s);
    if (st == B2SR_OK) st = dalloc(&lt, (size_t)cap * tile_bytes(k), s);
    if (st != B2SR_OK) return release(st);
    cudaError_t e = cudaMemsetAsync(lci, 0, (size_t)cap * sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(lt, 0, (size_t)cap * tile_bytes(k), s);
    if (e != cudaSuccess) return release(cuda_fail(e, "memset lower"));
    st = with_tile(k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        lower_fill_kernel<K><<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div((int64_t)ntr + 1, 8),
                                                                                   (int64_t)sm_count() * 16)),
                               256, 0, s>>>(h->rowptr, h->colind, h->tiles, ntr, off.as<int64_t>(), pre.as<int32_t>(),
                                            lrp, lci, lt);
        B2SR_LAUNCH_CHECK("lower_fill_kernel");
        return B2SR_OK;
    });
    if (st != B2SR_OK) return release(st);
    b2sr_matrix* L = nullptr;
    B2SR_TRY(new_handle_from_tiles(h->n, k, T, lrp, lci, lt, cap, s, &L));
    *out = L;
    return B2SR_OK;
}

extern "C" b2sr_status b2sr_weights_from_csr(b2sr_handle h, const int32_t* rowptr, const int32_t* colind,
                                             const float* w_csr, float* w_bits, void* stream) {
    clear_error();
    B2SR_TRY(check_handle(h));
    if (h->nnz == 0) return B2SR_OK;
    if (!rowptr || !colind || !w_csr || !w_bits) return fail(B2SR_ERR_INVALID_ARG, "null pointer");
    cudaStream_t s = to_stream(stream);
    B2SR_TRY(ensure_voff(h, s));
    DevBuf bad(s);
    B2SR_TRY(bad.alloc(sizeof(int)));
    B2SR_CUDA_TRY(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    B2SR_TRY(with_tile(h->k, [&](auto kc) -> b2sr_status {
        constexpr int K = decltype(kc)::value;
        weights_kernel<K><<<grid_wide(h->nnz), 256, 0, s>>>(h->n, rowptr, colind, w_csr, h->nnz, h->rowptr,
                                                           h->colind, h->tiles, h->voff, w_bits, bad.as<int>());
        B2SR_LAUNCH_CHECK("weights_kernel");
        return B2SR_OK;
    }));
    int hbad = 0;
    B2SR_CUDA_TRY(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    B2SR_CUDA_TRY(cudaStreamSynchronize(s));
    if (hbad) return fail(B2SR_ERR_INVALID_ARG, "CSR does not match the handle");
    return B2SR_OK;
}
