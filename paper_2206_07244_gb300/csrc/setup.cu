// Setup, binning and scan kernels (Sec. 5 steps 1, 2, 4; Sec. 5.1, 5.3).
//
//  - setup_kernel: n_prod per output row (Sec. 5 step 1), written into the
//    int64 C.rpt array that later holds n_nz and then the row offsets
//    (the metadata reuse of Sec. 5.3), and the check of B's column order.
//    Work is split evenly over non-zeros, not over rows, so power-law rows
//    cannot stall a warp.
//  - bin_pass1_kernel: Algorithm 1. Per-bin counts of each warp in shared
//    memory (groups of same-bin lanes, found with __match_any_sync), one
//    global atomic per bin per block; also the maximum and the int64 total
//    of the sizes, and per-tile sums that the scan reuses.
//  - bin_pass2_kernel: Algorithm 2. Scatters row ids into one M-length
//    `bins` array at offsets the host computed from the pass-1 counts.
//  - scan kernels: exclusive sum of n_nz into C.rpt in place (Sec. 5.3),
//    from the tile sums of pass 1.
#include "common.cuh"
#include "internal.h"

namespace ops {

// Tiles of A's (or B's) non-zeros: a block takes a contiguous range of tiles,
// finds the row of its first entry once (all threads probe together: three
// rounds of loads for 16M rows) and then only steps forward through the row
// pointers. A tile's entries are loaded with unit stride and staged in
// shared memory; groups of `lanes` threads then reduce one row's part of the
// tile each. What bounds it: one 4-byte load and two row-pointer gathers per
// entry. (Before: every 2048-entry tile started with two binary searches by
// one thread and every thread loaded 8 neighbouring entries; 27-point
// stencil 128^3, 55.7M entries: 0.342 ms for n_prod and about 1.3 ms for the
// order check.)
constexpr int kTileBlock = 256;
constexpr int kTileItems = 8;
constexpr int kTileEntries = kTileBlock * kTileItems;

// Largest r in [lo, hi) with rpt[r] <= p (rpt[lo] <= p assumed), found by
// the whole block; every thread gets it.
__device__ __forceinline__ int64_t block_row_of(const void *rpt, int is64, int64_t lo, int64_t hi, int64_t p) {
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + kTileBlock - 1) / kTileBlock;
        const int64_t i = lo + static_cast<int64_t>(threadIdx.x) * step;
        const int below = __syncthreads_count(i < hi && ld_rpt(rpt, is64, i) <= p);
        lo += static_cast<int64_t>(below - 1) * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// What is left of a tile after kWalkSteps steps from row to row is not walked:
// its entries search their rows. Runs of empty rows in one tile are one
// block's: 8.4M of them in A 24.0 ms when walked and 2.1 ms this way (whole
// product), in B 9.5 and 0.17, 16.8M rows with 2,000 entries 44.5 and 2.4.
constexpr int kWalkSteps = 32;

// The entries [p0, t1) of A's tile that begins at t0, in the rows [row, row + n)
// of which the first begins at or before p0; s_len as in row_lengths. (One entry
// at a time, added by atomics: merging neighbours would cost the walk registers.)
template <bool FEAT>
__device__ __forceinline__ void sparse_tile_lengths(const Operands &op, int64_t *nprod, unsigned *maxlen,
                                                    unsigned *minlen, const RepWord *words, int64_t row, int n,
                                                    int64_t p0, int64_t t0, int64_t t1, const int *s_len) {
#pragma unroll 1
    for (int e = static_cast<int>(p0 - t0) + static_cast<int>(threadIdx.x); t0 + e < t1; e += kTileBlock) {
        const int64_t r = upper_bound_rpt(op.arpt, op.a64, row, row + n, t0 + e) - op.row0;
        unsigned len;
        if (words) {
            if ((words[r >> 5].fol >> (r & 31)) & 1u) continue;
            const int c = __ldg(op.acol + t0 + e);
            len = static_cast<unsigned>(ld_rpt(op.brpt, op.b64, c + 1) - ld_rpt(op.brpt, op.b64, c));
        } else {
            len = static_cast<unsigned>(s_len[e]);
        }
        atomicAdd(reinterpret_cast<unsigned long long *>(nprod + r), static_cast<unsigned long long>(len));
        if (FEAT) {
            atomicMax(maxlen + r, len);
            atomicMin(minlen + r, len);
        }
    }
}

// Threads that reduce one row's part of a tile: a quarter of the mean row
// length, so that a mean row takes about four steps and a tile of short rows
// about as many rounds as its rows over the block.
__device__ __forceinline__ int lanes_per_row(int64_t entries, int64_t rows) {
    int l = 1;
    while (l < 32 && static_cast<int64_t>(l) * 4 * rows < entries) l <<= 1;
    return l;
}

// Block `blk` of `nblk`: lengths of the B rows that A's entries in the
// window reference, reduced per row: the sum into nprod and, with FEAT, the
// largest and smallest into maxlen / minlen (all set to their neutral value
// before). WORDS: the repeating rows are left out, and the entries of the others
// are not staged (most of the tile is not read). A row inside one tile is stored
// by one thread, a row cut by a tile's edge is combined with atomics.
template <bool FEAT, bool WORDS>
__device__ __forceinline__ void row_lengths(const Operands &op, int64_t *nprod, unsigned *maxlen, unsigned *minlen,
                                            const RepWord *words, int blk, int nblk, int *s_len) {
    const int64_t lo = op.row0, hi = op.row0 + op.mw;
    const int64_t pb = ld_rpt(op.arpt, op.a64, lo), pe = ld_rpt(op.arpt, op.a64, hi);
    const int64_t tiles = (pe - pb + kTileEntries - 1) / kTileEntries;
    const int64_t per = (tiles + nblk - 1) / nblk;
    const int64_t first = per * blk, last = first + per < tiles ? first + per : tiles;
    if (first >= last) return;
    const int L = lanes_per_row(pe - pb, op.mw);
    const int rows_per = kTileBlock / L, g = threadIdx.x / L, l = threadIdx.x % L;
    int64_t row = block_row_of(op.arpt, op.a64, lo, hi, pb + first * kTileEntries);
    for (int64_t t = first; t < last; ++t) {
        const int64_t t0 = pb + t * kTileEntries, t1 = t0 + kTileEntries < pe ? t0 + kTileEntries : pe;
        __syncthreads();   // readers of the previous tile are done
        int k[kTileItems];
#pragma unroll
        for (int j = 0; j < kTileItems; ++j) {
            const int64_t p = t0 + j * kTileBlock + threadIdx.x;
            k[j] = !WORDS && p < t1 ? __ldg(op.acol + p) : -1;
        }
#pragma unroll
        for (int j = 0; j < kTileItems; ++j)
            if (k[j] >= 0)
                s_len[j * kTileBlock + threadIdx.x] =
                    static_cast<int>(ld_rpt(op.brpt, op.b64, k[j] + 1) - ld_rpt(op.brpt, op.b64, k[j]));
        __syncthreads();
        for (int step = 1;; ++step, row += rows_per) {
            const int64_t i = row + g;
            long long sum = 0;
            unsigned mx = 0, mn = UINT_MAX;
            int64_t s = t1, e = t1;
            if (i < hi) {
                s = ld_rpt(op.arpt, op.a64, i);
                e = ld_rpt(op.arpt, op.a64, i + 1);
            }
            const int a = static_cast<int>((s > t0 ? s : t0) - t0), b = static_cast<int>((e < t1 ? e : t1) - t0);
            bool own = s < t1 && !(WORDS && ((words[(i - lo) >> 5].fol >> ((i - lo) & 31)) & 1u));
            // A piece of more than 32 steps of its row's threads (hub rows among
            // short ones) is the whole warp's: tridiagonal matrix of 2^17 rows with
            // a full last row 236 us for n_prod, now 33; n = 2^20 522 and 117. (The
            // check costs a walk without such rows 4%: 27-point stencil 128^3 164 us,
            // now 171.)
            for (unsigned many = __ballot_sync(0xffffffffu, own && l == 0 && b - a > 32 * L && L < 32); many;
                 many &= many - 1) {
                const int src = __ffs(many) - 1, lane = threadIdx.x & 31;
                const int a1 = __shfl_sync(0xffffffffu, a, src), b1 = __shfl_sync(0xffffffffu, b, src);
                long long total = 0;
                unsigned most = 0, least = UINT_MAX;
                for (int q = a1 + lane; q < b1; q += 32) {
                    int len;
                    if (WORDS) {
                        const int c = __ldg(op.acol + t0 + q);
                        len = static_cast<int>(ld_rpt(op.brpt, op.b64, c + 1) - ld_rpt(op.brpt, op.b64, c));
                    } else {
                        len = s_len[q];
                    }
                    total += len;
                    if (FEAT) {
                        most = max(most, static_cast<unsigned>(len));
                        least = min(least, static_cast<unsigned>(len));
                    }
                }
                for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
                if (FEAT) {
                    most = __reduce_max_sync(0xffffffffu, most);
                    least = __reduce_min_sync(0xffffffffu, least);
                }
                if (lane == src) {
                    atomicAdd(reinterpret_cast<unsigned long long *>(nprod + (i - lo)),
                              static_cast<unsigned long long>(total));
                    if (FEAT) {
                        atomicMax(maxlen + (i - lo), most);
                        atomicMin(minlen + (i - lo), least);
                    }
                }
                if (lane / L == src / L) own = false;
            }
            if (own)
                for (int q = a + l; q < b; q += L) {
                    int len;
                    if (WORDS) {
                        const int c = __ldg(op.acol + t0 + q);
                        len = static_cast<int>(ld_rpt(op.brpt, op.b64, c + 1) - ld_rpt(op.brpt, op.b64, c));
                    } else {
                        len = s_len[q];
                    }
                    sum += len;
                    if (FEAT) {
                        mx = max(mx, static_cast<unsigned>(len));
                        mn = min(mn, static_cast<unsigned>(len));
                    }
                }
            for (int o = __any_sync(0xffffffffu, own) ? L >> 1 : 0; o > 0; o >>= 1) {
                sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (FEAT) {
                    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                }
            }
            if (l == 0 && own && a < b) {
                const int64_t r = i - lo;
                if (s >= t0 && e <= t1) {
                    nprod[r] = sum;
                    if (FEAT) {
                        maxlen[r] = mx;
                        minlen[r] = mn;
                    }
                } else {
                    atomicAdd(reinterpret_cast<unsigned long long *>(nprod + r), static_cast<unsigned long long>(sum));
                    if (FEAT) {
                        atomicMax(maxlen + r, mx);
                        atomicMin(minlen + r, mn);
                    }
                }
            }
            // stop at the batch that reaches the end of the tile; the next
            // tile starts in its last row that begins at or before the end
            const int64_t next = row + rows_per;
            const bool stop = next >= hi || ld_rpt(op.arpt, op.a64, next) >= t1;   // uniform
            if (stop) {
                const int begun = __syncthreads_count(l == 0 && i < hi && s <= t1);
                row += begun - 1;
                break;
            }
            if (step == kWalkSteps) {
                row = block_row_of(op.arpt, op.a64, next, hi, t1);
                sparse_tile_lengths<FEAT>(op, nprod, maxlen, minlen, WORDS ? words : nullptr, next, static_cast<int>(row - next + 1),
                                          ld_rpt(op.arpt, op.a64, next), t0, t1, s_len);
                break;
            }
        }
    }
}

// Is every row of B sorted by column (bit 0 of flags set when not), and
// are its columns distinct (bit 1 set when a row repeats a column)? The
// column-window kernels need non-decreasing rows; the numeric hash kernels
// update values without atomics when the columns of every B row are
// distinct. Neighbouring entries are compared unless the second one starts a
// row (a byte per entry of the tile, set from the row pointers).
__device__ __forceinline__ void order_check(const Operands &op, int64_t brows, int64_t bnnz, Counters *cnt, int blk,
                                            int nblk, unsigned char *s_start) {
    const int64_t tiles = (bnnz + kTileEntries - 1) / kTileEntries;
    const int64_t per = (tiles + nblk - 1) / nblk;
    const int64_t first = per * blk, last = first + per < tiles ? first + per : tiles;
    if (first >= last) return;
    bool bad = false, dup = false;
    int64_t row = block_row_of(op.brpt, op.b64, 0, brows, first * kTileEntries);
    for (int64_t t = first; t < last; ++t) {
        const int64_t t0 = t * kTileEntries, t1 = t0 + kTileEntries < bnnz ? t0 + kTileEntries : bnnz;
        __syncthreads();   // readers of the previous tile are done
        for (int i = threadIdx.x; i < kTileEntries / 4 + 1; i += kTileBlock) reinterpret_cast<unsigned *>(s_start)[i] = 0u;
        int c0[kTileItems], c1[kTileItems];
#pragma unroll
        for (int j = 0; j < kTileItems; ++j) {
            const int64_t e = t0 + j * kTileBlock + threadIdx.x;
            c0[j] = e < t1 ? __ldg(op.bcol + e) : 0;
            c1[j] = e + 1 < bnnz && e < t1 ? __ldg(op.bcol + e + 1) : INT_MAX;
        }
        __syncthreads();
        bool sparse = true;
        for (int step = 0; step < kWalkSteps; ++step, row += kTileBlock) {   // row starts in (t0, t1]
            const int64_t i = row + threadIdx.x;
            const int64_t s = i < brows ? ld_rpt(op.brpt, op.b64, i) : INT64_MAX;
            if (s > t0 && s <= t1) s_start[s - t0] = 1;
            const int64_t next = row + kTileBlock;
            const bool stop = next >= brows || ld_rpt(op.brpt, op.b64, next) > t1;   // uniform
            if (stop) {
                const int begun = __syncthreads_count(s <= t1);
                row += begun - 1;
                sparse = false;
                break;
            }
        }
        if (sparse) {
            // the starts from row `row` on are searched for
            const int64_t end = block_row_of(op.brpt, op.b64, row, brows, t1);
#pragma unroll 1
            for (int e = static_cast<int>(ld_rpt(op.brpt, op.b64, row) - t0) + static_cast<int>(threadIdx.x); t0 + e <= t1;
                 e += kTileBlock) {
                const int64_t r = upper_bound_rpt(op.brpt, op.b64, row, end + 1, t0 + e);
                if (ld_rpt(op.brpt, op.b64, r) == t0 + e) s_start[e] = 1;
            }
            __syncthreads();
            row = end;
#pragma unroll 1
            for (int e = threadIdx.x; t0 + e < t1 && t0 + e + 1 < bnnz; e += kTileBlock) {
                const int a = __ldg(op.bcol + t0 + e), b = __ldg(op.bcol + t0 + e + 1);
                if (b <= a && !s_start[e + 1]) {
                    bad |= b < a;
                    dup |= b == a;
                }
            }
            continue;
        }
#pragma unroll
        for (int j = 0; j < kTileItems; ++j)
            if (c1[j] <= c0[j] && !s_start[j * kTileBlock + threadIdx.x + 1]) {
                bad |= c1[j] < c0[j];
                dup |= c1[j] == c0[j];
            }
    }
    const bool any_bad = __any_sync(0xffffffffu, bad), any_dup = __any_sync(0xffffffffu, dup);
    if ((threadIdx.x & 31u) == 0 && (any_bad || any_dup))
        atomicOr(&cnt->flags, (any_bad ? 1ull : 0ull) | (any_dup ? 2ull : 0ull));
}

// Both scans in one launch: the first `nprod_blocks` blocks count products,
// the others check B's order (either part may have no blocks). WORDS: with
// repeating rows; the two walks are apart because one that decides at run time
// keeps the registers of both (27-point stencil 128^3 174 us, now 155). Five
// blocks on an SM, 48 registers: at six the searches of sparse tiles spill into
// the walk (160 us).
template <bool WORDS>
__global__ void __launch_bounds__(kTileBlock, 5)
setup_kernel(Operands op, int64_t *nprod, const RepWord *words, RepGate gate, bool only_open, int nprod_blocks,
             int64_t brows, int64_t bnnz, Counters *cnt) {
    __shared__ int s_len[kTileEntries + 4];
    if (static_cast<int>(blockIdx.x) < nprod_blocks) {
        const bool shut = gate.shut();
        if (shut && only_open) return;   // uniform over the block
        if (WORDS && !shut) row_lengths<false, WORDS>(op, nprod, nullptr, nullptr, words, blockIdx.x, nprod_blocks, s_len);
        else row_lengths<false, false>(op, nprod, nullptr, nullptr, nullptr, blockIdx.x, nprod_blocks, s_len);
    } else
        order_check(op, brows, bnnz, cnt, blockIdx.x - nprod_blocks, gridDim.x - nprod_blocks,
                    reinterpret_cast<unsigned char *>(s_len));
}

__global__ void __launch_bounds__(kTileBlock, 5)
feature_scan_kernel(Operands op, int64_t *nprod, unsigned *maxlen, unsigned *minlen, RepGate gate) {
    __shared__ int s_len[kTileEntries];
    if (gate.found && !gate.shut()) return;   // uniform over the grid
    row_lengths<true, false>(op, nprod, maxlen, minlen, nullptr, blockIdx.x, gridDim.x, s_len);
}

// Blocks for `entries` entries: at most `grid`, no more than there are tiles.
static int tile_grid(int64_t entries, int grid) {
    const int64_t tiles = (entries + kTileEntries - 1) / kTileEntries;
    return static_cast<int>(tiles < 1 ? 1 : (tiles < grid ? tiles : grid));
}

cudaError_t launch_setup(const Operands &op, int64_t annz, int64_t *nprod, int64_t brows, int64_t bnnz,
                         Counters *cnt, int grid, cudaStream_t s, const RepWord *words, const RepGate &gate,
                         bool only_open) {
    const int na = nprod && op.mw > 0 ? tile_grid(annz, grid) : 0;
    const int nb = cnt && bnnz > 1 && brows > 0 ? tile_grid(bnnz, grid) : 0;
    if (na + nb == 0) return cudaSuccess;
    const auto kernel = words ? &setup_kernel<true> : &setup_kernel<false>;
    kernel<<<na + nb, kTileBlock, 0, s>>>(op, nprod, words, gate, only_open, na, brows, bnnz, cnt);
    return cudaGetLastError();
}

cudaError_t launch_feature_scan(const Operands &op, int64_t annz, int64_t *nprod, unsigned *maxlen, unsigned *minlen,
                                int grid, cudaStream_t s, const RepGate &gate) {
    if (op.mw <= 0) return cudaSuccess;
    feature_scan_kernel<<<tile_grid(annz, grid), kTileBlock, 0, s>>>(op, nprod, maxlen, minlen, gate);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
constexpr int kBinBlock = 256;
constexpr int kBinItems = 4;                       // rows per thread
constexpr int kBinTile = kBinBlock * kBinItems;    // rows per block (tile)

int64_t bin_tile_rows() { return kBinTile; }

__device__ __forceinline__ int bin_of(long long v, const Ranges &rg) {
    // Algorithm 1: the first bin whose inclusive upper range holds v; a
    // negative range means "no bound".
    for (int j = 0; j < rg.nb; ++j)
        if (rg.r[j] < 0 || v <= rg.r[j]) return j;
    return rg.nb - 1;
}

// Sum of x over the lanes of `same` (a group of __match_any_sync), on its
// first lane. `small`: no value of the warp reaches 2^26, so one 32-bit warp
// reduction holds the sum; otherwise the value's 22-bit parts are summed.
__device__ __forceinline__ unsigned long long group_total(unsigned same, unsigned long long x, bool small) {
    if (small) return __reduce_add_sync(same, static_cast<unsigned>(x));
    const unsigned a = __reduce_add_sync(same, static_cast<unsigned>(x) & 0x3fffffu);
    const unsigned b = __reduce_add_sync(same, static_cast<unsigned>(x >> 22) & 0x3fffffu);
    const unsigned c = __reduce_add_sync(same, static_cast<unsigned>(x >> 44));
    return a + (static_cast<unsigned long long>(b) << 22) + (static_cast<unsigned long long>(c) << 44);
}

// Counts, size sums and A entries per bin: the lanes of a warp that share a
// bin are summed by a warp reduction and their first lane adds the result to
// the warp's own counters in shared memory, without atomics (a warp's groups
// have different bins); one global atomic per non-empty bin and block. Bound
// by the loads of the sizes and row pointers. (Before: two 64-bit shared
// atomics per row, compare-and-swap loops that all rows of a bin contend
// for: 57 us for 4,096 rows, 0.265 ms for 2.1M rows in one bin.)
// REP: with repeating rows (rep.words).
template <bool REP>
__global__ void __launch_bounds__(kBinBlock)
bin_pass1_kernel(const int64_t *sizes, int64_t n, Ranges rg, Operands op, Counters *cnt,
                 long long *tile_sums, RepArgs rep) {
    constexpr int kWarps = kBinBlock / 32;
    __shared__ unsigned s_own[kWarps][kMaxBins];
    __shared__ unsigned s_rep[kRepClasses];
    __shared__ unsigned s_cnt[kWarps][kMaxBins];
    __shared__ unsigned long long s_bsum[kWarps][kMaxBins];
    __shared__ unsigned long long s_bnza[kWarps][kMaxBins];
    __shared__ unsigned long long s_max[kWarps];
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    if (lane < kMaxBins) {
        s_cnt[w][lane] = 0;
        s_own[w][lane] = 0;
        s_bsum[w][lane] = 0;
        s_bnza[w][lane] = 0;
    }
    if (REP) {
        if (threadIdx.x < kRepClasses) s_rep[threadIdx.x] = 0;
        __syncthreads();
    }
    __syncwarp();
    const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * kBinTile;
    unsigned long long v[kBinItems], na[kBinItems];
#pragma unroll
    for (int it = 0; it < kBinItems; ++it) {
        const int64_t i = tile0 + it * kBinBlock + threadIdx.x;
        v[it] = na[it] = 0;
        if (i < n) {
            const int64_t ar = op.row0 + i;
            v[it] = static_cast<unsigned long long>(sizes[i]);
            na[it] = static_cast<unsigned long long>(ld_rpt(op.arpt, op.a64, ar + 1) - ld_rpt(op.arpt, op.a64, ar));
        }
    }
    unsigned out = 0;   // bit it: the row is left out of the bins
    if (REP) {
#pragma unroll
        for (int it = 0; it < kBinItems; ++it) {
            const int64_t i = tile0 + it * kBinBlock + threadIdx.x;
            const RepWord rw = i < n ? rep.words[i >> 5] : RepWord{};
            int c = -1;
            if ((rw.fol >> (i & 31)) & 1u) {
                if (rep.fill) {
                    const long long np = rep.nprod ? rep.nprod[i] : static_cast<long long>(v[it]);
                    v[it] = static_cast<unsigned long long>(sizes[rep_own(rw, i)]);
                    rep.fill[i] = static_cast<int64_t>(v[it]);
                    if (static_cast<long long>(v[it]) <= rep.max_nnz) c = rep_class(np, static_cast<long long>(v[it]));
                }
                if (static_cast<long long>(v[it]) <= rep.max_nnz) out |= 1u << it;
            }
            const unsigned same = __match_any_sync(0xffffffffu, c);
            if (c >= 0 && lane == static_cast<unsigned>(__ffs(same) - 1)) atomicAdd(&s_rep[c], __popc(same));
        }
    }
    unsigned long long my_max = 0;
#pragma unroll
    for (int it = 0; it < kBinItems; ++it) {
        const bool valid = tile0 + it * kBinBlock + threadIdx.x < n;
        const unsigned left = REP ? __ballot_sync(0xffffffffu, (out >> it) & 1u) : 0u;
        my_max = my_max > v[it] ? my_max : v[it];
        const int j = valid ? bin_of(static_cast<long long>(v[it]), rg) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, j);
        const bool small = __all_sync(0xffffffffu, (v[it] | na[it]) < (1ull << 26));
        const unsigned long long sv = group_total(same, v[it], small), sn = group_total(same, na[it], small);
        if (valid && lane == static_cast<unsigned>(__ffs(same) - 1)) {
            s_cnt[w][j] += static_cast<unsigned>(__popc(same));
            s_own[w][j] += static_cast<unsigned>(__popc(same & ~left));
            s_bsum[w][j] += sv;
            s_bnza[w][j] += sn;
        }
        __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long m = __shfl_xor_sync(0xffffffffu, my_max, o);
        if (m > my_max) my_max = m;
    }
    if (lane == 0) s_max[w] = my_max;
    __syncthreads();
    if (w == 0) {
        unsigned c = 0, own = 0;
        unsigned long long bs = 0, bn = 0, mx = 0;
        for (int q = 0; q < kWarps; ++q) {
            if (lane < kMaxBins) {
                c += s_cnt[q][lane];
                own += s_own[q][lane];
                bs += s_bsum[q][lane];
                bn += s_bnza[q][lane];
            }
            mx = mx > s_max[q] ? mx : s_max[q];
        }
        unsigned long long sum = bs;
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (c) {
            atomicAdd(&cnt->bin_cnt[lane], static_cast<unsigned long long>(c));
            atomicAdd(&cnt->bin_sum[lane], bs);
            atomicAdd(&cnt->bin_nnza[lane], bn);
            if (own) atomicAdd(&cnt->bin_own[lane], static_cast<unsigned long long>(own));
        }
        if (REP && lane < kRepClasses && s_rep[lane])
            atomicAdd(&cnt->rep_cnt[lane], static_cast<unsigned long long>(s_rep[lane]));
        if (lane == 0) {
            atomicMax(&cnt->max_size, mx);
            atomicAdd(&cnt->total, sum);
            if (tile_sums) tile_sums[blockIdx.x] = static_cast<long long>(sum);
        }
    }
}

__global__ void __launch_bounds__(kBinBlock)
bin_pass2_kernel(const int64_t *sizes, int64_t n, Ranges rg, Counters *cnt, int32_t *bins,
                 Ranges off, RepArgs rep) {
    __shared__ unsigned s_cnt[kMaxBins];
    __shared__ long long s_base[kMaxBins];
    if (threadIdx.x < kMaxBins) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const unsigned lane = threadIdx.x & 31u;
    const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * kBinTile;
    int jv[kBinItems];
    unsigned pos[kBinItems];
#pragma unroll
    for (int it = 0; it < kBinItems; ++it) {
        const int64_t i = tile0 + it * kBinBlock + threadIdx.x;
        bool valid = i < n;
        const long long v = valid ? sizes[i] : 0;
        if (rep.words && valid) valid = !((rep.words[i >> 5].fol >> (i & 31)) & 1u) || v > rep.max_nnz;
        const int j = valid ? bin_of(v, rg) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, j);
        const int leader = __ffs(same) - 1;
        unsigned wbase = 0;
        if (valid && static_cast<int>(lane) == leader)
            wbase = atomicAdd(&s_cnt[j], static_cast<unsigned>(__popc(same)));
        wbase = __shfl_sync(0xffffffffu, wbase, leader);
        jv[it] = j;
        pos[it] = wbase + __popc(same & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (threadIdx.x < rg.nb) {
        const unsigned c = s_cnt[threadIdx.x];
        s_base[threadIdx.x] = off.r[threadIdx.x] +
            (c ? static_cast<long long>(atomicAdd(&cnt->cursor[threadIdx.x],
                                                  static_cast<unsigned long long>(c)))
               : 0);
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kBinItems; ++it) {
        const int64_t i = tile0 + it * kBinBlock + threadIdx.x;
        if (jv[it] >= 0) bins[s_base[jv[it]] + pos[it]] = static_cast<int32_t>(i);
    }
}

cudaError_t launch_bin_pass1(const int64_t *sizes, int64_t n, const Ranges &rg,
                             const Operands &op, Counters *cnt, long long *tile_sums,
                             cudaStream_t s, const RepArgs &rep) {
    if (n <= 0) return cudaSuccess;
    const int64_t grid = (n + kBinTile - 1) / kBinTile;
    const auto kernel = rep.words ? &bin_pass1_kernel<true> : &bin_pass1_kernel<false>;
    kernel<<<static_cast<unsigned>(grid), kBinBlock, 0, s>>>(sizes, n, rg, op, cnt, tile_sums, rep);
    return cudaGetLastError();
}

cudaError_t launch_bin_pass2(const int64_t *sizes, int64_t n, const Ranges &rg,
                             const long long *offsets, Counters *cnt, int32_t *bins,
                             cudaStream_t s, const RepArgs &rep) {
    if (n <= 0) return cudaSuccess;
    Ranges off{};
    off.nb = rg.nb;
    for (int j = 0; j < rg.nb; ++j) off.r[j] = offsets[j];
    const int64_t grid = (n + kBinTile - 1) / kBinTile;
    bin_pass2_kernel<<<static_cast<unsigned>(grid), kBinBlock, 0, s>>>(sizes, n, rg, cnt, bins,
                                                                       off, rep);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Exclusive scan of the row sizes into C.rpt, in place (Sec. 5.3). Tile t
// covers rows [t*kBinTile, (t+1)*kBinTile), the same tiles whose sums
// bin_pass1_kernel stored.
constexpr int kScanBlock = 1024;

__global__ void __launch_bounds__(kScanBlock)
scan_tiles_kernel(long long *tile_sums, int64_t ntiles) {
    // Exclusive scan of tile_sums[0..ntiles) in place; tile_sums[ntiles] = total.
    __shared__ long long s_warp[32];
    __shared__ long long s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    for (int64_t base = 0; base < ntiles; base += kScanBlock) {
        const int64_t i = base + threadIdx.x;
        const long long x = i < ntiles ? tile_sums[i] : 0;
        long long inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= static_cast<unsigned>(o)) inc += y;
        }
        if (lane == 31) s_warp[w] = inc;
        __syncthreads();
        if (w == 0) {
            long long t = s_warp[lane];
            long long ti = t;
            for (int o = 1; o < 32; o <<= 1) {
                long long y = __shfl_up_sync(0xffffffffu, ti, o);
                if (lane >= static_cast<unsigned>(o)) ti += y;
            }
            s_warp[lane] = ti - t;
        }
        __syncthreads();
        const long long carry = s_carry;
        const long long excl = carry + s_warp[w] + inc - x;
        if (i < ntiles) tile_sums[i] = excl;
        __syncthreads();
        if (threadIdx.x == kScanBlock - 1) s_carry = excl + x;
        __syncthreads();
    }
    if (threadIdx.x == 0) tile_sums[ntiles] = s_carry;
}

__global__ void __launch_bounds__(kBinBlock)
scan_apply_kernel(int64_t *crpt, int64_t n, const long long *tile_prefix, int64_t ntiles) {
    // One block per tile of kBinTile rows; each thread scans kBinItems
    // consecutive rows.
    __shared__ long long s_warp[kBinBlock / 32];
    const int64_t t = blockIdx.x;
    const int64_t r0 = t * kBinTile + static_cast<int64_t>(threadIdx.x) * kBinItems;
    long long v[kBinItems];
    long long local = 0;
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        v[k] = (r0 + k < n) ? crpt[r0 + k] : 0;
        local += v[k];
    }
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    long long inc = local;
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= static_cast<unsigned>(o)) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        long long x = lane < kBinBlock / 32 ? s_warp[lane] : 0;
        long long xi = x;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= static_cast<unsigned>(o)) xi += y;
        }
        if (lane < kBinBlock / 32) s_warp[lane] = xi - x;
    }
    __syncthreads();
    long long run = tile_prefix[t] + s_warp[w] + inc - local;
#pragma unroll
    for (int k = 0; k < kBinItems; ++k) {
        if (r0 + k < n) crpt[r0 + k] = run;
        run += v[k];
    }
    if (t == ntiles - 1 && threadIdx.x == 0) crpt[n] = tile_prefix[ntiles];
}

cudaError_t launch_scan(int64_t *crpt, int64_t n, long long *tile_sums, cudaStream_t s) {
    if (n <= 0) {
        return cudaMemsetAsync(crpt, 0, sizeof(int64_t), s);
    }
    const int64_t ntiles = (n + kBinTile - 1) / kBinTile;
    scan_tiles_kernel<<<1, kScanBlock, 0, s>>>(tile_sums, ntiles);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    scan_apply_kernel<<<static_cast<unsigned>(ntiles), kBinBlock, 0, s>>>(crpt, n, tile_sums, ntiles);
    return cudaGetLastError();
}

__global__ void iota_kernel(int32_t *out, int64_t n) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) out[i] = static_cast<int32_t>(i);
}

cudaError_t launch_iota(int32_t *out, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    iota_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(out, n);
    return cudaGetLastError();
}

}  // namespace ops
