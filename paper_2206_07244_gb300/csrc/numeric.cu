// Numeric phase (Sec. 2.2, Sec. 5.2, Algorithm 5, Sec. 5.6.2): the sorted
// column indices and summed values of each output row, written at the row
// offsets that the scan left in C.rpt.
//
// Bins 0..8: a row group of TPR threads owns a shared-memory table of T
// (int32 key, float64 value) slots, 12 bytes each, keys -1 = empty. Each
// product probes with one atomicCAS; on an empty slot or the same key its
// fused multiply-add is a 64-bit compare-and-swap loop (Algorithm 5), or a
// plain update where a warp or less takes one B row per step and B's rows are
// strictly ascending. Then the three phases of Sec. 5.6.2 follow: condense the
// occupied slots to the front of the table (ballot/popc prefix per chunk of TPR
// slots, in place), sort them by column (in a warp's registers, by a span bitmap,
// or a bitonic network in shared memory) and store them coalesced. The row size
// is known from the symbolic phase and checked. Three kinds of rows go another
// way:
//  - rows of at most 8 products stay in the registers of 8 lanes (tiny_load);
//  - a warp adds a row that spans few columns by column in the table's memory,
//    without probes and sort (span_walk; kSpanShort says when);
//  - the 512- and 1024-slot tables have a warp-per-row form, and num_row_limits
//    decides which rows take it and which the block-per-row form.
// Rows that repeat the pattern of the row before are not in the bins (repeat.cu).
//
// Rows past the largest table go to num_bitmap_kernel (one 1024-thread block
// per row). Pass 1 marks the row's columns in a shared-memory bitmap (set
// with 32-bit atomicOr, read as 64-bit words) and forms per-word prefix counts,
// which give every column its rank in the sorted row: C.col is written straight
// from the bitmap in column order, no sort needed. Pass 2 adds each product into
// C.val[rank] with a float64 atomicAdd in global memory (L2). 227 KB cover 1.2M
// columns per pass; wider matrices take several column windows. This replaces the
// paper's global-memory hash kernel (its kernel 7) and its condense/sort.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "internal.h"

namespace ops {

// Returns false when every slot holds another key (the table is full).
// MULTI: the access pattern the paper measures against (Sec. 6, the hashing
// comparison), a plain read of the slot first and the compare-and-swap only
// on an empty one; otherwise one access per probe (Algorithm 5).
template <int T, bool MULTI = false>
__device__ __forceinline__ bool num_insert(int *tk, double *tv, int key, double a, double b) {
    uint32_t h = hash_slot<T>(key);
    for (int it = 0; it < T; ++it) {
        if (MULTI) {
            const int cur = *static_cast<volatile int *>(tk + h);
            bool hit = cur == key;
            if (!hit && cur == -1) {
                const int old = atomicCAS(tk + h, -1, key);
                hit = old == -1 || old == key;
            }
            if (hit) {
                smem_fma_add(tv + h, a, b);
                return true;
            }
        } else {
            const int old = atomicCAS(tk + h, -1, key);
            if (old == -1 || old == key) {
                smem_fma_add(tv + h, a, b);
                return true;
            }
        }
        h = next_slot<T>(h);
    }
    return false;
}

// The same probe with the value updated by a plain read, fused
// multiply-add and write: for row groups whose steps touch distinct entries
// only (group_row_walk with SYNC), where no other thread can update the
// entry in between. The key still takes a compare-and-swap: distinct keys of
// one step may probe the same slot.
template <int T>
__device__ __forceinline__ bool num_insert_owned(int *tk, double *tv, int key, double a, double b) {
    uint32_t h = hash_slot<T>(key);
    for (int it = 0; it < T; ++it) {
        const int old = atomicCAS(tk + h, -1, key);
        if (old == -1 || old == key) {
            tv[h] = fma(a, b, tv[h]);
            return true;
        }
        h = next_slot<T>(h);
    }
    return false;
}

// Mean referenced B-row length decides how many threads walk one B row; the
// symbolic phase's n_prod is gone by now (C.rpt holds offsets), so the row
// group recomputes it from B.rpt (those lines are needed right after).
template <int TPR>
__device__ __forceinline__ int numeric_lanes(const Operands &op, int fixed, int64_t p0,
                                             int64_t p1, int lg, long long *red, long long &sum) {
    sum = 0;   // products of the row, unless the lanes are fixed
    if (fixed > 0) return pick_lanes_distinct(fixed, 0, 1, TPR);
    for (int64_t p = p0 + lg; p < p1; p += TPR) {
        const int k = __ldg(op.acol + p);
        sum += ld_rpt(op.brpt, op.b64, k + 1) - ld_rpt(op.brpt, op.b64, k);
    }
    sum = group_sum<TPR>(sum, red);
    return pick_lanes_distinct(0, sum, p1 - p0, TPR);
}

// Accumulator of a column that no product has reached: a signalling NaN, which
// no arithmetic result is; the upper half tells it from every other value that
// an accumulator holds.
constexpr long long kNoEntry = 0x7ff0000100000000ll;
__device__ __forceinline__ bool no_entry(double v) { return __double2hiint(v) == static_cast<int>(kNoEntry >> 32); }

// Adds the products of the row [p0, p1) of A to acc[column - col0], by one
// warp. A's entries go through shared memory 32 at a time (ent: their values
// and B rows, len: lengths), and a lane loads its product of kU B rows before
// using any (8 where the tables leave the registers for it); one B row at a time is added (distinct columns: no atomics), in
// the order of A's entries. False when a column lies outside [0, span): B
// changed since its order was checked. Bound by latency: the tables leave 16
// to 40 warps on an SM, each waiting for its own loads and shared-memory
// updates (49% of issue slots, 35% of the float64 pipe). Block-diagonal n =
// 2^20, blocks of 1024 columns: numeric 9.49 ms by the table, 4.39 ms this way.
struct __align__(16) SpanEntry {
    double a;
    long long q;
};
// PRE: q0 / len0 hold the B row of A's entry p0 + lane (from row_span; the
// 256-slot kernel has no registers for them).
template <int kU, bool PRE>
__device__ __forceinline__ bool span_walk(const Operands &op, int64_t p0, int64_t p1, long long q0, int len0, int col0,
                                          int span, double *acc, SpanEntry *ent, int *len) {
    const int lane = threadIdx.x & 31;
    bool inside = true;
    auto add = [&](int c, double a, double b) {
        const unsigned at = static_cast<unsigned>(c) - static_cast<unsigned>(col0);
        if (at < static_cast<unsigned>(span)) {
            const double v = acc[at];
            acc[at] = fma(a, b, no_entry(v) ? 0.0 : v);
        } else {
            inside = false;
        }
    };
    for (int64_t p = p0; p < p1; p += 32) {
        const int cnt = static_cast<int>(p1 - p < 32 ? p1 - p : 32);
        __syncwarp();   // readers of the entries before are done
        int mine = 0;
        if (lane < cnt) {
            long long q = q0;
            mine = len0;
            if (!PRE || p > p0) {
                const int k = __ldg(op.acol + p + lane);
                q = ld_rpt(op.brpt, op.b64, k);
                mine = static_cast<int>(ld_rpt(op.brpt, op.b64, k + 1) - q);
            }
            ent[lane] = SpanEntry{__ldg(op.aval + p + lane), q};
        }
        len[lane] = mine;   // 0 past the entries
        const bool one_piece = __all_sync(0xffffffffu, mine <= 32);
        __syncwarp();
        if (one_piece) {
            for (int e = 0; e < cnt; e += kU) {   // uniform over the warp
                int c[kU];
                double a[kU], b[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    c[u] = -1;
                    a[u] = b[u] = 0.0;
                    if (lane < len[(e + u) & 31] && e + u < cnt) {
                        const SpanEntry x = ent[e + u];
                        a[u] = x.a;
                        c[u] = __ldg(op.bcol + x.q + lane);
                        b[u] = __ldg(op.bval + x.q + lane);
                    }
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (c[u] >= 0) add(c[u], a[u], b[u]);
                    __syncwarp();
                }
            }
        } else {
            for (int e = 0; e < cnt; ++e) {
                const int n = len[e];
                const SpanEntry x = ent[e];
                for (int o = lane; o < n; o += 32 * kU) {
                    int c[kU];
                    double b[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        c[u] = -1;
                        b[u] = 0.0;
                        if (o + 32 * u < n) {
                            c[u] = __ldg(op.bcol + x.q + o + 32 * u);
                            b[u] = __ldg(op.bval + x.q + o + 32 * u);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u)
                        if (c[u] >= 0) add(c[u], x.a, b[u]);
                }
                __syncwarp();
            }
        }
    }
    __syncwarp();
    return inside;
}

// Ascending bitonic sort of the NR * 32 values one warp holds in registers,
// element e = r * 32 + lane in x[r] (striped, so the sorted result stores
// coalesced). Every loop has a compile-time trip count and unrolls fully, so
// register indices are constants: strides below 32 exchange through
// shuffles, larger ones between a lane's own registers.
template <int NR>
__device__ __forceinline__ void warp_bitonic(unsigned (&x)[NR]) {
    constexpr int P = NR * 32;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= P; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const int r2 = r ^ (j >> 5);
                    if (r2 > r) {
                        const bool up = ((r * 32 + lane) & k) == 0;
                        const unsigned a = x[r], b = x[r2];
                        const unsigned mn = a < b ? a : b, mx = a < b ? b : a;
                        x[r] = up ? mn : mx;
                        x[r2] = up ? mx : mn;
                    }
                }
            } else {
                const bool lower = (lane & j) == 0;
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const unsigned o = __shfl_xor_sync(0xffffffffu, x[r], j);
                    const bool up = ((r * 32 + lane) & k) == 0;
                    const unsigned mn = x[r] < o ? x[r] : o, mx = x[r] < o ? o : x[r];
                    x[r] = lower == up ? mn : mx;
                }
            }
        }
    }
}

// One warp: sort the n condensed entries (tk[e], tv[e]), e < n <= NR * 32,
// by column and store the first m to ocol/oval. Keys are (column << BITS | e):
// columns below 2^(32 - BITS), n <= 2^BITS.
template <int NR, int BITS>
__device__ __forceinline__ void warp_sort_store(const int *tk, const double *tv, int n, int64_t m,
                                                int32_t *ocol, double *oval, bool store) {
    const int lane = threadIdx.x & 31;
    unsigned x[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        const int e = q * 32 + lane;
        x[q] = e < n ? (static_cast<unsigned>(tk[e]) << BITS) | static_cast<unsigned>(e) : 0xffffffffu;
    }
    warp_bitonic<NR>(x);
    if (!store) return;
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        const int e = q * 32 + lane;
        if (e < m) {
            ocol[e] = static_cast<int32_t>(x[q] >> BITS);
            oval[e] = tv[x[q] & ((1u << BITS) - 1u)];
        }
    }
}

// Minimum resident blocks: enough for 2048 threads per SM (<= 32 registers
// per thread, Sec. 5.6) for sub-warp row groups, unless the table is so
// large that one block fills the SM's shared memory anyway. Kernels whose
// walks and sorts spill at 32 registers get fewer threads and more
// registers: warp-per-row kernels that sort in registers 1280 threads (48
// registers; 27-point stencil 128^3: 10.64 -> 9.72 ms against 1536 threads),
// block-per-row kernels 1536 (40 registers; block-diagonal n = 2^20:
// 12.43 -> 10.44 ms against 2048). The warp-per-row forms of the 512- and
// 1024-slot tables get the threads that their shared memory allows.
// ONE_PHASE (learned sizing): the row's size is not known; the table was
// chosen from a prediction. A probe that finds no free slot, or more keys
// than the table can sort in place, marks the row as mispredicted: it is
// queued for the exact path and nothing is written. Otherwise the row's
// size goes to C.rpt and its sorted entries to its temporary slot.
// QUEUE: warp-per-row kernels leave rows past their limit in the queue, block-per-
// row kernels take theirs from it, a block one row after the other.
template <int TPR, int BLOCK, int T, bool ONE_PHASE = false, bool MULTI = false, bool QUEUE = false>
__global__ void __launch_bounds__(BLOCK, (T * 12 * (BLOCK / TPR) > 110 * 1024) ? 1
                                         : (TPR == 32 ? (T <= 256 ? 1280 : T <= 512 ? 896 : 576) : (TPR > 32 ? 1536 : 2048)) / BLOCK)
num_hash_kernel(Operands op, BinWork w) {
    constexpr int RPB = BLOCK / TPR;
    constexpr bool kTake = QUEUE && TPR > 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long red64[32];
    __shared__ int red32[33];
    __shared__ int full[RPB];   // one-phase: a probe found no free slot in this row's table
    const int g = threadIdx.x / TPR, lg = threadIdx.x % TPR;
    double *tv = reinterpret_cast<double *>(smem_raw + static_cast<size_t>(g) * (T * 12));   // the row's table
    int *tk = reinterpret_cast<int *>(tv + T);
    unsigned turn = blockIdx.x;
[[maybe_unused]] next_row:
    if constexpr (kTake) {
        if (turn >= __ldcg(w.queued)) return;   // uniform over the block
        __syncthreads();   // readers of the row before are done
    }
    bool failed = false;
    if (lg == 0) full[g] = 0;
    const int64_t r = kTake ? w.queue[turn] : static_cast<int64_t>(blockIdx.x) * RPB + g;   // the row's place in the bin
    turn += gridDim.x;
    const bool valid = r < w.cnt;
    const int64_t row = valid ? (w.bins ? static_cast<int64_t>(w.bins[w.off + r]) : w.off + r) : 0;
    int64_t cbase = 0, n_expect = 0, p0 = 0, p1 = 0;
    if (valid) {
        if (!ONE_PHASE) {
            cbase = w.crpt[row];
            n_expect = w.crpt[row + 1] - cbase;
        }
        const int64_t ar = op.row0 + row;
        p0 = ld_rpt(op.arpt, op.a64, ar);
        p1 = ld_rpt(op.arpt, op.a64, ar + 1);
    }
    if constexpr (TPR == 8 && !ONE_PHASE && !MULTI) {
        // all four rows of the warp have at most 8 products (2.1M rows of 7:
        // 862 -> 277 us)
        TinyRow t;
        if (tiny_load<true>(op, p0, p1, t)) {
            double sum = 0.0;
            unsigned m = t.first ? t.eq : 0u;
            while (__any_sync(0xffffffffu, m)) {   // in the order of A's entries
                const int j = m ? __ffs(m) - 1 : 0;
                const double a = __shfl_sync(0xffffffffu, t.a, j, 8), b = __shfl_sync(0xffffffffu, t.b, j, 8);
                if (m) sum = fma(a, b, sum);
                m &= m - 1;
            }
            const int rank = __popc(t.lt & t.heads);
            if (t.first && rank < n_expect) {
                w.ccol[cbase + rank] = t.col;
                w.cval[cbase + rank] = sum;
            }
            if (valid && lg == 0 && __popc(t.heads) != n_expect) set_error(w.err, DERR_COUNT_MISMATCH);
            return;   // uniform over the warp; no block barrier follows
        }
    }
    // A warp's row whose columns span at most kSpan columns is accumulated by
    // column in the table's memory (B's rows strictly ascending and not too short,
    // kSpanShort): no probes, no condense and no sort.
    constexpr bool kMaySpan = TPR == 32 && !MULTI;
    constexpr int kSpan = (T * 12 / 8) / 32 * 32;
    int S = TPR, col0 = 0, span = 0, len0 = 0;
    long long q0 = 0, sum = 0;
    bool far = false;   // QUEUE: a block would sort the row's entries, not place them by its span bitmap
    if (kMaySpan && w.by_column && w.lanes == 0) {
        row_span(op, p0, p1, sum, col0, span, q0, len0);
        S = pick_lanes_distinct(0, sum, p1 - p0, TPR);
        far = QUEUE && (ONE_PHASE ? T / 2 : n_expect) + 2 * ((static_cast<int64_t>(span) + 31) >> 5) > T;
        if (span > kSpan || S < 8 || (S == 8 && p1 - p0 > kSpanShort)) span = 0;
    } else {
        S = numeric_lanes<TPR>(op, w.lanes, p0, p1, lg, red64, sum);
    }
    if constexpr (QUEUE && TPR == 32) {
        if (sum > (span > 0 && S >= 16 ? w.long_col : far ? w.long_far : w.long_near)) {
            if (lg == 0) w.queue[atomicAdd(w.queued, 1u)] = static_cast<int32_t>(r);   // r < cnt: sum > 0
            return;   // uniform over the warp; no block barrier follows
        }
    }
    const bool dense = kMaySpan && span > 0;   // uniform over the warp, and over the row group
    if (dense) {
        long long *acc = reinterpret_cast<long long *>(tv);
#pragma unroll 4
        for (int s = lg; s < span; s += TPR) acc[s] = kNoEntry;
    } else {
        for (int s = lg; s < T; s += TPR) {
            tk[s] = -1;
            tv[s] = 0.0;
        }
    }
    group_sync<TPR>();
    if constexpr (TPR > 32) {
        // one row per block: flattened walk over B-row pieces
        WalkScratch *sc = reinterpret_cast<WalkScratch *>(
            smem_raw + (sizeof(int) + sizeof(double)) * (size_t)RPB * T);
        block_row_walk<BLOCK, true>(op, p0, p1, S, sc, [&](int key, double a, double b) {
            if (!num_insert<T, MULTI>(tk, tv, key, a, b)) failed = true;
        });
    } else if (!MULTI && w.distinct && (S == TPR || dense)) {
        // one B row per step, its columns distinct: values without atomics,
        // B's entries staged in shared memory by cp.async (after the tables:
        // kStage * TPR values, then as many columns, per row group)
        double *sv = reinterpret_cast<double *>(smem_raw + (sizeof(int) + sizeof(double)) * (size_t)RPB * T) +
                     static_cast<size_t>(g) * kStage * TPR;
        int *sc = reinterpret_cast<int *>(reinterpret_cast<double *>(smem_raw +
                                                                      (sizeof(int) + sizeof(double)) * (size_t)RPB * T) +
                                          static_cast<size_t>(RPB) * kStage * TPR) +
                  static_cast<size_t>(g) * kStage * TPR;
        if (dense)
            failed = !span_walk<(T >= 1024 ? 8 : 4), (T >= 512)>(op, p0, p1, q0, len0, col0, span, tv,
                                                   reinterpret_cast<SpanEntry *>(sv), sc);
        else
            group_row_walk_staged<TPR>(op, p0, p1, sc, sv, [&](int key, double a, double b) {
                if (!num_insert_owned<T>(tk, tv, key, a, b)) failed = true;
            });
    } else {
        group_row_walk<TPR, true>(op, p0, p1, S, [&](int key, double a, double b) {
            if (!num_insert<T, MULTI>(tk, tv, key, a, b)) failed = true;
        });
    }
    if (failed) {
        if (ONE_PHASE) full[g] = 1;
        else set_error(w.err, DERR_TABLE_FULL);
    }
    group_sync<TPR>();
    // condense: occupied slots move to the front, chunk by chunk; a write
    // never lands past the chunk that was just read.
    int n = 0;
    int kmin = INT_MAX, kmax = -1;   // this thread's smallest and largest key
    if (dense) {
        if (ONE_PHASE) {
            for (int s = lg; s < span; s += TPR) n += !no_entry(tv[s]);
            if constexpr (TPR <= 32) n = warp_sum_xor(n, TPR);
        } else {
            n = static_cast<int>(n_expect < span ? n_expect : span);   // counted as it is stored
        }
    }
    for (int c = 0; c < T && !dense; c += TPR) {
        const int s = c + lg;
        int k = -1;
        double v = 0.0;
        if (s < T) {
            k = tk[s];
            v = tv[s];
        }
        if (k >= 0) {
            kmin = min(kmin, k);
            kmax = max(kmax, k);
        }
        int pre, tot;
        group_excl_count<TPR>(k >= 0, pre, tot, red32);
        group_sync<TPR>();
        if (k >= 0) {
            tk[n + pre] = k;
            tv[n + pre] = v;
        }
        n += tot;
        group_sync<TPR>();
    }
    int P = 1;
    while (P < n) P <<= 1;
    if constexpr (ONE_PHASE) {
        // mispredicted: queue the row for the exact path, write nothing else
        if (full[g] || P > T) {
            if (valid && lg == 0) {   // C.rpt keeps n_prod for the exact symbolic kernel
                w.pred[row] = -1;
                if (w.fb)
                    atomicAdd(w.fb + (3 * kMaxBins + w.lcls[row]) * kLoadSlots + blockIdx.x % kLoadSlots, 1ull);
                const unsigned long long at = atomicAdd(w.xcount, 1ull);
                if (at < static_cast<unsigned long long>(w.xlimit)) w.xlist[at] = static_cast<int32_t>(row);
                else set_error(w.err, DERR_BOUNDS);
            }
            if constexpr (kTake) goto next_row;
            else return;   // uniform over the row group
        }
        n_expect = n;
        if (valid && lg == 0) {
            w.crpt[row] = n;
            // load feedback: more than 3/4 full, or at most 3/4 of the next smaller table
            const int grp = 4 * n > 3 * T ? 1 : (w.tprev > 0 && 4ll * n <= 3 * w.tprev ? 2 : 0);
            if (w.fb && grp)
                atomicAdd(w.fb + (grp * kMaxBins + w.lcls[row]) * kLoadSlots + blockIdx.x % kLoadSlots, 1ull);
        }
    } else {
        if (valid && n != n_expect) set_error(w.err, DERR_COUNT_MISMATCH);
        if (P > T) {  // cannot happen within the kernel's capacity; never index past the table
            set_error(w.err, DERR_TABLE_FULL);
            P = 1;
        }
    }
    if constexpr (kMaySpan) {
        if (dense) {
            // entries in column order: the ones before in their 32 columns by
            // ballot, the ones before those by a running count
            int32_t *ocol = w.ccol + cbase;
            double *oval = w.cval + cbase;
            int m = valid ? n : 0;   // entries to store
            if (ONE_PHASE) {
                ocol = w.tcol + w.tbase + r * w.tcap;
                oval = w.tval + w.tbase + r * w.tcap;
                if (m > w.tcap || w.tbase + r * w.tcap + m > w.tlimit) {
                    if (lg == 0) set_error(w.err, DERR_BOUNDS);
                    m = 0;
                }
            }
            int at = 0;
#pragma unroll 4
            for (int s = lg; s < span + lg; s += 32) {   // uniform over the warp
                const double v = s < span ? tv[s] : __longlong_as_double(kNoEntry);
                const bool here = !no_entry(v);
                const unsigned bal = __ballot_sync(0xffffffffu, here);
                const int o = at + __popc(bal & ((1u << lg) - 1u));
                if (here && o < m) {
                    ocol[o] = col0 + s;
                    oval[o] = v;
                }
                at += __popc(bal);
            }
            if (!ONE_PHASE && valid && lg == 0 && at != n_expect) set_error(w.err, DERR_COUNT_MISMATCH);
            return;   // uniform over the warp; no block barrier follows
        }
    }
    if constexpr (TPR == 32 && T <= 1024) {
        constexpr int kBits = T <= 256 ? 8 : 9;
        if (op.ncols <= (int64_t{1} << (32 - kBits)) && n <= (1 << kBits)) {   // uniform over the warp
            // one warp per row: sort (column << 8 | slot) in registers, then
            // store columns and the values of their slots in order
            const int64_t m = n < n_expect ? n : n_expect;
            int32_t *ocol = w.ccol + cbase;
            double *oval = w.cval + cbase;
            bool in_bounds = true;
            if (ONE_PHASE) {
                ocol = w.tcol + w.tbase + r * w.tcap;
                oval = w.tval + w.tbase + r * w.tcap;
                in_bounds = m <= w.tcap && w.tbase + r * w.tcap + m <= w.tlimit;
                if (valid && !in_bounds && lg == 0) set_error(w.err, DERR_BOUNDS);
            }
            const bool store = valid && in_bounds;
            if (n <= 32) warp_sort_store<1, kBits>(tk, tv, n, m, ocol, oval, store);
            else if (n <= 64) warp_sort_store<2, kBits>(tk, tv, n, m, ocol, oval, store);
            else if (n <= 128) warp_sort_store<4, kBits>(tk, tv, n, m, ocol, oval, store);
            else if (n <= 256) warp_sort_store<8, kBits>(tk, tv, n, m, ocol, oval, store);
            else if constexpr (kBits > 8) warp_sort_store<16, kBits>(tk, tv, n, m, ocol, oval, store);
            return;   // uniform over the warp; no block barrier follows
        }
    }
    if constexpr (TPR > 32) {
        // One row per block. When the row's columns span few enough words,
        // each entry goes straight to its place in the sorted row: bit
        // (column - min) of a span bitmap is set for every entry, and the
        // set bits below it give its rank. The bitmap (nw words) and its
        // per-word prefix counts (nw words) take the top 2 nw words of the
        // key table, above the n condensed keys.
        if (n > 0) {   // uniform: n is the block's count
            kmin = block_min<TPR>(kmin, red32);
            kmax = -block_min<TPR>(-kmax, red32);
            const long long span = static_cast<long long>(kmax) - kmin + 1;
            const long long nwl = (span + 31) >> 5;
            if (n + 2 * nwl <= T) {   // uniform
                const int nw = static_cast<int>(nwl);
                unsigned *bits = reinterpret_cast<unsigned *>(tk + T - 2 * nw);
                unsigned *pre = bits + nw;
                for (int i = lg; i < nw; i += TPR) bits[i] = 0u;
                __syncthreads();
                for (int s = lg; s < n; s += TPR) {
                    const unsigned rel = static_cast<unsigned>(tk[s] - kmin);
                    atomicOr(bits + (rel >> 5), 1u << (rel & 31));
                }
                __syncthreads();
                // rank of each word's first column: thread lg owns words
                // [lg * per, (lg + 1) * per)
                const int per = (nw + TPR - 1) / TPR;
                const int w0 = lg * per, w1 = min(w0 + per, nw);
                unsigned mine = 0;
                for (int i = w0; i < w1; ++i) mine += __popc(bits[i]);
                unsigned total;
                unsigned run = block_excl_scan<TPR>(mine, total, reinterpret_cast<unsigned *>(red32));
                for (int i = w0; i < w1; ++i) {
                    pre[i] = run;
                    run += __popc(bits[i]);
                }
                __syncthreads();
                if (valid) {
                    const int64_t m = n < n_expect ? n : n_expect;
                    int32_t *ocol = w.ccol + cbase;
                    double *oval = w.cval + cbase;
                    bool in_bounds = true;
                    if (ONE_PHASE) {
                        ocol = w.tcol + w.tbase + r * w.tcap;
                        oval = w.tval + w.tbase + r * w.tcap;
                        in_bounds = m <= w.tcap && w.tbase + r * w.tcap + m <= w.tlimit;
                        if (!in_bounds && lg == 0) set_error(w.err, DERR_BOUNDS);
                    }
                    for (int s = lg; in_bounds && s < n; s += TPR) {
                        const int key = tk[s];
                        const unsigned rel = static_cast<unsigned>(key - kmin);
                        const unsigned wd = rel >> 5;
                        const int64_t rank = pre[wd] + __popc(bits[wd] & ((1u << (rel & 31)) - 1u));
                        if (rank < m) {
                            ocol[rank] = key;
                            oval[rank] = tv[s];
                        }
                    }
                }
                if constexpr (kTake) goto next_row;
                else return;   // uniform over the block
            }
        }
    }
    for (int s = n + lg; s < P; s += TPR) tk[s] = INT_MAX;
    group_sync<TPR>();
    // bitonic sort of (key, value) pairs over P entries, ascending
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lg; i < P; i += TPR) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const int ka = tk[i], kb = tk[ixj];
                    const bool up = (i & k) == 0;
                    if ((ka > kb) == up) {
                        tk[i] = kb;
                        tk[ixj] = ka;
                        const double va = tv[i];
                        tv[i] = tv[ixj];
                        tv[ixj] = va;
                    }
                }
            }
            group_sync<TPR>();
        }
    }
    if (valid) {
        const int64_t m = n < n_expect ? n : n_expect;
        int32_t *ocol = w.ccol + cbase;
        double *oval = w.cval + cbase;
        bool in_bounds = true;
        if (ONE_PHASE) {
            ocol = w.tcol + w.tbase + r * w.tcap;
            oval = w.tval + w.tbase + r * w.tcap;
            in_bounds = m <= w.tcap && w.tbase + r * w.tcap + m <= w.tlimit;
            if (!in_bounds && lg == 0) set_error(w.err, DERR_BOUNDS);
        }
        for (int64_t t = lg; in_bounds && t < m; t += TPR) {
            ocol[t] = tk[t];
            oval[t] = tv[t];
        }
    }
    if constexpr (kTake) goto next_row;
}

// Rank of every bitmap word's first column: pre[i] = set bits in words
// [0, i). Warp w owns words [w * per, (w + 1) * per) (per a multiple of 32)
// and its lanes read consecutive words, so no two lanes of a warp hit one
// bank. Returns the total. Synchronises the block; pre is complete on return.
template <int BLOCK>
__device__ __forceinline__ unsigned bitmap_ranks(const unsigned long long *bm, unsigned *pre, int nw,
                                                 unsigned *sw) {
    constexpr int kWarps = BLOCK / 32;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int per = (((nw + kWarps - 1) / kWarps) + 31) & ~31;
    const int w0 = wp * per;
    const int w1 = w0 + per < nw ? w0 + per : nw;
    unsigned cnt = 0;
    for (int i = w0 + lane; i < w1; i += 32) cnt += static_cast<unsigned>(__popcll(bm[i]));
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    __syncthreads();   // earlier readers of sw are done
    if (lane == 0) sw[wp] = cnt;
    __syncthreads();
    if (wp == 0) {
        const unsigned t = lane < kWarps ? sw[lane] : 0u;
        unsigned inc = t;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane < kWarps) sw[lane] = inc - t;
        if (lane == 31) sw[32] = inc;
    }
    __syncthreads();
    unsigned base = sw[wp];
    const unsigned total = sw[32];
    for (int i0 = w0; i0 < w1; i0 += 32) {
        const int i = i0 + lane;
        const unsigned c = i < w1 ? static_cast<unsigned>(__popcll(bm[i])) : 0u;
        unsigned inc = c;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (i < w1) pre[i] = base + inc - c;
        base += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncthreads();
    return total;
}

// Pass 2 by column windows (B rows sorted, run boundaries from bsplit): the
// row's products whose columns fall in sub-ranges [g, g2) of the column
// space are, per A entry, one run of its B row; the runs of a window are
// concatenated into one flat index space that the block's warps split into
// equal contiguous ranges. Windows hold about w.wentries entries of C, so
// the C.val lines that the float64 reductions of a window hit stay in L2.
struct RunMeta {
    long long q0[kWinMaxLists];      // first B entry of each A entry's B row
    double aval[kWinMaxLists];       // A values of the row
    int32_t ks[kWinMaxLists];        // B row of each A entry
    int32_t rs[kWinMaxLists];        // run start (offset in the B row) of the current window
    long long lp[kWinMaxLists + 1];  // exclusive prefix of the run lengths
    long long red[33];               // block scan scratch
    int g2;                          // end sub-range of the current window
};


size_t num_bitmap_head_bytes(bool runs) {
    const size_t a = sizeof(WalkScratch), b = sizeof(RunMeta);
    const size_t h = runs && b > a ? b : a;
    return (h + 15) & ~static_cast<size_t>(15);
}

// Calls f(col, a_value, b_value) for every product of the current window's
// runs (rm->lp holds their exclusive prefix, `total` the sum). A lane loads
// UNROLL products before using any.
template <int BLOCK, int UNROLL, typename F>
__device__ __forceinline__ void run_walk(const Operands &op, const RunMeta *rm, int nl, long long total,
                                         F &&f) {
    constexpr int kWarps = BLOCK / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long per = (total + kWarps - 1) / kWarps;
    const long long f0 = per * warp;
    const long long f1 = f0 + per < total ? f0 + per : total;
    if (f0 >= f1) return;
    int t = 0;
    {   // run of the lane's first index: last t with lp[t] <= f0 + lane
        const long long first = f0 + lane;
        int lo = 0, hi = nl;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (rm->lp[mid] <= first) lo = mid; else hi = mid;
        }
        t = lo;
    }
    for (long long base = f0; base < f1; base += 32 * UNROLL) {
        int c[UNROLL], tt[UNROLL];
        double b[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const long long idx = base + u * 32 + lane;
            c[u] = -1;
            tt[u] = t;
            b[u] = 0.0;
            if (idx < f1) {
                while (rm->lp[t + 1] <= idx) ++t;   // runs are visited in order
                tt[u] = t;
                const long long q = rm->q0[t] + rm->rs[t] + (idx - rm->lp[t]);
                c[u] = __ldg(op.bcol + q);
                b[u] = __ldg(op.bval + q);
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (c[u] >= 0) f(c[u], rm->aval[tt[u]], b[u]);
    }
}

// RUNS: the row is covered in several column windows and B's rows are
// sorted; each window's passes walk only the runs of B rows inside it
// (w.bslot / w.bidx), so a window costs its own products, not the row's.
template <int BLOCK, int ITERS, bool RUNS = false>
__global__ void __launch_bounds__(BLOCK, BLOCK == 1024 ? 1 : (RUNS ? 1024 : 1536) / BLOCK)
num_bitmap_kernel(Operands op, BinWork w, int words) {
    constexpr int kBmBlock = BLOCK;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the head holds the walk scratch of pass 1, then the run metadata of a
    // windowed pass 2
    WalkScratch *sc = reinterpret_cast<WalkScratch *>(smem_raw);
    RunMeta *rm = reinterpret_cast<RunMeta *>(smem_raw);
    unsigned long long *bm = reinterpret_cast<unsigned long long *>(smem_raw + w.head);
    unsigned *bm32 = reinterpret_cast<unsigned *>(bm);   // same words, 32-bit halves
    unsigned *pre = reinterpret_cast<unsigned *>(bm + words);
    __shared__ unsigned sw[33];
    // phase clocks (profiling, w.clk set; 1024-thread blocks, whose
    // registers have room): a block barrier ends each phase, then thread 0
    // adds the SM clock cycles since the previous mark
    constexpr bool kClk = BLOCK == 1024;
    long long tmark = 0;
    if (kClk && w.clk && threadIdx.x == 0) tmark = clock64();
    auto phase_end = [&](int k) {
        if (!kClk || !w.clk) return;   // uniform: a kernel argument
        __syncthreads();
        if (threadIdx.x == 0) {
            const long long t = clock64();
            atomicAdd(w.clk + k, static_cast<unsigned long long>(t - tmark));
            tmark = t;
        }
    };
    // Block b takes the bin's row (b * P) mod cnt, P a prime that does not
    // divide cnt (a permutation): the binning leaves the bin's rows in row
    // order, and on power-law inputs the heaviest rows come first, so blocks
    // in launch order would sum dozens of multi-MB C.val segments at once and
    // push them out of L2 before their rows are done. Spread over the launch,
    // the rows summed together are a sample of the whole bin (R-MAT n = 2^20:
    // 192 -> 178 ms; groups of 256 consecutive rows spread the same way:
    // 183 ms).
    const long long kSpread = (w.cnt % 1000003ll == 0) ? 999983ll : 1000003ll;
    const int64_t pos = static_cast<int64_t>((static_cast<long long>(blockIdx.x) * kSpread) % w.cnt);
    const int64_t row = w.bins ? static_cast<int64_t>(w.bins[w.off + pos]) : w.off + pos;
    const int64_t cbase = w.crpt[row];
    const int64_t n_expect = w.crpt[row + 1] - cbase;
    const int64_t ar = op.row0 + row;
    const int64_t p0 = ld_rpt(op.arpt, op.a64, ar);
    const int64_t p1 = ld_rpt(op.arpt, op.a64, ar + 1);
    // threads per B row from the row's size instead of its n_prod (C.rpt
    // holds offsets by now): n_nz <= n_prod, so the choice is at most one
    // step narrower, and the A row is first read by pass 1 itself
    const int S = pick_lanes_distinct(w.lanes, n_expect, p1 - p0, 32);
    const int64_t span = static_cast<int64_t>(words) * 64;
    int64_t done = 0;
    bool ok = true;
    for (int64_t c0 = 0; c0 < op.ncols; c0 += span) {
        const int nw = static_cast<int>(((op.ncols - c0 < span ? op.ncols - c0 : span) + 63) / 64);
        for (int i = threadIdx.x; i < nw; i += kBmBlock) bm[i] = 0ull;
        __syncthreads();
        phase_end(0);
        // pass 1: the row's columns inside this window. 32-bit atomics on the
        // two halves of a 64-bit word: shared 64-bit atomics run several
        // times slower on this GPU
        const int c0i = static_cast<int>(c0);
        const unsigned span32 = static_cast<unsigned>(span);
        RunSel rsel{w.bslot, w.bidx, w.cs, w.ncells, c0i,
                    static_cast<int>(c0 + span < op.ncols ? c0 + span : op.ncols)};
        block_row_walk<kBmBlock, false, ITERS, 1, RUNS>(op, p0, p1, S, sc, [&](int key, double, double) {
            const unsigned rel = static_cast<unsigned>(key - c0i);   // one compare covers both ends
            if (rel < span32) atomicOr(bm32 + (rel >> 5), 1u << (rel & 31));
        }, &rsel);
        phase_end(1);
        // per-word prefix counts = rank of a word's first column in the
        // window. Warps own contiguous ranges of words and their lanes read
        // consecutive words (no bank conflicts): a warp scan per 32 words,
        // one block scan of the warp totals.
        const unsigned run = bitmap_ranks<kBmBlock>(bm, pre, nw, sw);
        phase_end(2);
        const int64_t cnt = run;
        if (done + cnt > n_expect) ok = false;   // uniform: cnt and done are block-wide
        if (ok) {
            int32_t *ccol = w.ccol + cbase + done;
            double *cval = w.cval + cbase + done;
            // Each warp takes a contiguous range of words of about equal
            // cost, a word costing its column count plus kWordCost for its
            // scan: the cost of the words before word i is pre[i] +
            // kWordCost * i, increasing in i, so a binary search over pre
            // finds a warp's range. (Equal word counts per warp put most
            // columns of a skewed row on a few warps: on R-MAT rows, whose
            // low columns are dense, one warp of 32 held about a quarter of
            // the row; cost ranges: 204 -> 194 ms on R-MAT n = 2^20.)
            // Lanes take consecutive words. A lane writes its own word's
            // columns (32-bit halves in turn: 32-bit bit scans are cheaper
            // than 64-bit ones) when the word holds fewer than kDenseWord of
            // them; denser words are written by the whole warp, one word at a
            // time with one lane per bit, so that each store covers one run
            // of consecutive entries of C.col (measured: 1.5% faster than
            // every lane writing its own word, on R-MAT n = 2^20). The
            // write is bound by instruction issue: a lane loop runs as often
            // as the fullest word of the 32 asks, so words of 12 columns or
            // more go to the whole warp (R-MAT n = 2^20 rows: 8.0 instead of
            // 9.2 loop trips per 32 words; this phase 3.6% faster than with
            // 24). Entry-parallel rounds (lane e finds the word of entry e by
            // a shuffle search) store fully coalesced but issue more: 27%
            // slower.
            constexpr int kDenseWord = 12;
            constexpr unsigned long long kWordCost = 2;
            const int lane = threadIdx.x & 31;
            const unsigned lt = (1u << lane) - 1u;
            const unsigned long long vtot =
                static_cast<unsigned long long>(cnt) + kWordCost * static_cast<unsigned long long>(nw);
            auto first_word = [&](unsigned long long cost) {   // first i in [0, nw] whose prefix cost >= cost
                int lo = 0, hi = nw;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (pre[mid] + kWordCost * static_cast<unsigned long long>(mid) >= cost) hi = mid;
                    else lo = mid + 1;
                }
                return lo;
            };
            const unsigned long long wq = static_cast<unsigned long long>(threadIdx.x >> 5);
            const int i_beg = first_word(vtot * wq / (kBmBlock / 32));
            const int i_end = first_word(vtot * (wq + 1) / (kBmBlock / 32));
            for (int ib = i_beg; ib < i_end; ib += 32) {   // uniform over the warp
                const int i = ib + lane;
                const unsigned long long x = i < i_end ? bm[i] : 0ull;
                const unsigned pos0 = i < i_end ? pre[i] : 0u;
                const bool dense = __popcll(x) >= kDenseWord;
                unsigned dm = __ballot_sync(0xffffffffu, dense);
                if (!dense) {
                    unsigned pos = pos0;
                    const int colbase = c0i + i * 64;
                    unsigned lo = static_cast<unsigned>(x), hi = static_cast<unsigned>(x >> 32);
                    while (lo) {
                        const int b = __ffs(lo) - 1;
                        lo &= lo - 1;
                        ccol[pos++] = colbase + b;
                    }
                    while (hi) {
                        const int b = __ffs(hi) - 1;
                        hi &= hi - 1;
                        ccol[pos++] = colbase + 32 + b;
                    }
                }
                while (dm) {
                    const int src = __ffs(dm) - 1;
                    dm &= dm - 1;
                    const unsigned long long xw = __shfl_sync(0xffffffffu, x, src);
                    const unsigned pw = __shfl_sync(0xffffffffu, pos0, src);
                    const int cb = c0i + (ib + src) * 64;
                    const unsigned lo = static_cast<unsigned>(xw), hi = static_cast<unsigned>(xw >> 32);
                    if ((lo >> lane) & 1u) ccol[pw + __popc(lo & lt)] = cb + lane;
                    if ((hi >> lane) & 1u) ccol[pw + __popc(lo) + __popc(hi & lt)] = cb + 32 + lane;
                }
            }
            phase_end(3);
            const unsigned long long pol = l2_evict_last_policy();
            const int nl = static_cast<int>(p1 - p0 < INT32_MAX ? p1 - p0 : INT32_MAX);
            // one thread per A entry: the row's A entries must fit the block
            if (w.bs && c0 == 0 && span >= op.ncols && nl <= w.wlists && nl <= kBmBlock) {
                // pass 2 by column windows of about w.wentries entries
                bool bad = false;
                if (threadIdx.x < nl) {
                    const int k = __ldg(op.acol + p0 + threadIdx.x);
                    rm->ks[threadIdx.x] = k;
                    rm->q0[threadIdx.x] = ld_rpt(op.brpt, op.b64, k);
                    rm->aval[threadIdx.x] = __ldg(op.aval + p0 + threadIdx.x);
                    rm->rs[threadIdx.x] = 0;
                }
                // rank of the first column of sub-range g (sub-ranges start on word boundaries)
                auto bnd_rank = [&](int g) -> unsigned {
                    const int64_t cb = static_cast<int64_t>(g) << w.gshift;
                    return cb >= op.ncols ? static_cast<unsigned>(cnt) : pre[cb >> 6];
                };
                for (int g = 0; g < w.G;) {
                    if (threadIdx.x == 0) {
                        const unsigned r0 = bnd_rank(g);
                        int g2 = g + 1;
                        while (g2 < w.G && bnd_rank(g2 + 1) - r0 <= static_cast<unsigned>(w.wentries)) ++g2;
                        rm->g2 = g2;
                    }
                    __syncthreads();
                    const int g2 = rm->g2;
                    const unsigned r_lo = bnd_rank(g), r_hi = bnd_rank(g2);
                    long long len = 0;
                    int re = 0;
                    if (threadIdx.x < nl) {
                        re = __ldg(w.bs + static_cast<int64_t>(rm->ks[threadIdx.x]) * (w.G + 1) + g2);
                        len = re - rm->rs[threadIdx.x];
                    }
                    for (unsigned t = r_lo + threadIdx.x; t < r_hi; t += kBmBlock) st_keep(cval + t, 0.0, pol);
                    long long total;
                    const long long ex = block_excl_scan_ll<kBmBlock>(len, total, rm->red);
                    if (threadIdx.x < nl) rm->lp[threadIdx.x] = ex;
                    if (threadIdx.x == 0) rm->lp[nl] = total;
                    __syncthreads();
                    if (total > 0)
                        run_walk<kBmBlock, kBmBlock == 1024 ? 8 : 4>(op, rm, nl, total,
                                                                      [&](int key, double a, double b) {
                            const unsigned rel = static_cast<unsigned>(key - c0i);
                            const unsigned wi = rel >> 6, bi = rel & 63u;
                            const unsigned rank = rel < span32 ? pre[wi] +
                                static_cast<unsigned>(__popcll(bm[wi] << (63u - bi))) - 1u : 0u;
                            if (rel < span32 && rank >= r_lo && rank < r_hi) red_add_keep(cval + rank, a * b, pol);
                            else bad = true;
                        });
                    __syncthreads();
                    const uintptr_t l0 = reinterpret_cast<uintptr_t>(cval + r_lo) & ~static_cast<uintptr_t>(127);
                    const uintptr_t l1 = reinterpret_cast<uintptr_t>(cval + r_hi);
                    for (uintptr_t l = l0 + 128 * static_cast<uintptr_t>(threadIdx.x); l < l1;
                         l += 128 * static_cast<uintptr_t>(kBmBlock))
                        l2_priority_normal(reinterpret_cast<const void *>(l));
                    if (threadIdx.x < nl) rm->rs[threadIdx.x] = re;
                    g = g2;
                    __syncthreads();
                }
                if (bad) set_error(w.err, DERR_WINDOW);
                done += cnt;
                __syncthreads();
                continue;
            }
            for (int64_t t = threadIdx.x; t < cnt; t += kBmBlock) st_keep(cval + t, 0.0, pol);
            __syncthreads();
            phase_end(4);
            // pass 2: each product lands on its column's rank (the walk
            // scratch of pass 1 is still in place)
            block_row_walk<kBmBlock, true, ITERS, 2, RUNS>(op, p0, p1, S, sc, [&](int key, double a, double b) {
                const unsigned rel = static_cast<unsigned>(key - c0i);
                if (rel < span32) {
                    const unsigned wi = rel >> 6, bi = rel & 63u;
                    // the column's own bit is set: bits 0..bi shifted to the
                    // top, counted, minus itself = columns before it in the word
                    const unsigned rank = pre[wi] +
                        static_cast<unsigned>(__popcll(bm[wi] << (63u - bi))) - 1u;
                    red_add_keep(cval + rank, a * b, pol);
                }
            }, &rsel);
            __syncthreads();
            phase_end(5);
            // back to normal priority: every 128-byte line the segment touches
            const uintptr_t l0 = reinterpret_cast<uintptr_t>(cval) & ~static_cast<uintptr_t>(127);
            const uintptr_t l1 = reinterpret_cast<uintptr_t>(cval + cnt);
            for (uintptr_t l = l0 + 128 * static_cast<uintptr_t>(threadIdx.x); l < l1;
                 l += 128 * static_cast<uintptr_t>(kBmBlock))
                l2_priority_normal(reinterpret_cast<const void *>(l));
            phase_end(6);
        }
        done += cnt;
        __syncthreads();
    }
    if (threadIdx.x == 0 && (!ok || done != n_expect)) set_error(w.err, DERR_COUNT_MISMATCH);
}

// --- kernel table ---------------------------------------------------------------
using NumFn = void (*)(Operands, BinWork);

#define NUM_TABLE(X)                 \
    X(8, 256, 32)                    \
    X(16, 256, 128)                  \
    X(32, 256, 256)                  \
    X(64, 64, 512)                   \
    X(128, 128, 1024)                \
    X(256, 256, 2048)                \
    X(512, 512, 4096)                \
    X(1024, 1024, 8192)              \
    X(1024, 1024, 18432)

struct NumEntry {
    KernelDesc d;
    NumFn fn;
};

// Largest row the table can sort in place: the bitonic network needs the
// next power of two of the row size to fit in the table.
constexpr long long pow2_floor(long long t) {
    long long p = 1;
    while (p * 2 <= t) p *= 2;
    return p;
}

// Row groups of a warp or less also get kStage B-piece slots per lane for
// the staged walk (12 bytes each).
#define NUM_ENTRY(TPR, BLOCK, T)                                                         \
    {{TPR, BLOCK, T, pow2_floor(T), 0,                                                   \
      (sizeof(int) + sizeof(double)) * (BLOCK / TPR) * (size_t)T +                       \
          (TPR > 32 ? sizeof(WalkScratch) : (sizeof(int) + sizeof(double)) * kStage * (size_t)BLOCK)}, \
     &num_hash_kernel<TPR, BLOCK, T>},

static NumEntry g_num[] = {NUM_TABLE(NUM_ENTRY)};

#define NUM_ONEPHASE_ENTRY(TPR, BLOCK, T) &num_hash_kernel<TPR, BLOCK, T, true>,
static NumFn g_num_onephase[] = {NUM_TABLE(NUM_ONEPHASE_ENTRY)};
// the plain kernels with the read-then-swap probe (BinWork::multi)
#define NUM_MULTI_ENTRY(TPR, BLOCK, T) &num_hash_kernel<TPR, BLOCK, T, false, true>,
static NumFn g_num_multi[] = {NUM_TABLE(NUM_MULTI_ENTRY)};
// The 512- and 1024-slot kernels with a warp per row instead of 64 and 128
// threads: no block barriers in the walk, the condense and the sort, values
// without atomics where B's rows are distinct and long, and rows of up to 512
// entries sorted in registers, which needs the column and the slot in one 32-bit
// key, so B has at most 2^23 columns. Bound by the chain of table probes.
// (Rows of about 190 entries of unstructured factors, 25,069 rows: 401 ->
// 132 us; about 290 entries, 7,482 rows: 239 -> 94 us; block-diagonal n = 2^20
// with 437 entries a row: 11.9 -> 9.5 ms.) Wider B takes the block kernels,
// which sort by a span bitmap or in shared memory, 64 and 128 threads wide;
// so do the read-then-swap probe and rows of many products (num_row_limits).
constexpr int64_t kWarpRowCols = int64_t{1} << 23;
// [0] every row, [1] with a queue; fn and one-phase.
#define NUM_WARP(TPR, BLOCK, T)                                                                  \
    {BLOCK, (sizeof(int) + sizeof(double)) * (BLOCK / 32 * (size_t)T + kStage * (size_t)BLOCK),  \
     {{&num_hash_kernel<32, BLOCK, T>, &num_hash_kernel<32, BLOCK, T, true>},                    \
      {&num_hash_kernel<32, BLOCK, T, false, false, true>, &num_hash_kernel<32, BLOCK, T, true, false, true>}}, \
     {&num_hash_kernel<TPR, TPR, T, false, false, true>, &num_hash_kernel<TPR, TPR, T, true, false, true>}}
static const struct {
    int block;
    size_t smem;
    NumFn fn[2][2];
    NumFn queued[2];   // the block form over the queue
} g_num_warp[] = {NUM_WARP(64, 128, 512), NUM_WARP(128, 64, 1024)};
constexpr int kNumWarpFirst = 3;   // kernels 3 and 4 of the table
constexpr int kNumWarp = sizeof(g_num_warp) / sizeof(g_num_warp[0]);

static constexpr int kNumHash = sizeof(g_num) / sizeof(g_num[0]);
static KernelDesc g_num_bitmap{1024, 1024, 0, LLONG_MAX, 1, 0};

using BmFn = void (*)(Operands, BinWork, int);
// bitmap kernel variants: (threads per block, products in flight per lane)
static const struct { int block, iters; BmFn fn; } g_num_bm[] = {
    {1024, 4, &num_bitmap_kernel<1024, 4>}, {1024, 8, &num_bitmap_kernel<1024, 8>},
    {512, 4, &num_bitmap_kernel<512, 4>},   {256, 4, &num_bitmap_kernel<256, 4>},
};
// the same walked by column windows over sorted B (BinWork::bidx set): two
// 512-thread blocks per SM when a window's bitmap takes half the SM
static const struct { int block; BmFn fn; } g_num_bm_runs[] = {
    {1024, &num_bitmap_kernel<1024, 4, true>}, {512, &num_bitmap_kernel<512, 4, true>},
};

int num_kernel_count() { return kNumHash + 1; }

const KernelDesc &num_kernel(int id) {
    return id < kNumHash ? g_num[id].d : g_num_bitmap;
}

cudaError_t num_prepare(int smem_optin) {
    // Opt in for every kernel: the 48 KB default covers static plus dynamic
    // shared memory, so a table of exactly 48 KB already needs it.
    for (int i = 0; i < kNumHash; ++i) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(g_num[i].fn),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(g_num[i].d.smem));
        if (e != cudaSuccess) return e;
    }
    for (int i = 0; i < kNumHash; ++i) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(g_num_onephase[i]),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(g_num[i].d.smem));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(reinterpret_cast<const void *>(g_num_multi[i]),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(g_num[i].d.smem));
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < kNumWarp; ++k)
        for (int phase = 0; phase < 2; ++phase) {
            const auto &v = g_num_warp[k];
            for (const NumFn fn : {v.fn[0][phase], v.fn[1][phase], v.queued[phase]}) {
                const size_t smem = fn == v.queued[phase] ? g_num[kNumWarpFirst + k].d.smem : v.smem;
                const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(fn),
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           static_cast<int>(smem));
                if (e != cudaSuccess) return e;
            }
        }
    g_num_bitmap.table = static_cast<long long>((smem_optin - sizeof(WalkScratch)) / 12) * 64;
    for (const auto &v : g_num_bm) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(v.fn),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return e;
    }
    for (const auto &v : g_num_bm_runs) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(v.fn),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Bitmap kernel launch shape: the block size that keeps about 2048 threads
// per SM given how many blocks fit in shared memory (one 1024-thread block
// when a block needs most of the SM's 228 KB, as for a million columns;
// 256-thread blocks when the bitmap is small), and `iters` products in
// flight per lane (4 or 8; 0 = 4).
static int pick_bitmap_variant(size_t smem_total, int iters) {
    const size_t per_sm = 228 * 1024;
    const int fit = static_cast<int>(per_sm / (smem_total + 1024));
    int block = 1024;
    if (fit >= 8) block = 256;
    else if (fit >= 4) block = 512;
    if (iters == 8) block = 1024;
    for (int i = 0; i < static_cast<int>(sizeof(g_num_bm) / sizeof(g_num_bm[0])); ++i)
        if (g_num_bm[i].block == block && g_num_bm[i].iters == (iters == 8 ? 8 : 4)) return i;
    return 0;
}

// The warp-per-row form of kernel `id` for these operands, -1: none.
static int warp_row_form(int id, const Operands &op, const BinWork &w) {
    const int k = id - kNumWarpFirst;
    return k >= 0 && k < kNumWarp && op.ncols <= kWarpRowCols &&
                   !w.multi && !w.block_rows ? k : -1;
}

bool num_has_warp_form(int id) { return id >= kNumWarpFirst && id < kNumWarpFirst + kNumWarp; }

// A warp takes a row without block barriers, but a row of many products keeps
// it long after the others, and the 1024-slot table leaves half as many warps
// on an SM as the block form has. Numeric phase, block and warp form in us, n
// entries a row (n = 200: 512 slots, 400: 1024 slots):
//   unsorted, n = 200, 6,400 products: 300 rows 87 and 125, 3,000 rows 209 and
//     149; n = 400, 1,200 products: 300 rows 31 and 43, 20,000 rows 311 and 325;
//     400 products: 300 rows 26 and 31, 3,000 rows 51 and 52, 9,000 rows 112 and 94;
//   a hub of 10^6 products among 30,000 short rows: 10,500 and 25,600;
//   by column, n = 400, B rows of 48: 2,400 products, 300 rows 33 and 42, 20,000
//     rows 368 and 297; B rows of 24, 2,400 products, 3,000 rows 83 and 63;
//   columns too far apart for a block's span bitmap, so that it sorts: n = 400,
//     2,400 products: 300 rows 58 and 71, 3,000 rows 155 and 135, 20,000 rows
//     925 and 628; 12,800 products, 20,000 rows 1,857 and 1,856.
// The limits lie where the two meet. Where B is not ascending the span is not
// known: in large bins of wide B 2,048 products (1,600 products, 20,000 rows: 389
// and 405 if a row's columns are close, 721 and 321 if far apart). What most rows are like is told from the
// mean lengths and B's width, and whole bins past their limit take the block
// form; a row is looked at, and sent to the block form's queue, only when some
// row passes that limit (Counters::longest, from the symbolic kernels): a queue
// that nothing needed cost 4 us to 8 us, one that held most rows of a bin up to
// 60% of its time.
bool num_row_limits(int id, const Operands &op, double na, double mean_b, long long most, BinWork &w) {
    w.long_col = w.long_near = w.long_far = LLONG_MAX;
    const int k = warp_row_form(id, op, w);
    if (k < 0) return false;
    const double mean = na * mean_b;
    const auto or_mean = [&](long long limit) { return std::max(limit, static_cast<long long>(4.0 * mean)); };
    const long long table = g_num[id].d.table;
    const bool narrow = op.ncols <= 8 * table;                        // no row is too wide for the span bitmap
    const bool fits = op.ncols <= table * 12 / 8 / 32 * 32;           // every row's span fits the accumulator
    if (k == 0) {
        const bool many = w.cnt >= 2048;
        w.long_col = or_mean(16384);
        w.long_near = many ? or_mean(1024) : 1024;
        w.long_far = many ? or_mean(4096) : 2048;
    } else {
        const bool many = w.cnt >= 16384;
        w.long_col = many ? or_mean(2048) : w.cnt >= 2048 ? 3072 : w.cnt >= 512 ? 2048 : 1024;
        w.long_near = many && !narrow && !w.by_column ? 2048 : !narrow || w.cnt >= 1024 ? 1024 : 0;
        w.long_far = many ? 8192 : w.cnt >= 2048 ? 3072 : 1536;
    }
    long long least, most_rows;   // limits of the rows that the bin may hold
    if (w.by_column && fits) {
        least = most_rows = w.long_col;
    } else if (w.by_column && !narrow) {
        least = std::min(w.long_col, w.long_far);
        most_rows = std::max(w.long_col, w.long_far);
    } else {
        least = most_rows = w.long_near;
    }
    if (most <= least) return false;
    if (w.lanes > 0 || mean > static_cast<double>(most_rows)) {   // fixed lanes: products are not counted
        w.block_rows = 1;
        return false;
    }
    return true;
}

// Kernel `id` in its warp-per-row form k, then the rows in the queue.
static cudaError_t launch_warp_rows(int k, int phase, const Operands &op, const BinWork &w, cudaStream_t s) {
    const auto &v = g_num_warp[k];
    const int64_t rpb = v.block / 32;
    v.fn[w.queue ? 1 : 0][phase]<<<static_cast<unsigned>((w.cnt + rpb - 1) / rpb), v.block, v.smem, s>>>(op, w);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !w.queue) return e;
    const KernelDesc &d = g_num[kNumWarpFirst + k].d;
    v.queued[phase]<<<static_cast<unsigned>(std::min<int64_t>(w.cnt, w.queue_grid)), d.block, d.smem, s>>>(op, w);
    return cudaGetLastError();
}

cudaError_t launch_num_onephase(int id, const Operands &op, const BinWork &w, cudaStream_t s) {
    if (w.cnt <= 0) return cudaSuccess;
    if (id < 0 || id >= kNumHash) return cudaErrorInvalidValue;
    if (const int k = warp_row_form(id, op, w); k >= 0) return launch_warp_rows(k, 1, op, w, s);
    const KernelDesc &d = g_num[id].d;
    const int rpb = d.block / d.tpr;
    const int64_t grid = (w.cnt + rpb - 1) / rpb;
    g_num_onephase[id]<<<static_cast<unsigned>(grid), d.block, d.smem, s>>>(op, w);
    return cudaGetLastError();
}

// Copies the one-phase rows of a bin from their temporary slots into C: one
// warp per row, rows marked -1 in pred (mispredicted) are skipped.
template <bool COLS, bool VALS>
__global__ void copy_rows_kernel(BinWork w) {
    const int64_t r = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= w.cnt) return;
    const int64_t row = w.bins ? static_cast<int64_t>(w.bins[w.off + r]) : w.off + r;
    if (w.pred[row] < 0) return;
    const int64_t base = w.crpt[row];
    const int64_t n = w.crpt[row + 1] - base;
    const int32_t *scol = w.tcol + w.tbase + r * w.tcap;
    const double *sval = w.tval + w.tbase + r * w.tcap;
    if (n > w.tcap || w.tbase + r * w.tcap + n > w.tlimit) {
        if (lane == 0) set_error(w.err, DERR_BOUNDS);
        return;
    }
    // four loads in flight per lane before the stores (the temporary rows
    // are read-only here)
    for (int64_t t0 = 0; t0 < n; t0 += 128) {
        int32_t c[4];
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t t = t0 + u * 32 + lane;
            if (COLS && t < n) c[u] = __ldg(scol + t);
            if (VALS && t < n) v[u] = __ldg(sval + t);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t t = t0 + u * 32 + lane;
            if (COLS && t < n) w.ccol[base + t] = c[u];
            if (VALS && t < n) w.cval[base + t] = v[u];
        }
    }
}

cudaError_t launch_copy_rows(const BinWork &w, bool cols, bool vals, cudaStream_t s) {
    if (w.cnt <= 0) return cudaSuccess;
    const int64_t threads = w.cnt * 32;
    const auto kernel = !vals ? &copy_rows_kernel<true, false>
                              : !cols ? &copy_rows_kernel<false, true> : &copy_rows_kernel<true, true>;
    kernel<<<static_cast<unsigned>((threads + 255) / 256), 256, 0, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_num(int id, const Operands &op, const BinWork &w, size_t smem_bitmap,
                       cudaStream_t s) {
    if (w.cnt <= 0) return cudaSuccess;
    if (const int k = warp_row_form(id, op, w); k >= 0) return launch_warp_rows(k, 0, op, w, s);
    if (id < kNumHash) {
        const KernelDesc &d = g_num[id].d;
        const int rpb = d.block / d.tpr;
        const int64_t grid = (w.cnt + rpb - 1) / rpb;
        const NumFn fn = w.multi ? g_num_multi[id] : g_num[id].fn;
        fn<<<static_cast<unsigned>(grid), d.block, d.smem, s>>>(op, w);
    } else {
        const int words = static_cast<int>(smem_bitmap / 12);
        BinWork wk = w;
        wk.head = static_cast<int>(num_bitmap_head_bytes(w.bs != nullptr));
        if (!w.bs) wk.wlists = 0;
        const size_t smem = smem_bitmap + static_cast<size_t>(wk.head);
        if (w.bidx && !w.bs) {
            // two blocks per SM when two windows fit the SM's shared memory
            const int two = (228 * 1024) / static_cast<int>(smem + 1024) >= 2;
            const auto &v = g_num_bm_runs[two ? 1 : 0];
            v.fn<<<static_cast<unsigned>(w.cnt), v.block, smem, s>>>(op, wk, words);
            return cudaGetLastError();
        }
        const auto &v = g_num_bm[pick_bitmap_variant(smem, w.unroll)];
        v.fn<<<static_cast<unsigned>(w.cnt), v.block, smem, s>>>(op, wk, words);
    }
    return cudaGetLastError();
}

}  // namespace ops
