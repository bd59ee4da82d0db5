// Rows of C whose column pattern repeats the row before (the symbolic and
// numeric phases of Sec. 2.2 for structured operators).
//
// On a structured grid, in a band matrix or in a system with several unknowns
// per point, row i of A mostly has the columns of row i - 1 (unknowns of one
// point) or those columns plus one (the next point), and so has B. Then row i
// of C has the pattern of row i - 1, unchanged or moved by one:
//   A's columns unchanged                                 -> C's unchanged;
//   A's columns plus one, every B row that they reference
//   is the B row before it plus one                       -> C's plus one.
// Such a row needs no symbolic work (its size is the size of the row it goes
// back to), no hash probes and no sort: the products fall on the same ranks
// in the row as the products of the row it goes back to. row_patterns_kernel
// compares neighbouring rows of A and B, repeats_kernel marks the repeating
// rows of C in words of 32 rows, and after the rows that they go back to are
// complete repeat_numeric_kernel builds one map (product -> rank) per run of
// repeating rows and adds every row's products by it.
#include <climits>

#include "common.cuh"
#include "internal.h"

namespace ops {

// Threads per row for `entries` entries in `rows` rows: about four entries each.
static int row_lanes(int64_t entries, int64_t rows) {
    int l = 1;
    while (l < 32 && static_cast<int64_t>(l) * 4 * rows < entries) l <<= 1;
    return l;
}

// A row is compared only with a row of its own length, and a thread stops at
// the first entry that fits neither pattern, so rows without structure cost
// their row pointers and a few entries.
__global__ void __launch_bounds__(256)
row_patterns_kernel(const void *rpt, int is64, const int32_t *col, int64_t first, int64_t n, int L, uint8_t *code,
                    unsigned long long *found, RepGate gate) {
    if (gate.shut()) return;   // uniform over the grid
    const int64_t i = (static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x) / L;
    const int l = threadIdx.x & (L - 1);
    unsigned same = 0, moved = 0;
    if (i > 0 && i < n) {
        const int64_t r = first + i;
        const int64_t s0 = ld_rpt(rpt, is64, r - 1), s = ld_rpt(rpt, is64, r), e = ld_rpt(rpt, is64, r + 1);
        const int64_t len = e - s;
        if (len == s - s0 && len > 0 && len <= kRepMaxNnz) {
            same = moved = 1;
            for (int64_t p = l; p < len && (same | moved); p += L) {
                const int d = __ldg(col + s + p) - __ldg(col + s0 + p);
                same &= d == 0;
                moved &= d == 1;
            }
        }
    }
    for (int o = L >> 1; o > 0; o >>= 1) {
        same &= __shfl_xor_sync(0xffffffffu, same, o);
        moved &= __shfl_xor_sync(0xffffffffu, moved, o);
    }
    if (l == 0 && i < n) code[i] = static_cast<uint8_t>(moved | (same << 1));
    const int hits = __syncthreads_count(l == 0 && (moved | same));
    if (found && threadIdx.x == 0 && hits) atomicAdd(found, static_cast<unsigned long long>(hits));
}

// One warp per word of 32 rows; L threads per row look up the codes of the B
// rows that it references.
__global__ void __launch_bounds__(256)
repeats_kernel(Operands op, int L, const uint8_t *acode, const uint8_t *bcode, RepWord *words, int64_t nwords,
               RepGate gate) {
    const int64_t word = (static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x) >> 5;
    if (word >= nwords) return;   // uniform over the warp
    const int lane = threadIdx.x & 31, l = lane & (L - 1), per = 32 / L;
    unsigned fol = 0, one = 0;
    const bool shut = gate.shut();
    for (int j = 0; j < L && !shut; ++j) {
        const int b = j * per + lane / L;
        const int64_t i = word * 32 + b;
        const unsigned code = i % kRepSpan && i < op.mw ? acode[i] : 0u;
        unsigned ok = 0;
        if (code) {
            const int64_t s = ld_rpt(op.arpt, op.a64, op.row0 + i), e = ld_rpt(op.arpt, op.a64, op.row0 + i + 1);
            ok = e - s <= kRepMaxLen;
            if (!(code & 2u))
                for (int64_t p = s + l; p < e && ok; p += L) ok = bcode[__ldg(op.acol + p)] & 1u;
        }
        for (int o = L >> 1; o > 0; o >>= 1) ok &= __shfl_xor_sync(0xffffffffu, ok, o);
        if (ok) {
            fol |= 1u << b;
            if (!(code & 2u)) one |= 1u << b;
        }
    }
    fol = __reduce_or_sync(0xffffffffu, fol);
    one = __reduce_or_sync(0xffffffffu, one);
    // short runs do not pay for their rank map
    static_assert(kRepMinRun == 4, "two steps of doubling");
    unsigned keep = fol & (fol >> 1);
    keep &= keep >> 2;
    keep |= keep << 1;
    keep |= keep << 2;
    if (lane == 0) words[word] = RepWord{keep, one & keep, 0, 0};
}

// One warp per word: where a run that begins at bit 0 goes back to (at most
// kRepSpan - 1 rows), the products of the repeating rows, and the runs that
// have too many or none.
__global__ void __launch_bounds__(256)
repeats_finish_kernel(int64_t *nprod, long long max_prod, const RepWord *words, RepWord *out,
                      int64_t nwords) {
    const int64_t word = (static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x) >> 5;
    if (word >= nwords) return;   // uniform over the warp
    const int lane = threadIdx.x & 31;
    RepWord w = words[word];
    if (w.fol & 1u) {   // uniform; word > 0: row 0 does not repeat
        for (int64_t v = word - 1;; --v) {
            const RepWord x = words[v];
            const unsigned clear = ~x.fol;
            const int top = clear ? 31 - __clz(clear) : -1;   // the last row of the word that does not repeat
            w.back += 31 - top;
            w.moved += __popc(top < 0 ? x.one : x.one & ~((2u << top) - 1u));   // 2u << 31 is 0: no row
            if (clear) break;
        }
        w.back += 1;
    }
    const int64_t i = word * 32 + lane;
    bool keep = false;
    if ((w.fol >> lane) & 1u) {
        const int64_t np = nprod[rep_own(w, i)];
        nprod[i] = np;
        keep = np > 0 && np <= max_prod;
    }
    w.fol = __ballot_sync(0xffffffffu, keep);
    w.one &= w.fol;
    if (lane == 0) out[word] = w;
}

// One block per word of 32 rows, its runs of repeating rows in turn. For a
// run, the block reads the columns of the row that the run goes back to, maps
// every product to its rank there (binary search), and groups of G threads
// then take two repeating rows each: one piece of at most G products of one B
// row per step (distinct columns, so no atomics), b loaded with unit stride,
// accumulated in shared memory by rank. Sums run in the order of A's entries,
// as in the warp-row hash kernels. G is the power of two with the fewest
// float64 steps for the run, the larger of nearly equal ones: a step costs 16
// cycles of the SM's float64 pipe (2 multiply-adds a cycle), and more than
// that in the load-store pipe when it touches many separate lines. Two rows
// per group share the reads of the map and the lengths, and their steps
// overlap (one row per group: 4.77 ms instead of 4.11 for the rows of the
// 27-point stencil 128^3). What bounds it: the float64 pipe, 65% busy on that
// stencil (2.7 ms if it never waited), next to it the shared-memory reads and
// writes of the accumulators, 68%. Whole products, every row by the hash
// kernels and this way: 27-point stencil 128^3 13.59 -> 5.40 ms, band of 65
// columns and 2^17 rows 5.19 -> 1.90 ms, 5-point grid 1024^2 1.30 -> 0.46 ms.
// Short rows (class 0) run more warps with fewer registers: they wait for
// the chain of loads before a row's first product (5-point grid: 311 -> 241 us).
struct __align__(16) RepEntry {
    double a;       // A's value
    long long q;    // first entry of its B row, -1: leave it out
};

template <int CLS>
__global__ void __launch_bounds__(kRepClass[CLS].threads, (CLS == 0 ? 1280 : 768) / kRepClass[CLS].threads)
repeat_numeric_kernel(Operands op, const RepWord *words, const int64_t *crpt, int32_t *ccol, double *cval, int *err,
                      int present) {
    constexpr RepClass K = kRepClass[CLS];
    constexpr int kWarps = K.threads / 32;
    constexpr int kAccs = K.accs * (K.max_nnz + 1);   // accumulator entries
    constexpr int kU = CLS == 0 ? 2 : 4;              // products of a row that a lane loads before using any
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *acc = reinterpret_cast<double *>(smem_raw);
    int *scol = reinterpret_cast<int *>(acc + kAccs);                           // columns of the first row
    uint16_t *map = reinterpret_cast<uint16_t *>(scol + K.max_nnz);             // rank of every product
    __shared__ RepEntry s_ent[kWarps][2][32];
    __shared__ long long s_q[kRepMaxLen];
    __shared__ int s_len[kRepMaxLen], s_pre[kRepMaxLen];
    __shared__ int s_prod, s_lg, s_long;
    const RepWord rw = words[blockIdx.x];
    const int64_t row0 = static_cast<int64_t>(blockIdx.x) * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool bad = false;
    for (uint32_t m = rw.fol; m;) {   // uniform over the block
        const int s = __ffs(m) - 1;
        const uint32_t ends = ~(m >> s);
        const int cnt = ends ? __ffs(ends) - 1 : 32;
        m = s + cnt < 32 ? m & (0xffffffffu << (s + cnt)) : 0u;
        const int64_t own = s > 0 ? row0 + s - 1 : row0 - rw.back;   // the row that the run goes back to
        const int64_t cb = crpt[own];
        const int64_t n64 = crpt[own + 1] - cb;
        if (n64 > kRepMaxNnz) continue;   // binned as rows of their own
        const int n = static_cast<int>(n64);
        const int64_t p0 = ld_rpt(op.arpt, op.a64, op.row0 + own);
        const int64_t alen64 = ld_rpt(op.arpt, op.a64, op.row0 + own + 1) - p0;
        if (alen64 <= 0 || alen64 > kRepMaxLen) {   // another structure than the symbolic phase saw
            bad = true;
            continue;
        }
        const int alen = static_cast<int>(alen64);
        __syncthreads();   // readers of the run before are done
        for (int t = threadIdx.x; t < alen; t += K.threads) {
            const int k = __ldg(op.acol + p0 + t);
            const int64_t q = ld_rpt(op.brpt, op.b64, k);
            const int64_t len = ld_rpt(op.brpt, op.b64, k + 1) - q;
            s_q[t] = q;
            s_len[t] = static_cast<int>(len < kRepMaxProd + 1 ? len : kRepMaxProd + 1);
        }
        __syncthreads();
        const int stride = n | 1, fit = kAccs / stride;   // accumulators that fit
        if (warp == 0) {
            // products before each entry (at most kRepMaxLen * kRepMaxProd) and
            // float64 steps per row for groups of 8, 16 and 32 threads
            int run = 0, c8 = 0, c16 = 0, c32 = 0, big = 0;
            for (int t0 = 0; t0 < alen; t0 += 32) {
                const int len = t0 + lane < alen ? s_len[t0 + lane] : 0;
                int inc = len;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                if (t0 + lane < alen) s_pre[t0 + lane] = run + inc - len;
                run += __shfl_sync(0xffffffffu, inc, 31);
                c8 += (len + 7) >> 3;
                c16 += (len + 15) >> 4;
                c32 += (len + 31) >> 5;
                big = max(big, len);
            }
            c8 = __reduce_add_sync(0xffffffffu, c8);
            c16 = __reduce_add_sync(0xffffffffu, c16);
            c32 = __reduce_add_sync(0xffffffffu, c32);
            big = __reduce_max_sync(0xffffffffu, big);
            // warp steps for the run: rounds of at most 2 / 4 / 8 rows per
            // warp, as many rows at once as there are accumulators
            const int g32 = min(2 * kWarps, fit), g16 = min(4 * kWarps, fit), g8 = min(8 * kWarps, fit);
            const int w32 = (cnt + g32 - 1) / g32 * ((g32 + 1) >> 1) * c32;
            const int w16 = (cnt + g16 - 1) / g16 * ((g16 + 3) >> 2) * c16;
            const int w8 = (cnt + g8 - 1) / g8 * ((g8 + 7) >> 3) * c8;
            int lg = 5, best = w32;
            if (10 * w16 < 9 * best) {
                lg = 4;
                best = w16;
            }
            if (10 * w8 < 9 * best) lg = 3;
            if (lane == 0) {
                s_prod = run;
                s_lg = lg;
                s_long = big > (1 << lg);
            }
        }
        __syncthreads();
        // the first launched class that takes the run
        const int cls = rep_class(s_prod, n);
        const int take = cls < 0 ? 0 : __ffs(present >> cls);
        if (take == 0 || cls + take - 1 != CLS) {
            bad |= take == 0;
            continue;
        }
        const int lg = s_lg, G = 1 << lg, l = lane & (G - 1), sub = threadIdx.x >> lg;
        const int rows = min(2 * (K.threads >> lg), fit);   // rows at once
        for (int j = threadIdx.x; j < n; j += K.threads) scol[j] = ccol[cb + j];
        for (int j = threadIdx.x; j < rows * stride; j += K.threads) acc[j] = 0.0;
        __syncthreads();
        // four entries of A per warp at once: their loads and searches overlap
        for (int t = warp * 4; t < alen; t += kWarps * 4) {
            int big = 0;
            for (int u = 0; u < 4 && t + u < alen; ++u) big = max(big, s_len[t + u]);
            for (int o = lane; o < big; o += 32) {
                int c[4], lo[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    c[u] = t + u < alen && o < s_len[t + u] ? __ldg(op.bcol + s_q[t + u] + o) : -1;
                    lo[u] = 0;
                }
                // last rank with scol <= c: the interval [lo, lo + width) halves, the same width for every column
                for (int width = n; width > 1;) {
                    const int half = width >> 1;
#pragma unroll
                    for (int u = 0; u < 4; ++u) lo[u] = scol[lo[u] + half] <= c[u] ? lo[u] + half : lo[u];
                    width -= half;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (c[u] >= 0) {
                        bad |= scol[lo[u]] != c[u];
                        map[s_pre[t + u] + o] = static_cast<uint16_t>(lo[u]);
                    }
            }
        }
        __syncthreads();
        // rows base + 2 * sub and the one after it; rows that do not exist
        // take part with no products
        const int slot = min(2 * sub, rows - 1);
        double *my0 = acc + slot * stride;
        double *my1 = acc + min(slot + 1, rows - 1) * stride;
        RepEntry *ent0 = &s_ent[warp][0][lane & ~(G - 1)];
        RepEntry *ent1 = &s_ent[warp][1][lane & ~(G - 1)];
        const bool one_piece = !s_long;
        for (int base = 0; base < cnt; base += rows) {
            const int w0 = 2 * ((warp * 32) >> lg);   // the warp's first row of this round
            if (w0 >= rows || base + w0 >= cnt) continue;   // uniform over the warp
            const int64_t row = row0 + s + base + 2 * sub;
            const bool act0 = 2 * sub < rows && base + 2 * sub < cnt;
            const bool act1 = 2 * sub + 1 < rows && base + 2 * sub + 1 < cnt;
            int64_t ap0 = 0, ap1 = 0;
            bool fits0 = false, fits1 = false;
            if (act0) {
                ap0 = ld_rpt(op.arpt, op.a64, op.row0 + row);
                ap1 = ld_rpt(op.arpt, op.a64, op.row0 + row + 1);
                fits0 = ap1 - ap0 == alen;
                if (act1) fits1 = ld_rpt(op.arpt, op.a64, op.row0 + row + 2) - ap1 == alen;
                bad |= !fits0 || (act1 && !fits1);
            }
            for (int c = 0; c < alen; c += G) {
                __syncwarp();   // readers of the chunk before are done
                {
                    RepEntry x{0.0, -1}, y{0.0, -1};
                    if (c + l < alen) {
                        const int len = s_len[c + l];
                        const int kx = fits0 ? __ldg(op.acol + ap0 + c + l) : -1;
                        const int ky = fits1 ? __ldg(op.acol + ap1 + c + l) : -1;
                        if (fits0) x.a = __ldg(op.aval + ap0 + c + l);
                        if (fits1) y.a = __ldg(op.aval + ap1 + c + l);
                        if (kx >= 0) {
                            x.q = ld_rpt(op.brpt, op.b64, kx);
                            if (ld_rpt(op.brpt, op.b64, kx + 1) - x.q != len) x.q = -1;
                        }
                        if (ky >= 0) {
                            y.q = ld_rpt(op.brpt, op.b64, ky);
                            if (ld_rpt(op.brpt, op.b64, ky + 1) - y.q != len) y.q = -1;
                        }
                        bad |= (kx >= 0 && x.q < 0) || (ky >= 0 && y.q < 0);
                    }
                    ent0[l] = x;
                    ent1[l] = y;
                }
                __syncwarp();
                const int ce = alen - c < G ? alen - c : G;
                int pre = s_pre[c];
                if (one_piece) {
                    for (int e = 0; e < ce; e += kU) {   // uniform over the warp
                        double b0[kU], b1[kU], a0[kU], a1[kU];
                        int r[kU];
#pragma unroll
                        for (int u = 0; u < kU; ++u) {
                            r[u] = -1;
                            a0[u] = a1[u] = b0[u] = b1[u] = 0.0;
                            if (e + u < ce) {
                                const int len = s_len[c + e + u];
                                const RepEntry x = ent0[e + u], y = ent1[e + u];
                                a0[u] = x.a;
                                a1[u] = y.a;
                                if (l < len) {
                                    r[u] = map[pre + l];
                                    if (x.q >= 0) b0[u] = __ldg(op.bval + x.q + l);
                                    if (y.q >= 0) b1[u] = __ldg(op.bval + y.q + l);
                                }
                                pre += len;
                            }
                        }
#pragma unroll
                        for (int u = 0; u < kU; ++u) {
                            if (r[u] >= 0) {
                                const double v0 = my0[r[u]], v1 = my1[r[u]];
                                if (act0) my0[r[u]] = fma(a0[u], b0[u], v0);
                                if (act1) my1[r[u]] = fma(a1[u], b1[u], v1);
                            }
                            __syncwarp();
                        }
                    }
                } else {
                    for (int e = 0; e < ce; ++e) {
                        const int len = s_len[c + e];
                        const RepEntry x = ent0[e], y = ent1[e];
                        for (int o = 0; o < len; o += kU * G) {   // distinct columns: no two updates meet
                            double b0[kU], b1[kU];
                            int r[kU];
#pragma unroll
                            for (int u = 0; u < kU; ++u) {
                                const int at = o + u * G + l;
                                r[u] = -1;
                                b0[u] = b1[u] = 0.0;
                                if (at < len) {
                                    r[u] = map[pre + at];
                                    if (x.q >= 0) b0[u] = __ldg(op.bval + x.q + at);
                                    if (y.q >= 0) b1[u] = __ldg(op.bval + y.q + at);
                                }
                            }
#pragma unroll
                            for (int u = 0; u < kU; ++u)
                                if (r[u] >= 0) {
                                    const double v0 = my0[r[u]], v1 = my1[r[u]];
                                    if (act0) my0[r[u]] = fma(x.a, b0[u], v0);
                                    if (act1) my1[r[u]] = fma(y.a, b1[u], v1);
                                }
                        }
                        __syncwarp();
                        pre += len;
                    }
                }
            }
            auto store = [&](int64_t i, double *my) {
                const int64_t ob = crpt[i];
                if (crpt[i + 1] - ob != n) {
                    bad = true;
                    return;
                }
                // columns moved by one per `one` row since the first row
                const uint32_t upto = (2u << (i & 31)) - 1u;
                const int move = s > 0 ? __popc(rw.one & upto & (0xffffffffu << s)) : rw.moved + __popc(rw.one & upto);
                for (int j = l; j < n; j += G) {
                    ccol[ob + j] = scol[j] + move;
                    cval[ob + j] = my[j];
                    my[j] = 0.0;
                }
            };
            if (act0) store(row, my0);
            if (act1) store(row + 1, my1);
        }
    }
    if (bad) set_error(err, DERR_COUNT_MISMATCH);
}

template <int CLS>
constexpr size_t rep_smem() {
    constexpr RepClass K = kRepClass[CLS];
    return sizeof(double) * (size_t)K.accs * (K.max_nnz + 1) + sizeof(int) * (size_t)K.max_nnz +
           sizeof(uint16_t) * (size_t)K.max_prod;
}

template <int CLS>
static cudaError_t prepare_class() {
    if constexpr (CLS < kRepClasses) {
        const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&repeat_numeric_kernel<CLS>),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   static_cast<int>(rep_smem<CLS>()));
        return e != cudaSuccess ? e : prepare_class<CLS + 1>();
    }
    return cudaSuccess;
}

cudaError_t rep_prepare() { return prepare_class<0>(); }

template <int CLS>
static cudaError_t launch_class(int cls, int present, const Operands &op, const RepWord *words, const int64_t *crpt,
                                int32_t *ccol, double *cval, int *err, cudaStream_t s) {
    if constexpr (CLS < kRepClasses) {
        if (cls != CLS) return launch_class<CLS + 1>(cls, present, op, words, crpt, ccol, cval, err, s);
        repeat_numeric_kernel<CLS><<<static_cast<unsigned>((op.mw + 31) / 32), kRepClass[CLS].threads,
                                     rep_smem<CLS>(), s>>>(op, words, crpt, ccol, cval, err, present);
        return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_repeat_numeric(int cls, int present, const Operands &op, const RepWord *words, const int64_t *crpt,
                                  int32_t *ccol, double *cval, int *err, cudaStream_t s) {
    return launch_class<0>(cls, present, op, words, crpt, ccol, cval, err, s);
}

cudaError_t launch_row_patterns(const void *rpt, int is64, const int32_t *col, int64_t first, int64_t n,
                                int64_t entries, uint8_t *code, unsigned long long *found, const RepGate &gate,
                                cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int L = row_lanes(entries, n);
    row_patterns_kernel<<<static_cast<unsigned>((n * L + 255) / 256), 256, 0, s>>>(rpt, is64, col, first, n, L, code,
                                                                                        found, gate);
    return cudaGetLastError();
}

cudaError_t launch_repeats(const Operands &op, int64_t annz, const uint8_t *acode, const uint8_t *bcode,
                           RepWord *words, const RepGate &gate, cudaStream_t s) {
    if (op.mw <= 0) return cudaSuccess;
    const int L = row_lanes(annz, op.mw);
    const int64_t nwords = (op.mw + 31) / 32;
    repeats_kernel<<<static_cast<unsigned>((nwords + 7) / 8), 256, 0, s>>>(op, L, acode, bcode, words, nwords, gate);
    return cudaGetLastError();
}

cudaError_t launch_repeats_finish(int64_t mw, int64_t *nprod, long long max_prod, const RepWord *words, RepWord *out,
                                  cudaStream_t s) {
    if (mw <= 0) return cudaSuccess;
    const int64_t nwords = (mw + 31) / 32;
    repeats_finish_kernel<<<static_cast<unsigned>((nwords + 7) / 8), 256, 0, s>>>(nprod, max_prod, words, out, nwords);
    return cudaGetLastError();
}

}  // namespace ops
