// Internal interface between the host orchestration (api.cu) and the kernel
// translation units. Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ops {

constexpr int kMaxBins = 16;

// Learned sizing, load feedback: each class of rows (the numeric bin of a
// row's predicted size) has a factor 2^k on its predicted sizes,
// |k| <= kMaxFactorLog2. The one-phase kernels count, per class, the rows
// tried (group 0), those that ended more than 3/4 full (1), those that the
// next smaller table would hold at most 3/4 full (2) and the mispredicted
// ones (3), each spread over kLoadSlots counters (by block) against
// contention: counter (group * kMaxBins + class) * kLoadSlots + slot.
constexpr int kMaxFactorLog2 = 4;
constexpr int kLoadSlots = 8;
constexpr int kFbGroups = 4;
constexpr int kFbCounters = kFbGroups * kMaxBins * kLoadSlots;

struct SizeFactors {
    long long lim[kMaxBins];   // class j: sizes in (lim[j-1], lim[j]]; the last class takes the rest
    int k[kMaxBins];           // exponent of each class's factor
    int nb;
};

// Operands of one SpGEMM row window, as the kernels see them.
struct Operands {
    const void *arpt; int a64; const int32_t *acol; const double *aval;
    const void *brpt; int b64; const int32_t *bcol; const double *bval;
    int64_t row0;   // A row of window row 0
    int64_t mw;     // rows in the window
    int64_t ncols;  // columns of B (and C)
};

// What one bin kernel launch works on.
struct BinWork {
    const int32_t *bins;  // window row ids grouped by bin; nullptr = identity
    int64_t off, cnt;     // this bin's slice of `bins`
    int64_t *crpt;        // window C.rpt (int64, mw + 1)
    int32_t *ccol;        // numeric only
    double *cval;         // numeric only
    int lanes;            // threads per B row, 0 = per-row automatic
    int unroll;           // bitmap kernels: products in flight per lane (4 or 8; 0 = 4)
    int multi;            // plain hash kernels: read a slot before its compare-and-swap
    int distinct;         // every row of B has strictly ascending columns (checked): warp-row
                          // kernels may bound a row's columns by the ends of its B rows, and
                          // update values without atomics
    int by_column;        // numeric phase, with distinct: B's rows are long enough for a warp to
                          // add rows by column (span_rows)
    // warp-per-row forms of block-per-row numeric kernels (num_row_limits): rows of
    // more products than their limit go to the queue, for the block form
    long long long_col, long_near, long_far;
    int32_t *queue;       // places in the bin (room for cnt), nullptr: every row is taken
    unsigned *queued;     // their number (0 before)
    int queue_grid;       // blocks of the block form's launch over the queue, at most
    int block_rows;       // every row by the block form
    unsigned long long *longest;   // symbolic kernels: Counters::longest (nullptr: not wanted)
    int *err;             // device error word
    // numeric bitmap kernel, pass 2 by column windows (B rows sorted)
    const int32_t *bs;    // run boundaries of B rows at the sub-ranges (G + 1 per row), or nullptr
    int G, gshift;        // sub-ranges of 2^gshift columns
    int wlists;           // rows with more A entries use the whole-row pass 2
    int wentries;         // C entries per window, about
    int head;             // shared bytes before the bitmap (set by launch_num)
    // one-phase (learned sizing) numeric kernels only
    int32_t *tcol;        // temporary rows: bin-local row r of this bin at
    double *tval;         //   tcol/tval + tbase + r * tcap
    long long tbase, tcap;
    long long tlimit;     // entries of tcol/tval (bounds check)
    long long *pred;      // predicted sizes; set to -1 for a row that overflowed
    int32_t *xlist;       // rows for the exact path (overflowed rows are appended)
    unsigned long long *xcount;
    long long xlimit;     // entries of xlist (bounds check)
    const uint8_t *lcls;  // class of each window row (the bin of its prediction)
    unsigned long long *fb;   // load feedback counters (kFbCounters), or nullptr
    long long tprev;      // slots of the next smaller table (0: none)
    // symbolic bitmap kernel: per-cell entry counts for the column-window
    // numeric kernel (nullptr: not wanted)
    uint16_t *cells;      // bin-local row r: cells[r * ncells + c] = entries in cell c
    int32_t *cslot;       // window row -> its bin-local index in this bin
    int cs, ncells;       // cells of 2^cs columns
    // numeric bitmap kernel over several column windows with rows of B
    // sorted: cell index of the long B rows, so each window walks only its runs
    const int32_t *bslot;
    const int32_t *bidx;
    // symbolic bitmap kernel: bit 0 set = some row of B is not sorted (the
    // runs are then not used); nullptr = B known sorted
    const unsigned long long *bflags;
    // numeric bitmap kernel (whole-row form): per-phase SM clock sums
    // (kPhaseClocks), or nullptr; a profiling aid
    unsigned long long *clk;
};

// Phases of the numeric bitmap kernel that spgemm_bitmap_phase_clocks reports.
constexpr int kPhaseClocks = 7;

struct Ranges {
    long long r[kMaxBins];
    int nb;
};

// --- repeated rows (repeat.cu) ------------------------------------------------
// 32 consecutive window rows: bit b of `fol` set when row b's columns in C are
// those of the row before, all moved by one when bit b of `one` is set too.
// A run of repeating rows goes back to the last row before it whose bit is
// clear: a row of the same word or, when the run begins at bit 0, the row
// `back` rows before the word, with `moved` moves by one after that row and
// before the word. A run ends at the next multiple of kRepSpan rows.
struct __align__(16) RepWord {
    uint32_t fol, one;
    int32_t back, moved;
};
constexpr int kRepSpan = 256;

#ifdef __CUDACC__
// The row that repeating row i goes back to.
__device__ __forceinline__ int64_t rep_own(const RepWord &w, int64_t i) {
    const unsigned below = ~w.fol & ((1u << (i & 31)) - 1u);
    return below ? (i & ~int64_t{31}) + 31 - __clz(below) : (i & ~int64_t{31}) - w.back;
}
#endif

// Repeating rows by products and entries of C per row: one launch per class
// (threads per block, products in the rank map, accumulator entries).
struct RepClass {
    int threads;
    int max_prod, max_nnz;
    int accs;   // accumulators of max_nnz entries that the shared memory holds
};
constexpr int kRepClasses = 4;
constexpr RepClass kRepClass[kRepClasses] = {
    {128, 256, 64, 16}, {128, 1024, 256, 8}, {256, 4608, 512, 8}, {256, 18432, 1024, 7}};
constexpr int kRepMaxLen = 256;                                  // A entries of a repeating row
constexpr int kRepMaxProd = kRepClass[kRepClasses - 1].max_prod;
constexpr int kRepMaxNnz = kRepClass[kRepClasses - 1].max_nnz;   // larger rows are multiplied on their own
constexpr int kRepMinRun = 4;                                    // repeating rows in a row, at least
// When the symbolic phase looks for repeating rows (rows of the window, and
// products per row estimated from the mean lengths of A's and B's rows): the
// scans and extra launches cost 30 us to 40 us on products of that size, and
// a run's map about 10 us before its rows start. 27-point stencil, whole
// product without and with: 26^3 (11M products) 319 and 336 us, 32^3 (24M)
// 378 and 359, 48^3 1118 and 632; tridiagonal, 2^19 rows of 9 products, 428
// and 232 us. Rows of fewer products cost the hash kernels no more than the
// map (7-point times piecewise-constant prolongation, 7 products).
constexpr int64_t kRepMinRows = 4096;
constexpr int64_t kRepManyRows = 32768;
constexpr double kRepManyProducts = 16e6;
constexpr double kRepMinProducts = 8.0;

// First class that takes rows of `prod` products and `nnz` entries, -1: none.
template <int C = 0>
__host__ __device__ __forceinline__ int rep_class(long long prod, long long nnz) {
    if constexpr (C < kRepClasses) {
        constexpr RepClass k = kRepClass[C];
        return prod <= k.max_prod && nnz <= k.max_nnz ? C : rep_class<C + 1>(prod, nnz);
    } else {
        return -1;
    }
}

// The work that follows a pattern scan is skipped when the scan found fewer
// than `least` rows (found nullptr: never skipped).
struct RepGate {
    const unsigned long long *found = nullptr;
    unsigned long long least = 0;
#ifdef __CUDACC__
    __device__ __forceinline__ bool shut() const { return found && __ldcg(found) < least; }
#endif
};

// What a binning pass does with repeating rows: it leaves them out of the
// bins when their size is at most max_nnz, and with `fill` writes the size of
// the row they repeat over their own first (words nullptr: no such rows).
// nprod, read with `fill`: n_prod of the repeating rows, which their class
// depends on; nullptr: the sizes hold it (no pass has filled them in yet).
struct RepArgs {
    const RepWord *words = nullptr;
    int64_t *fill = nullptr;
    const int64_t *nprod = nullptr;
    long long max_nnz = 0;
};

// Counters written by the binning passes (device memory, zeroed per call).
struct Counters {
    unsigned long long bin_cnt[kMaxBins];   // pass 1: rows per bin
    unsigned long long cursor[kMaxBins];    // pass 2: fill cursor per bin
    unsigned long long bin_sum[kMaxBins];   // pass 1: sum of the sizes per bin
    unsigned long long bin_nnza[kMaxBins];  // pass 1: A entries of the bin's rows
    unsigned long long bin_own[kMaxBins];   // pass 1: the bin's rows that do not repeat a row before
    unsigned long long rep_cnt[kRepClasses];   // numeric pass 1: repeating rows per class
    unsigned long long rep_found;           // rows of A that look like the row before
    unsigned queued[kMaxBins];              // rows in the numeric kernels' queues
    unsigned long long longest;             // most products of a row of at most kLongMaxNnz entries (0: at
                                            // most kLongLeast)
    unsigned long long max_size;
    unsigned long long total;
    unsigned long long flags;         // bit 0: some row of B has decreasing columns; bit 1: repeated ones
    unsigned long long windows;       // column windows of the large rows (win_count_kernel)
    unsigned long long wcol;          // those of them that accumulate by column
};

// Windowed pass 2 of the numeric bitmap kernel: at most kWinMaxLists A
// entries per row, at most kRunMaxSub column sub-ranges.
constexpr int kWinMaxLists = 1024;
constexpr int kRunMaxSub = 64;
constexpr int kRunDefaultEntries = 12288;

// Kernel table entry (host side).
struct KernelDesc {
    int tpr;          // threads per row (row group)
    int block;        // threads per block
    long long table;  // hash slots per row, or bitmap columns per pass
    long long max_size;  // largest row size the kernel accepts
    int bitmap;       // 1: shared-memory column bitmap kernel
    size_t smem;      // dynamic shared memory per block
};

// Adding a row by column takes one B row per step, so short B rows leave most
// of the warp idle: it is used for rows whose own B rows fill 16 lanes, or 8
// when A has at most kSpanShort entries there, and looked at (the numeric phase
// then reads the ends of a row's B rows first) in bins whose mean lengths say
// so. Numeric phase by the table and by column, 20,000
// rows over 100 columns: B rows of 1 entry and 400 entries of A 151 and 520 us,
// of 4 and 400 299 and 536, of 8 and 50 87 and 84, of 8 and 1,600 1,855 and
// 2,049, of 16 and 50 133 and 84, of 16 and 400 841 and 559.
constexpr int kSpanShort = 128;
inline bool span_rows(double na, int64_t bnnz, int64_t brows) {
    return bnnz > 8 * brows || (bnnz > 4 * brows && na <= kSpanShort);
}

// Rows that a warp-per-row numeric kernel may leave to a block (num_row_limits):
// of at most kLongMaxNnz entries, and of more than kLongLeast products.
constexpr int kLongMaxNnz = 512;
constexpr int kLongLeast = 1024;

// --- setup.cu ----------------------------------------------------------------
// n_prod of every row of the window, added into nprod (zeroed by the caller;
// nullptr: not wanted), and B's column order: bit 0 of cnt->flags set when
// some row of B has a column smaller than the one before it, bit 1 when a
// row repeats a column (cnt nullptr: not wanted). annz: A's entries (sizes
// the grid); grid: blocks of each part, at most. words: rows with their bit
// of fol set are left out (nullptr, or gate shut: none). only_open: no n_prod
// when the gate is shut.
cudaError_t launch_setup(const Operands &op, int64_t annz, int64_t *nprod, int64_t brows, int64_t bnnz,
                         Counters *cnt, int grid, cudaStream_t s, const RepWord *words = nullptr,
                         const RepGate &gate = RepGate(), bool only_open = false);
// n_prod, and the longest and shortest referenced B row, of every row of the
// window (0, 0 and UINT_MAX before); with a gate only when it is shut (n_prod
// may be there already).
cudaError_t launch_feature_scan(const Operands &op, int64_t annz, int64_t *nprod, unsigned *maxlen, unsigned *minlen,
                                int grid, cudaStream_t s, const RepGate &gate = RepGate());
cudaError_t launch_bin_pass1(const int64_t *sizes, int64_t n, const Ranges &rg,
                             const Operands &op, Counters *cnt, long long *tile_sums,
                             cudaStream_t s, const RepArgs &rep = RepArgs());
cudaError_t launch_bin_pass2(const int64_t *sizes, int64_t n, const Ranges &rg,
                             const long long *offsets, Counters *cnt, int32_t *bins,
                             cudaStream_t s, const RepArgs &rep = RepArgs());
// In-place exclusive scan of crpt[0..n) using per-tile sums from pass 1;
// writes crpt[n] = total. tile_sums needs room for ntiles + 1 entries.
cudaError_t launch_scan(int64_t *crpt, int64_t n, long long *tile_sums, cudaStream_t s);
int64_t bin_tile_rows();
cudaError_t launch_iota(int32_t *out, int64_t n, cudaStream_t s);


// --- symbolic.cu / numeric.cu -------------------------------------------------
int sym_kernel_count();
int num_kernel_count();
const KernelDesc &sym_kernel(int id);
const KernelDesc &num_kernel(int id);
cudaError_t sym_prepare(int device_smem_optin);
cudaError_t num_prepare(int device_smem_optin);
// Default symbolic bin ranges and kernels (returns the bin count).
int default_sym_bins(long long *range, int32_t *kernel);
// Kernel attributes of every kernel on device `dev` (the current device),
// once per device; serialised by a lock, so handles and the
// allocation-free entry point may be set up from several host threads.
cudaError_t prepare_device(int dev, int smem_dyn_max);
cudaError_t launch_sym(int id, const Operands &op, const BinWork &w, size_t smem_bitmap,
                       cudaStream_t s);
cudaError_t launch_num(int id, const Operands &op, const BinWork &w, size_t smem_bitmap,
                       cudaStream_t s);
// Which rows of the bin `w` kernel `id` multiplies by a warp each and which by a
// block each: sets the limits and block_rows of w (cnt, lanes, multi and
// by_column set before). na: A entries of the bin's rows, mean_b: entries of B's
// rows, both on average; most: products of any row. True when rows may have to
// change form, so that the launch needs a queue.
bool num_has_warp_form(int id);
bool num_row_limits(int id, const Operands &op, double na, double mean_b, long long most, BinWork &w);
// one-phase numeric kernel `id` (a hash kernel of the numeric table)
cudaError_t launch_num_onephase(int id, const Operands &op, const BinWork &w, cudaStream_t s);

// --- repeat.cu -----------------------------------------------------------------
cudaError_t rep_prepare();
// code[i] of rows first + i, i < n: bit 0 when the row's columns are those
// of the row before moved by one, bit 1 when they are the same (row `first`,
// empty rows and rows of more than kRepMaxNnz entries: 0); their number is
// added to *found (nullptr: not wanted).
cudaError_t launch_row_patterns(const void *rpt, int is64, const int32_t *col, int64_t first, int64_t n,
                                int64_t entries, uint8_t *code, unsigned long long *found, const RepGate &gate,
                                cudaStream_t s);
// fol and one of the window's rows from the codes of A's rows (window rows)
// and of B's rows.
cudaError_t launch_repeats(const Operands &op, int64_t annz, const uint8_t *acode, const uint8_t *bcode,
                           RepWord *words, const RepGate &gate, cudaStream_t s);
// The words complete (words -> out), without the runs of more than max_prod
// products a row; nprod, known for the other rows, filled in for the
// repeating ones.
cudaError_t launch_repeats_finish(int64_t mw, int64_t *nprod, long long max_prod, const RepWord *words, RepWord *out,
                                  cudaStream_t s);
// The repeating rows of class `cls` and of the smaller classes that are not
// launched (C.rpt holds offsets, the rows that they repeat are complete).
// present: bit c set when class c is launched.
cudaError_t launch_repeat_numeric(int cls, int present, const Operands &op, const RepWord *words, const int64_t *crpt,
                                  int32_t *ccol, double *cval, int *err, cudaStream_t s);

// --- runs.cu -------------------------------------------------------------------
// Run boundaries of B rows at column sub-ranges of 2^gshift columns
// (G + 1 int32 per row of B: offset of the first entry of each sub-range).
cudaError_t launch_bsplit(const Operands &op, int64_t brows, int64_t bnnz, int gshift, int G,
                          int32_t *bs, int grid, cudaStream_t s);
// numeric.cu: shared bytes before the bitmap of num_bitmap_kernel (walk
// scratch, or the run metadata of a windowed pass 2).
size_t num_bitmap_head_bytes(bool runs);

// --- window.cu -----------------------------------------------------------------
// Column-window numeric kernel for the rows of the last numeric bin (the
// large rows), used when every row of B is sorted. The column space is cut
// into cells of 2^cs columns (at most kWinMaxCells); the symbolic bitmap
// kernel counts each large row's entries per cell, and a planner cuts the
// row into windows of whole cells that fit one block's shared memory:
//   column window: a dense accumulator indexed by column (8 bytes per
//                  column) plus a presence bitmap; one pass over the products;
//   rank window:   a column bitmap with per-word ranks; one pass marks the
//                  columns, a second adds the values into C.val in L2.
// Rows with at most e1 entries take one rank window over all columns and need
// no cell counts.
constexpr int kWinMaxCells = 256;
constexpr int kWinMinCellLog2 = 12;
constexpr int kWinMaxColsLog2 = 22;
enum : int { kWinRank = 0, kWinCol = 1 };
constexpr long long kWinSingleMax = 16384;   // rows up to this size: one rank window

struct WinPlan {
    int cs = 0, ncells = 0;
    long long ncols = 0;
    long long budget = 0;   // shared bytes of a window's accumulator, bitmap and ranks
    int kc = 0;             // cells of a column window, at most (0: no column windows)
    long long e1 = -1;      // rows with at most e1 entries: one rank window
    long long cut = 0;      // rows of the last numeric bin have more than `cut` entries
};

struct Win {
    int32_t row;            // window row
    int32_t c0, c1;         // columns [c0, c1)
    int32_t mode;           // kWinRank / kWinCol
    uint32_t r0;            // rank of the window's first entry in its row
    uint32_t n;             // entries of the window
};

struct WinWork {
    const Win *win;
    long long nwin;
    unsigned long long *next;      // work counter of the persistent kernel (zeroed)
    const int32_t *bslot;          // B row -> slot of its cell index, or -1
    const int32_t *bidx;           // slot s: (ncells + 1) offsets of the first entry of each cell
    int cs, ncells;
    long long budget;
    // L2 spill of contended accumulations: block b owns spill[b * spill_stride ..),
    // one double per accumulator entry, zero between windows
    double *spill;
    long long spill_stride;
};

long long win_rank_bytes(long long width, long long n);
long long win_col_bytes(long long width);
size_t win_head_bytes();
cudaError_t win_prepare(int smem_optin);
// Window count of each row of the window with more than plan.cut entries
// (crpt holds n_nz), summed into *total.
cudaError_t launch_win_count(const WinPlan &plan, const int64_t *crpt, int64_t mw, const uint16_t *cells,
                             const int32_t *cslot, unsigned long long *total, unsigned long long *total_col,
                             int *err, cudaStream_t s);
// Cell index of the rows of B with at least `min_len` entries (slots up to
// cap). nslot: two counters, 0 before.
cudaError_t launch_win_bindex(const Operands &op, int64_t brows, const WinPlan &plan, long long min_len,
                              int32_t *bslot, int32_t *bidx, long long cap, unsigned long long *nslot,
                              cudaStream_t s);
// Windows of the rows of bin w (crpt holds offsets), appended at *cursor.
cudaError_t launch_win_plan(const WinPlan &plan, const BinWork &w, const uint16_t *cells, const int32_t *cslot,
                            Win *list, long long cap, unsigned long long *cursor, cudaStream_t s);
cudaError_t launch_win_numeric(const Operands &op, const BinWork &w, const WinWork &ww, int grid, size_t smem,
                               cudaStream_t s);

// --- batch.cu ------------------------------------------------------------------
struct BatchProb {
    const void *arpt; int a64; const int32_t *acol; const double *aval;
    const void *brpt; int b64; const int32_t *bcol; const double *bval;
    int64_t M, N;
    int64_t *crpt; int32_t *ccol; double *cval; int64_t ccap;
    int32_t ntiles;
    int32_t dep;        // product whose C is this B, -1 when B is an input
    int32_t tiny;       // 1: every row has at most kBatchTiny products; 0: rows try one thread
                        // per row first (kBatchTiny distinct columns); -1: hash tables only
    int32_t pad;
    long long *tsum;    // per row tile: n_nz sum (symbolic tiles), then its exclusive prefix (scan)
};

constexpr int kBatchTiny = 8;
constexpr int kBatchMaxTile = 1024;   // rows per work item, at most

struct BatchItem {
    int32_t type;       // 0 symbolic tile, 1 scan, 2 numeric tile
    int32_t prob;
    int32_t tile;
    int32_t pad;
};

// Device state, zeroed before every run: queue head, error word and where,
// then per product: symbolic tiles done, scan done, numeric tiles done.
struct BatchState {
    unsigned long long head;
    int err;
    int where;
};

int batch_variant_count();
int batch_variant_table(int v);
int batch_variant_lanes(int v);
int batch_blocks_per_sm(int variant);
cudaError_t launch_batch(int variant, int grid, const BatchProb *probs, const BatchItem *items,
                         int nitems, BatchState *st, int *done_s, int *xflag, int *done_n,
                         int tile_rows, long long spin_limit, cudaStream_t s);

// --- learned.cu ----------------------------------------------------------------
int mlp_param_count();
cudaError_t launch_features(const Operands &op, int64_t annz, int64_t mrows, long long *nprod, unsigned *maxlen,
                            unsigned *minlen, float *X, int grid, cudaStream_t s);
cudaError_t launch_mlp_forward(const float *theta, const float *X, int64_t n, float *y, cudaStream_t s);
cudaError_t launch_mlp_train(const float *theta, const float *X, const float *t, int64_t n,
                             int64_t n_total, float *grad, float *loss, cudaStream_t s);
cudaError_t launch_adam(float *theta, const float *grad, float *m, float *v, int n, int step,
                        float lr, float b1, float b2, float eps, cudaStream_t s);
// sizes[i] = min(pred[i], n_prod[i]), or `huge` when n_prod[i] > exact_above
cudaError_t launch_learned_sizes(const int64_t *nprod, const long long *pred, int64_t n,
                                 long long exact_above, long long huge, int64_t *sizes,
                                 const SizeFactors &sf, uint8_t *cls, unsigned long long *fb,
                                 cudaStream_t s);
// Predicted sizes max(1, ceil(expm1(y) * (1 + margin))), at most cap, of all
// rows, after launch_feature_scan.
cudaError_t launch_predict(const Operands &op, int64_t mrows, const float *theta, const int64_t *nprod,
                           const unsigned *maxlen, const unsigned *minlen, long long *pred, float margin,
                           long long cap, cudaStream_t s);
// The same for the rows that do not repeat a row before (gate as in
// launch_feature_scan), and launch_learned_sizes of all rows (repeating rows
// take n_prod) in one launch.
cudaError_t launch_predict_few(const Operands &op, int64_t mrows, const float *theta, const int64_t *nprod,
                               const unsigned *maxlen, const unsigned *minlen, const RepWord *words,
                               const RepGate &gate, long long exact_above, long long huge, long long *pred,
                               int64_t *sizes, const SizeFactors &sf, uint8_t *cls, unsigned long long *fb,
                               float margin, long long cap, cudaStream_t s);
// copy one-phase rows from temporary memory into C (rows whose pred is -1
// skipped): their columns, their values or both
cudaError_t launch_copy_rows(const BinWork &w, bool cols, bool vals, cudaStream_t s);

}  // namespace ops
