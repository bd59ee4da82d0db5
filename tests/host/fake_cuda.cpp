// A host stand-in for the CUDA runtime and the kernel launches, linked with
// the object of api.cu: device memory is host memory, a launch only notes
// that its stream has work, and launch number `k` fails. Drives one product
// per k and reports memory that is freed, or a call that returns, while a
// side stream has work that the handle's stream does not wait for.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>

#include "internal.h"
#include "opsparse.h"

using namespace ops;

namespace {

constexpr int64_t kRows = 40000;

struct Event {
    cudaStream_t s = nullptr;
    long long at = 0;     // last work of the stream
    long long when = 0;   // when it was recorded
};
std::map<cudaStream_t, long long> work, waited;   // last work of a stream; of it, what the main stream waits for
std::map<cudaEvent_t, Event> events;
long long now_ = 0, handles = 0;
long long launches = 0, fail_at = 0;
bool faults = false;
double mean_entries = 0;   // of a row, in the pattern scans' launches
const cudaStream_t kMain = reinterpret_cast<cudaStream_t>(uintptr_t{1});
const char *where = "";

void check(const char *what) {
    for (const auto &[s, at] : work)
        if (s != kMain && at > waited[s]) {
            std::printf("%s, launch %lld failed: %s while a side stream has work\n", where, fail_at, what);
            faults = true;
            waited[s] = at;   // once
        }
}

cudaError_t launch(cudaStream_t s) {
    if (++launches == fail_at) return cudaErrorLaunchOutOfResources;
    work[s] = ++now_;
    return cudaSuccess;
}

long long allocations = 0, fail_allocation = 0;
size_t live = 0, most = SIZE_MAX;   // bytes handed out, and at most
std::map<void *, size_t> held;
std::map<void *, long long> born;                 // when memory was allocated
std::map<cudaStream_t, long long> started;        // what a side stream waited for, last
long long queued = 0;                             // launches with a row queue
// Memory that a side stream's kernel uses is allocated before that stream starts.
void check_order(const void *p, cudaStream_t s) {
    queued += p != nullptr;
    if (!p || s == kMain) return;
    auto it = born.upper_bound(const_cast<void *>(p));
    if (it != born.begin() && (--it)->second > started[s]) {
        std::printf("%s: a side stream's kernel uses memory that was allocated after the stream started\n", where);
        faults = true;
    }
}
void *take(size_t bytes, void *, void *) {
    if (++allocations == fail_allocation || live + bytes > most) return nullptr;
    void *p = std::calloc(1, bytes);
    live += held[p] = bytes;
    born[p] = ++now_;
    return p;
}
void give(void *p, void *, void *) {
    check("memory is freed");
    live -= held[p];
    held.erase(p);
    born.erase(p);
    std::free(p);
}

const KernelDesc kKernels[] = {{8, 256, 64, 32, 0, 0}, {32, 128, 256, 128, 0, 0}, {1024, 1024, 0, LLONG_MAX, 1, 0}};

}  // namespace

// --- the runtime ---------------------------------------------------------------
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(static_cast<uintptr_t>(100 + ++handles));
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { if (s != kMain) waited[s] = work[s]; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (s != kMain) started[s] = events[e].when;
    if (s == kMain && events[e].s && waited[events[e].s] < events[e].at) waited[events[e].s] = events[e].at;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = reinterpret_cast<cudaEvent_t>(static_cast<uintptr_t>(1000 + ++handles)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { events[e] = Event{s, work[s], ++now_}; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
}

// --- the kernels -----------------------------------------------------------------
namespace ops {
int num_kernel_count() { return 3; }
int sym_kernel_count() { return 3; }
const KernelDesc &num_kernel(int id) { return kKernels[id]; }
const KernelDesc &sym_kernel(int id) { return kKernels[id]; }
cudaError_t num_prepare(int) { return cudaSuccess; }
cudaError_t sym_prepare(int) { return cudaSuccess; }
cudaError_t win_prepare(int) { return cudaSuccess; }
cudaError_t rep_prepare() { return cudaSuccess; }
int64_t bin_tile_rows() { return 4096; }
size_t num_bitmap_head_bytes(bool) { return 1024; }
bool num_has_warp_form(int id) { return id == 1; }
bool num_row_limits(int id, const Operands &, double, double, long long, BinWork &) { return id == 1; }
int mlp_param_count() { return 4673; }
int default_sym_bins(long long *range, int32_t *kernel) {
    const long long r[] = {32, 128, -1};
    for (int j = 0; j < 3; ++j) {
        range[j] = r[j];
        kernel[j] = j;
    }
    return 3;
}
cudaError_t launch_setup(const Operands &, int64_t, int64_t *, int64_t, int64_t, Counters *, int, cudaStream_t s, const RepWord *,
                         const RepGate &, bool) { return launch(s); }
cudaError_t launch_feature_scan(const Operands &, int64_t, int64_t *, unsigned *, unsigned *, int, cudaStream_t s, const RepGate &) { return launch(s); }
// every bin has rows, most of the rows repeat
cudaError_t launch_bin_pass1(const int64_t *, int64_t n, const Ranges &rg, const Operands &, Counters *cnt, long long *tiles, cudaStream_t s,
                             const RepArgs &) {
    for (int j = 0; j < rg.nb; ++j) {
        cnt->bin_cnt[j] = j + 1 < rg.nb ? 8000 : static_cast<unsigned long long>(n - 8000 * (rg.nb - 1));
        cnt->bin_own[j] = static_cast<unsigned long long>(n / 10);
    }
    cnt->rep_cnt[0] = static_cast<unsigned long long>(n - n / 10 * rg.nb);
    cnt->total = 100;
    cnt->longest = 5000;   // some rows may go to a queue
    (void)tiles;
    return launch(s);
}
cudaError_t launch_bin_pass2(const int64_t *, int64_t, const Ranges &, const long long *, Counters *, int32_t *, cudaStream_t s, const RepArgs &) { return launch(s); }
cudaError_t launch_scan(int64_t *, int64_t, long long *, cudaStream_t s) { return launch(s); }
cudaError_t launch_iota(int32_t *, int64_t, cudaStream_t s) { return launch(s); }
cudaError_t launch_sym(int, const Operands &, const BinWork &, size_t, cudaStream_t s) { return launch(s); }
cudaError_t launch_num(int, const Operands &, const BinWork &w, size_t, cudaStream_t s) {
    check_order(w.queue, s);
    return launch(s);
}
cudaError_t launch_num_onephase(int, const Operands &, const BinWork &w, cudaStream_t s) {
    check_order(w.queue, s);
    *w.xcount += 5;   // mispredicted rows
    return launch(s);
}
cudaError_t launch_copy_rows(const BinWork &, bool, bool, cudaStream_t s) { return launch(s); }
cudaError_t launch_predict(const Operands &, int64_t, const float *, const int64_t *, const unsigned *, const unsigned *, long long *, float, long long,
                           cudaStream_t s) { return launch(s); }
cudaError_t launch_predict_few(const Operands &, int64_t, const float *, const int64_t *, const unsigned *, const unsigned *, const RepWord *,
                               const RepGate &, long long, long long, long long *, int64_t *, const SizeFactors &, uint8_t *, unsigned long long *,
                               float, long long, cudaStream_t s) { return launch(s); }
cudaError_t launch_learned_sizes(const int64_t *, const long long *, int64_t, long long, long long, int64_t *, const SizeFactors &, uint8_t *,
                                 unsigned long long *, cudaStream_t s) { return launch(s); }
cudaError_t launch_row_patterns(const void *, int, const int32_t *, int64_t, int64_t n, int64_t entries, uint8_t *, unsigned long long *, const RepGate &,
                                cudaStream_t s) {
    mean_entries = std::max(mean_entries, static_cast<double>(entries) / static_cast<double>(n));
    return launch(s);
}
cudaError_t launch_repeats(const Operands &op, int64_t entries, const uint8_t *, const uint8_t *, RepWord *, const RepGate &, cudaStream_t s) {
    mean_entries = std::max(mean_entries, static_cast<double>(entries) / static_cast<double>(op.mw));
    return launch(s);
}
cudaError_t launch_repeats_finish(int64_t, int64_t *, long long, const RepWord *, RepWord *, cudaStream_t s) { return launch(s); }
cudaError_t launch_repeat_numeric(int, int, const Operands &, const RepWord *, const int64_t *, int32_t *, double *, int *, cudaStream_t s) { return launch(s); }
cudaError_t launch_win_bindex(const Operands &, int64_t, const WinPlan &, long long, int32_t *, int32_t *, long long, unsigned long long *,
                              cudaStream_t s) { return launch(s); }
}  // namespace ops

// One product, launch number `k` failing; false when the product has fewer.
static bool product(int mode, long long k, int64_t row_entries = 16, int64_t rows = kRows, bool same = true, int patterns = 1,
                    int *result = nullptr) {
    work.clear();
    waited.clear();
    events.clear();
    launches = allocations = 0;
    fail_at = k;
    where = mode == SPGEMM_MODE_LEARNED ? "learned" : "plain";
    spgemm_handle *h = nullptr;
    if (spgemm_create(&h, nullptr, take, give, nullptr, kMain) != SPGEMM_OK) std::abort();
    if (mode == SPGEMM_MODE_LEARNED) {
        static float theta[4673];
        const int rc = spgemm_set_predictor(h, theta, 0.f);
        if (rc == SPGEMM_ERR_OOM && result) {
            *result = rc;
            spgemm_destroy(h);
            return true;
        }
        if (rc != SPGEMM_OK || spgemm_set_mode(h, mode) != SPGEMM_OK) std::abort();
    }
    if (!patterns) {   // the read-then-swap probe: every row on its own
        spgemm_config cfg;
        spgemm_get_config(h, &cfg);
        cfg.hash_access = 1;
        if (spgemm_set_config(h, &cfg) != SPGEMM_OK) std::abort();
    }
    static int32_t rpt[kRows + 1], col[1];
    static double val[1];
    spgemm_csr_in A{};
    A.rows = A.cols = kRows;
    A.nnz = row_entries * kRows;
    A.rpt = rpt;
    A.col = col;
    A.val = val;
    static int32_t other[1];
    spgemm_csr_in B = A;
    if (!same) B.col = other;
    spgemm_csr_out C{};
    int64_t nnz = 0;
    int rc = spgemm_symbolic(h, &A, &B, 0, rows, &nnz);
    check("spgemm_symbolic returns");
    if (rc == SPGEMM_OK) {
        rc = spgemm_numeric(h, &A, &B, &C);
        check("spgemm_numeric returns");
    }
    if (rc == SPGEMM_OK && mode == SPGEMM_MODE_PLAIN) {
        rc = spgemm_numeric_values(h, &A, &B, &C);
        check("spgemm_numeric_values returns");
    }
    if (result) *result = rc;
    const bool failed = (k > 0 && launches >= k) || (fail_allocation > 0 && allocations >= fail_allocation && rc == SPGEMM_ERR_OOM);
    if ((rc != SPGEMM_OK) != failed) {
        std::printf("%s, launch %lld failed: result %d\n", where, k, rc);
        faults = true;
    }
    for (void *p : {static_cast<void *>(C.rpt), static_cast<void *>(C.col), static_cast<void *>(C.val)})
        if (p) spgemm_free(h, p);
    spgemm_destroy(h);
    return failed;
}

// A plain product, or a learned one of half the rows, after a learned one, with
// no more memory than that one left: it gets what is kept for the next one.
static void kept_memory(bool back_to_plain) {
    work.clear();
    waited.clear();
    events.clear();
    fail_at = 0;
    where = back_to_plain ? "plain after learned" : "learned after learned";
    static float theta[4673];
    static int32_t rpt[kRows + 1], col[1];
    static double val[1];
    spgemm_handle *h = nullptr;
    spgemm_csr_in A{};
    A.rows = A.cols = kRows;
    A.nnz = 64 * kRows;
    A.rpt = rpt;
    A.col = col;
    A.val = val;
    spgemm_csr_out C{};
    int64_t nnz = 0;
    if (spgemm_create(&h, nullptr, take, give, nullptr, kMain) || spgemm_set_predictor(h, theta, 0.f) ||
        spgemm_set_mode(h, SPGEMM_MODE_LEARNED) || spgemm_multiply(h, &A, &A, &C))
        std::abort();
    for (void *p : {static_cast<void *>(C.rpt), static_cast<void *>(C.col), static_cast<void *>(C.val)}) spgemm_free(h, p);
    const size_t before = live;
    if (back_to_plain) {
        spgemm_set_mode(h, SPGEMM_MODE_PLAIN);
        if (live + 4000 * (32 + 128) * 12 > before) {
            std::printf("%s: temporary rows kept in plain mode\n", where);
            faults = true;
        }
    }
    most = before;
    C = spgemm_csr_out{};
    const int rc = back_to_plain ? spgemm_multiply(h, &A, &A, &C) : spgemm_symbolic(h, &A, &A, 0, kRows / 2, &nnz);
    most = SIZE_MAX;
    if (rc != SPGEMM_OK) {
        std::printf("%s: result %d\n", where, rc);
        faults = true;
    }
    for (void *p : {static_cast<void *>(C.rpt), static_cast<void *>(C.col), static_cast<void *>(C.val)})
        if (p) spgemm_free(h, p);
    spgemm_destroy(h);
    if (live != 0) {
        std::printf("%s: %zu bytes not given back\n", where, live);
        faults = true;
    }
}

int main() {
    for (int mode : {SPGEMM_MODE_PLAIN, SPGEMM_MODE_LEARNED}) {
        long long k = 1;
        queued = 0;
        while (product(mode, k)) ++k;
        std::printf("%s: %lld launches\n", where, k - 1);
        if (queued == 0) {
            std::printf("%s: no row queue\n", where);
            faults = true;
        }
    }
    // a row window: its rows' mean length, not the whole matrix's entries over them
    for (bool same : {true, false}) {
        mean_entries = 0;
        product(SPGEMM_MODE_PLAIN, 0, 64, 5000, same);
        if (mean_entries < 63 || mean_entries > 65) {
            std::printf("pattern scans of a window launched for %.0f entries a row, not 64\n", mean_entries);
            faults = true;
        }
    }
    // an allocation that fails: looking for repeating rows takes memory of its
    // own, without which every row is multiplied on its own
    for (int mode : {SPGEMM_MODE_PLAIN, SPGEMM_MODE_LEARNED}) {
        int refused[2] = {};
        for (int patterns : {0, 1})
            for (fail_allocation = 1;; ++fail_allocation) {
                int rc = SPGEMM_OK;
                product(mode, 0, 16, kRows, true, patterns, &rc);
                if (allocations < fail_allocation) break;
                refused[patterns] += rc != SPGEMM_OK;
            }
        fail_allocation = 0;
        if (refused[0] != refused[1]) {
            std::printf("%s: %d allocations that fail the product, %d without the pattern scans\n", where, refused[1], refused[0]);
            faults = true;
        }
    }
    for (bool back_to_plain : {true, false}) kept_memory(back_to_plain);
    return faults ? 1 : 0;
}
