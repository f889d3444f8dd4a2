// psf_internal.h -- host-side internals shared by the translation units of
// the library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>

#include "../../include/psf.h"
#include "psf_kernels.h"
#include "psf_plan.h"

// ---------------------------------------------------------------- objects
struct psf_series_s {
    std::vector<double> a;
    // PSF_Z_SQUARE: the coefficients c_k of g (f(Z) = g(Z^2) or Z g(Z^2))
    std::vector<double> c;
    bool odd = false;
    double tol = 0.0;
    uint32_t flags = 0;
    int s = 0;
    double e_r = 0.1;
    int maxit = 1000;
    unsigned long long pool_hint = 0;  // user-set initial capacity (entries)
    unsigned long long z_need = 0;     // largest pool the norm phase has needed
    unsigned long long ps_need = 0;    // largest pool the PS phase has needed
    // B-operand mean row lengths seen by the previous evaluation, per step:
    // they pick the thread-group size of the product kernel (tuning only)
    std::vector<double> len_z, len_baby, len_giant;
    // mean output row length before the filter of each giant step (the
    // product kernel's accumulator variant for long rows)
    std::vector<double> out_giant;
    double len_odd = 0.0;  // row length of G-hat in F = Z G-hat (odd series, PSF_Z_SQUARE)
    // widest column window of each step's rows (the bitmap map's wide window
    // is used where it exceeded kBitmapColumns); batches, which may run
    // concurrently on one series, read and write them under span_mu
    std::vector<unsigned> span_z, span_baby, span_giant;
    // most words of 32 columns that one of a step's rows has entries in (the
    // list map is used for wide windows of few words), of the evaluation that
    // recorded the spans; 0 or none: not counted
    std::vector<unsigned> words_z, words_baby, words_giant;
    std::mutex span_mu;
    // steps whose rows k_band mostly left to the accumulator (the filter cuts
    // a band to pieces), on matrices of general_n rows: k_product takes them
    std::vector<char> general_z, general_baby, general_giant;
    int general_n = -1;
    int kernel = 0;       // PSF_PARAM_KERNEL
    int chunk_cols = 0;   // PSF_PARAM_CHUNK_COLS
    int chunk_slots = 0;  // PSF_PARAM_CHUNK_SLOTS
    double dense_xover = -1.0;  // PSF_PARAM_DENSE_XOVER (-1: the process-wide PSF_TUNE_DENSE_XOVER)
    // multiply-adds of each giant step in the previous evaluation (the
    // dense-tile choice of the next one)
    std::vector<double> fma_giant;
};

struct psf_result_s {
    int n = 0;
    long long nnz = 0;
    int* rowptr = nullptr;
    int* col = nullptr;
    double* val = nullptr;
    cudaStream_t stream = nullptr;
    psf_info_t info{};
    std::vector<psf_step_info_t> steps;
    // set when rowptr/col/val point into storage shared by several results
    // (a batch); the storage is released with the last of them
    std::shared_ptr<void> owner;
};

namespace psf {
namespace host {

// Record a failure message for psf_last_error and return `code`.
int fail(int code, const char* fmt, ...);

#define CU(expr)                                                                             \
    do {                                                                                     \
        cudaError_t e_ = (expr);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return fail(e_ == cudaErrorMemoryAllocation ? PSF_ENOMEM : PSF_ECUDA, "%s: %s (%s:%d)", \
                        #expr, cudaGetErrorString(e_), __FILE__, __LINE__);                  \
    } while (0)

// Stream-ordered device buffer released on the stream it was made on.
struct DevBuf {
    void* p = nullptr;
    cudaStream_t st = nullptr;
    DevBuf() = default;
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    ~DevBuf() { release(); }
    cudaError_t alloc(size_t bytes, cudaStream_t s) {
        release();
        st = s;
        if (bytes == 0) bytes = 16;
        const cudaError_t e = cudaMallocAsync(&p, bytes, s);
        if (e != cudaSuccess) p = nullptr;
        return e;
    }
    void release() {
        if (p) cudaFreeAsync(p, st);
        p = nullptr;
    }
    template <class T>
    T* as() const {
        return static_cast<T*>(p);
    }
};

// Optional event timing of the product kernel (psf_profile).
struct Profile {
    bool on = false;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev;
    double fma = 0.0;
};
extern Profile g_prof;

// Largest entry pool: pool positions are 32-bit in the kernels, and loops
// step at most a row (plus a few hundred entries) past a row's end, so the
// capacity stays 2^20 below 2^31 and no position plus offset overflows.
constexpr unsigned long long kMaxPool = (1ull << 31) - (1ull << 20);

// Mailboxes: pinned host buffers mapped into the device's address space,
// {host, device} pointers, into which k_export writes the control block, the
// norm slots and the step records that the host reads back.  A kernel's stores take no copy engine, so these
// reads do not wait behind a large device-to-host copy in flight on another
// stream (a user copying one result out while the next evaluation runs).
// Each evaluation's workspace takes one from a process-wide free list and
// gives it back; they are kept for the life of the process (which must not
// outlive a cudaDeviceReset).  {nullptr, nullptr} if none could be made: the
// read-backs then use copies.
constexpr size_t kMboxBytes = 64 * 1024;
// The front of a workspace's zeroed block, read back as one piece: control
// block, norm slots, step records (those of a longer plan have a buffer of
// their own).
constexpr size_t kFrontSlots = 256, kFrontStats = 512;
constexpr int kFrontRecords = 96;  // the norm phase's first 16, then the PS phase's
constexpr size_t kFrontBytes = (kFrontStats + sizeof(StepStat) * kFrontRecords + 255) & ~(size_t)255;
static_assert(sizeof(Ctl) % 4 == 0 && sizeof(Ctl) <= kFrontSlots, "control block in its part");
static_assert(kFrontSlots + sizeof(NormSlot) * kMaxNorms <= kFrontStats, "norm slots in their part");
static_assert(kFrontBytes <= kMboxBytes / 2, "the front fits a mailbox");
std::pair<void*, void*> mailbox_take();
void mailbox_give(std::pair<void*, void*> m);

// Device workspace shared by the phases of one evaluation.
// products mark their output pattern from column bitmaps of B's rows
// (PSF_TUNE_ROW_BITMAPS: 0 never, 1 when A's rows average at least
// kBitmapMinA entries and B's kBitmapMinB, 2 always)
extern std::atomic<int> g_row_bitmaps;
constexpr double kBitmapMinA = 12.0;
constexpr double kBitmapMinB = 32.0;

// A matrix's row arrays: descriptors, first and end entries.
struct Rows {
    int* rb = nullptr;
    int* re = nullptr;
    RowDesc* rd = nullptr;
};

struct Work {
    int n = 0;
    cudaStream_t st = nullptr;
    // one block, zeroed with one memset: the front (control block, norm slots,
    // step records), the column sums of Algorithm 1 (and their sticky counts,
    // and the norms'), and the norm phase's 24-bit-piece column sums (zero
    // between uses)
    DevBuf slab, pool_col, pool_val, cand_col, cand_x, scan, more_stats;
    unsigned long long* words = nullptr;
    unsigned* sticky = nullptr;
    unsigned long long* nwords = nullptr;
    size_t sums_bytes = 0;  // words and sticky
    DevBuf dense[3];  // the dense-tile path's A, B and C (n^2 doubles each), allocated on first use
    DevBuf bhdr, pool_bits;  // column bitmaps of a product's B rows: n headers, a word per pool entry
    DevBuf pool_lists;       // the list map's form: a pair per pool entry, allocated on first use
    unsigned long long lists_cap = 0;
    bool no_lists = false;   // there was no memory for them in this call
    int bandwidth = 0;       // of the checked inputs
    double dense_xover = 1e300;  // dense tiles for a step with at least this many multiply-adds per n^3
    bool dense_estimate = false;  // a step without a recorded count may use the row-length estimate
    unsigned long long cap = 0, ccap = 0, bits_cap = 0;
    static constexpr size_t kRowsChunk = 8;  // matrices' row arrays allocated at a time
    std::vector<DevBuf*> rows;  // per matrix: n row descriptors, then rb and re (n ints each)
    bool band = false;           // input rows are runs of columns whose products are runs: k_band computes them
    int slot_map = 0;            // 0 auto (by products per row), 1 table, 2 bitmap, 3 wide window, 4 CTA per row
    int chunk_cols = 0, chunk_slots = 0;

    std::pair<void*, void*> mbox{nullptr, nullptr};
    bool mbox_pending = false;  // an export into the mailbox may still be in flight
    ~Work() {
        for (DevBuf* b : rows) delete b;
        if (mbox.first) {
            // (an error path can leave an export unsynchronised: let it land
            // before another evaluation takes the mailbox)
            if (mbox_pending) cudaStreamSynchronize(st);
            mailbox_give(mbox);
        }
    }
    char* front() const { return slab.as<char>(); }
    Ctl* C() const { return slab.as<Ctl>(); }
    NormSlot* slots() const { return reinterpret_cast<NormSlot*>(front() + kFrontSlots); }
    StepStat* front_stats() const { return reinterpret_cast<StepStat*>(front() + kFrontStats); }
    // norms: matrices whose exact norms are taken by row tiles
    int init(int n_, cudaStream_t s, int norms) {
        n = n_;
        st = s;
        if (!mbox.first) mbox = mailbox_take();
        const size_t nn = (size_t)(n > 0 ? n : 1);
        const size_t b_words = sizeof(unsigned long long) * kChunks * nn;
        const size_t b_sticky = (sizeof(unsigned) * nn * (size_t)(norms > 1 ? norms : 1) + 7) & ~(size_t)7;
        const size_t bytes = kFrontBytes + b_words + b_sticky +
                             sizeof(unsigned long long) * (size_t)kNormPieces * nn * (size_t)norms;
        CU(slab.alloc(bytes, st));
        words = reinterpret_cast<unsigned long long*>(front() + kFrontBytes);
        sticky = reinterpret_cast<unsigned*>(front() + kFrontBytes + b_words);
        nwords = reinterpret_cast<unsigned long long*>(front() + kFrontBytes + b_words + b_sticky);
        sums_bytes = b_words + b_sticky;
        CU(cudaMemsetAsync(slab.p, 0, bytes, st));
        return PSF_OK;
    }
    // scratch of the products' launches
    int init_products() {
        CU(scan.alloc(sizeof(long long) * scan_scratch_len(n), st));
        CU(bhdr.alloc(sizeof(int2) * (size_t)(n > 0 ? n : 1), st));
        return PSF_OK;
    }
    // `count` zeroed step records (not the norm phase's first 16); again: they
    // were used before
    int stats_for(int count, bool again, StepStat** out) {
        if (count <= kFrontRecords - 16) {
            *out = front_stats() + 16;
            if (!again) return PSF_OK;
        } else {
            if (!again) CU(take(more_stats, sizeof(StepStat) * (size_t)count));
            *out = more_stats.as<StepStat>();
        }
        CU(cudaMemsetAsync(*out, 0, sizeof(StepStat) * (size_t)count, st));
        return PSF_OK;
    }
    // (re)allocate the entry pool and reset the device control block
    int reset_pool(unsigned long long entries) {
        if (entries > kMaxPool) return fail(PSF_ETOOBIG, "pool of %llu entries exceeds 2^31 - 2^20", entries);
        if (entries > cap) {
            CU(take(pool_col, sizeof(int) * entries));
            CU(take(pool_val, sizeof(double) * entries));
            cap = entries;
            // two Algorithm 1 candidate lists of half the pool each (a step
            // whose candidates do not fit falls back to full scans)
            ccap = cap / 2 > 1024 ? cap / 2 : 1024;
            CU(take(cand_col, sizeof(int) * 2 * ccap));
            CU(take(cand_x, sizeof(unsigned long long) * 2 * ccap));
        }
        if (g_row_bitmaps.load() > 0 && bits_cap < cap) {
            CU(take(pool_bits, sizeof(unsigned) * cap));
            bits_cap = cap;
        }
        CU(launch_reset(C(), cap, ccap, cand_chunk(), st));
        return PSF_OK;
    }
    // the lists' memory; null where there is none left (the step then takes the
    // wide bitmap window, which needs none).  It is a convenience: whatever
    // else the call allocates later may have it (take), a larger pool and the
    // result among them.
    uint2* lists() {
        if (lists_cap < cap && !no_lists) {
            lists_cap = 0;
            if (pool_lists.alloc(sizeof(uint2) * cap, st) == cudaSuccess) {
                lists_cap = cap;
            } else {
                cudaGetLastError();
                no_lists = true;
            }
        }
        return lists_cap >= cap ? pool_lists.as<uint2>() : nullptr;
    }
    // bytes of device memory, the lists' if there is no other
    cudaError_t take(void** p, size_t bytes) {
        cudaError_t e = cudaMallocAsync(p, bytes, st);
        if (e == cudaErrorMemoryAllocation && pool_lists.p) {
            cudaGetLastError();
            pool_lists.release();
            lists_cap = 0;
            no_lists = true;
            e = cudaMallocAsync(p, bytes, st);
        }
        if (e != cudaSuccess) *p = nullptr;
        return e;
    }
    cudaError_t take(DevBuf& b, size_t bytes) {
        b.release();
        b.st = st;
        return take(&b.p, bytes > 0 ? bytes : 16);
    }
    // Entries a warp reserves in a candidate list at a time: up to 128, so
    // that about 12k warps' unused chunk ends take at most a quarter of it.
    unsigned cand_chunk() const {
        unsigned long long c = ccap / (4ull * 12288ull);
        c = c < 32ull ? 32ull : (c > 128ull ? 128ull : c);
        return (unsigned)(c & ~31ull);
    }
    // Column-sum accumulators are zero between steps; a phase cut short by a
    // pool overflow can leave some set, so they are cleared before its retry.
    int clear_sums() {
        CU(cudaMemsetAsync(words, 0, sums_bytes, st));
        return PSF_OK;
    }
    // row arrays of matrix slot i
    int rows_for(size_t i, Rows* out) {
        const size_t c = i / kRowsChunk, nn = ((size_t)(n > 0 ? n : 1) + 3) & ~(size_t)3;
        while (rows.size() <= c) rows.push_back(new DevBuf());
        const size_t each = (sizeof(RowDesc) + 2 * sizeof(int)) * nn;
        if (!rows[c]->p) CU(take(*rows[c], each * kRowsChunk));
        out->rd = reinterpret_cast<RowDesc*>(rows[c]->as<char>() + each * (i % kRowsChunk));
        out->rb = reinterpret_cast<int*>(out->rd + nn);
        out->re = out->rb + nn;
        return PSF_OK;
    }
    RowView pooled(const Rows& r) const { return RowView{r.rb, r.re, pool_col.as<int>(), pool_val.as<double>(), r.rd}; }
    int* pcol() const { return pool_col.as<int>(); }
    double* pval() const { return pool_val.as<double>(); }
};

// Process-wide tuning (psf_tune_*, psf_autotune): the products per output
// row from which the product kernel uses the column-table slot map.
extern std::atomic<double> g_table_crossover;
// the PS phase of a batch runs as one captured CUDA graph (PSF_TUNE_BATCH_GRAPH)
extern std::atomic<bool> g_batch_graph;
// batched baby steps copy the norm phase's powers while nothing was dropped (PSF_TUNE_BATCH_REUSE)
extern std::atomic<bool> g_batch_reuse;
// Algorithm 1 sets candidates at or below eps_g / 2^g_far_shift apart (PSF_TUNE_ALG1_FAR_SHIFT)
extern std::atomic<int> g_far_shift;
// fault injection: the k-th server admission from now fails (PSF_TUNE_FAIL_ADMISSION)
extern std::atomic<long long> g_fail_admission;
// the dense-tile crossover in multiply-adds per n^3 (PSF_TUNE_DENSE_XOVER)
constexpr double kDenseXoverDefault = 0.15;
constexpr int kDenseMinN = 512;  // the automatic choice leaves smaller products sparse
extern std::atomic<double> g_dense_xover;
// slot_map 1: table, 2: bitmap, 0: by the work per row and the crossover
inline bool use_table(int slot_map, double work_per_row) {
    return slot_map == 1 || (slot_map == 0 && work_per_row >= g_table_crossover.load(std::memory_order_relaxed));
}

// One output row per block of four warps (k_product_cta) for a product of
// the single-matrix path when its rows fit one wave of blocks (7 per SM), so
// that warps would otherwise sit idle, and its B rows average at least 16
// entries (they are shared by the block's 128 threads); PSF_PARAM_KERNEL 4
// forces it.  Measured on GB300: the banded N(0, 1) family at n = 1000 runs
// 1.3-1.6x faster from bandwidth 8 on; at n = 4096 and above the warp per row
// is faster (1.4-2.7x).
inline bool use_cta(int n, double alen, double blen) {
    (void)alen;
    return n > 0 && n <= 7 * num_sms() && blen >= 16.0;
}

// k_band against k_product: more than one row in kGeneralShare that it would
// leave to the accumulator (its narrow map, three or more warps of a shared
// tile waiting) and k_product, with its windows, row bitmaps and the row per
// block, takes the step
constexpr unsigned kGeneralShare = 8;
inline bool mostly_runs(unsigned long long general, int n) { return general * kGeneralShare <= (unsigned long long)n; }

// A step's column window: the bitmap map's own, its wide one, or the list map
// (wide, and its rows have entries in few words).  span, words: the widest
// row's columns and the most words of a row, in the previous evaluation or as
// far as this one can tell (words 0: unknown).  The line lies at the narrow
// window's edge because the two are level there: on a 512 x 512 grid (tol
// 1e-12) a product of rows spanning 4097 columns takes 740 us in the narrow
// window, and one of 5121 takes 846 with the list map and 1155 in the wide
// window; then 6145: 900 / 1303, 10241: 1519 / 2277, and the giant steps
// S_1..S_5 4.1 / 3.9, 5.7 / 9.0, 8.0 / 12.5, 11.3 / 17.4, 16.1 / 37.8 ms (the
// last ones exceed the wide window's 16384 columns).
enum Window { kNarrow = 0, kWide = 1, kLists = 2 };
inline int window_for(double span, double words) {
    if (!(span > kBitmapColumns)) return kNarrow;
    return words > 0.0 && words <= kListMapWords ? kLists : kWide;
}

// A row may keep holes (stored zeros: k_band, filter_row) where no operand of
// a product can have overflowed: the fold takes a hole as an entry, and
// 0 * inf would put a NaN where an entry that is not there gives nothing.
// By the norms' bounds (Plan::bound), with room for norms that are estimates
// (their error grows with the power: 2^323 to the largest double).  Past it a
// plan's thresholds are 0 wherever an operand is infinite, so the filter
// leaves no holes either.
constexpr double kHoleBound = 0x1p700;

// Recorder of product launches for psf_autotune (set on the calling thread
// only): each launch's work per row and its event pair.
struct TuneRecorder {
    std::vector<double> work;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev;
};
extern thread_local TuneRecorder* g_tune_rec;

int lsb_for_bound_host(double x);
RowView view_of(const psf_csr_t& m);
int check_csr(const psf_csr_t* m, int n, const char* what);
int read_back(Work& w, Ctl& c, NormSlot* slots = nullptr, StepStat* stats = nullptr,
              const StepStat* dev_stats = nullptr, size_t count = 0);
int status_to_code(int st);
unsigned long long arena_for(double row_len);
void destroy_result(psf_result_s* r);
int prepare(cudaStream_t st);
// Estimates of ||Z^k||_1, k = 2..10, into norms[2..10] (psf_normest.cu);
// *fallback: a column of Z is too long for the estimator, nothing computed.
int estimate_power_norms(Work& w, const psf_csr_t& Z, double* norms, bool* fallback);

}  // namespace host
}  // namespace psf
