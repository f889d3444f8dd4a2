// psf_kernels.cu -- CUDA kernels of the filtered Paterson-Stockmeyer
// evaluator (sm_103a, FP64 throughout).
//
//  k_product      one fused step C = sum_t alpha_t M_t + A B: output pattern
//                 and slot map of each row, exact row reservation in the
//                 pool, FP64 accumulation in shared memory, write-back of the
//                 nonzero entries, and the first pass of Algorithm 1 (exact
//                 column sums and the candidate list of the entries
//                 |x| <= eps_g); a batch instantiation reads per-row
//                 instance parameters.
//  k_product_cta  the same step with one output row per block of four warps
//                 (matrices of at most one wave of rows with long B rows).
//  k_band         the same step where rows span consecutive columns: outputs
//                 folded in registers.
//  k_row_bitmaps  column bitmaps of B's rows for the symbolic pass.
//  k_row_lists    the same as lists of the words in use, for the list map.
//  k_reuse_pass1  a baby step equal to a power of the norm phase: the first
//                 pass of Algorithm 1 on that power's rows.
//  k_reuse_copy_batch  the same for the instances of a batch: those rows
//                 copied into the step's pool range, with that first pass.
//  k_alg1         the remaining passes of Algorithm 1 (Sec. 3.1.1) and the
//  k_alg1_batch   final in-place compaction, one cooperative launch (single
//                 instance, or every filtered instance of a batched step).
//  k_norms_rows   exact 1-norms of Z^1..Z^10 (Eq. 37's z_i) by row tiles,
//  k_norms_finish column sums in shared memory; rounding and maxima.
//  k_norms        exact 1-norms from flat pool ranges (psf_norm1 and its
//                 allocation-free variant).
//  k_export       small device records written into pinned, device-mapped
//                 host memory (the host's read-backs take no copy engine).
//  k_copy_result  a result's arrays into the caller's.
//  k_absmax, k_validate*, k_copy_rows*, k_scan_*, k_gather*, k_identity,
//  k_inst_table, k_compose_rows, k_bounds: plumbing.
#include <atomic>
#include <climits>
#include <mutex>
#include <utility>

#include "psf_device.cuh"
#include "psf_kernels.h"

namespace psf {

// Programmatic launches.  The kernels of a call follow one another on a stream,
// and most of a small call is the time between them: a kernel's blocks are
// scheduled only when the last one has drained.  Launched programmatically
// (launch_pdl) a kernel is brought onto the SMs while the one before it runs;
// it starts by waiting for that one's end (all of its blocks, and what they
// wrote) and then lets the next one come.  Every kernel here does so first of
// all, so that whatever ran two launches earlier has ended too, with one
// exception: k_band in a batch's paired step lets the next one come at once and
// waits in its last lines.  It may read what earlier steps wrote because the
// launch just before it is its own step's k_product, launched ordinarily (all
// before that has ended when it starts), whose blocks have all started when
// k_band does.  Neither may be changed without the other.  A launch that is no
// such kernel's neighbour behaves as an ordinary one.  Pointers to what a
// predecessor writes carry no __restrict__: the compiler may not take the data
// for constant.
// Measured on whole calls (us, ordinary / programmatic): norm1 of a 37 x 29 grid
// 46.5 / 38.3, one banded product of 30001 rows 259 / 246, exp of the 1D
// Laplacian, n = 256, 511 / 430, cos of banded N(0, 1), n = 1000, 1084 / 1014,
// banded n = 65536 3843 / 3778.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
    pdl_wait();
    pdl_release();
}
template <class... Params, class... Args>
static cudaError_t launch_pdl(void (*k)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------- k_product
// Compact-accumulator kernel: one warp computes one output row, with no
// block-level synchronisation.  The row's output pattern is found first (the
// symbolic pass), each output column gets an accumulator slot (its rank in
// the pattern), then the products are folded in (the numeric pass).  Two
// ways to map a column offset o = c - c0 to its slot, a template parameter:
//
//  table  (TAB = true)   tab[o] (16 bit) holds first a flag, set by plain
//         stores of every contributing entry, then the slot, after a ballot
//         scan.  O(window) set-up per row, one load per lookup: for rows with
//         many products per column of the window.
//  bitmap (TAB = false)  pm[o / 32] holds a 32-column bitmap word, set by
//         atomic ORs (one per run of columns a lane meets), and the number of
//         set bits before it; slot = prefix + popcount of the lower bits.
//         O(window / 32) set-up per row: for thin rows.
//
// Numeric pass: the addends in order, then the B rows in ascending k, each
// entry folded as acc[slot] = fma(a, b, acc[slot]); a warp barrier separates
// consecutive rows (the fixed rounding order of the product).  B rows are
// read in 128-entry chunks (four 32-entry pieces; the entries of a chunk
// have distinct columns, so its four read-modify-writes are independent).
// A row whose pattern exceeds the chunk (wider than the map or with more
// than kAccCap entries) is processed in several column chunks.
constexpr int kTabCap = 4160;  // columns of the table map
constexpr int kBmWords = 144;  // bitmap words of the bitmap map (4608 columns)
constexpr int kBmBits = kBmWords * 32;
// The wide-window bitmap (16384 columns) for steps whose rows span more
// columns than kBmBits (a grid of side M spreads a row over about 2rM
// columns for a pattern of radius r): one column chunk instead of several,
// at 5 blocks per SM instead of 7.
constexpr int kBmWordsBig = 512;
static_assert(kBmBits == kBitmapColumns, "the host's notion of the bitmap window");
// The list map, for rows that span yet more columns but have entries in few
// of their 32-column words (on a grid of side M a row of radius r has 2r + 1
// runs of at most 2r + 1 columns, M apart): a byte per word of a 32768-column
// window says which of up to kListIds words in use it is; prefix and bitmap
// are kept for those alone.  B rows come as lists of their words, so marking
// one costs its words, not its columns, and the map of a row with more
// entries than slots serves all its column chunks.  Bound by instructions
// issued (the last giant step of exp on a 512 x 512 grid: 6.6 G warp
// instructions at 40 % of the issue slots, FP64 pipe 53 %); 160 ids leave six
// blocks an SM their shared memory (192: five).  That step took
// 37.8 ms with 16384-column bitmaps and takes 16.1; the evaluation 104 -> 64.
constexpr int kListWords = 1024;
constexpr int kListIds = kListMapWords;
constexpr unsigned kNoId = 0xffu;
static_assert(kListIds < (int)kNoId, "an id fits a byte");
// Accumulator slots; with 7 bitmap blocks of 4 warps per SM shared memory is
// full.  The bitmap map keeps a segment's a_rk in the last 32 slots, so a row
// has kAccCap - 32 of them; its WIDE instantiation, for steps whose rows are
// long, reads a_rk from A's row instead and gives a row every slot (a row of
// up to kAccCap entries then takes one pass, not two column chunks).
constexpr int kAccCap = 640;

template <bool TAB, int W = kBmWords>
struct ProdSmem;

template <>
struct ProdSmem<true, kBmWords> {
    static constexpr int kCols = kTabCap;
    static constexpr int kWarps = 2;
    static constexpr int kBlocksPerSm = 7;
    unsigned short tab[kTabCap];
    double acc[kAccCap];
    double ka[32];
    int kb[32];
    int kl[32];
    unsigned short colbuf[kAccCap];
};

template <int W>
struct ProdSmem<false, W> {
    static constexpr int kCols = W * 32;
    static constexpr int kWarps = 4;
    // 28 warps: registers (72) and shared memory; 20 with the wide window
    static constexpr int kBlocksPerSm = W > kBmWords ? 5 : 7;
    uint2 pm[W];  // .x = set bits before the word, .y = bitmap word
    double acc[kAccCap];  // the last 32 hold a_rk of the segment (not in WIDE)
    int kb[32];
    int kl[32];
    unsigned short colbuf[kAccCap];
};

template <>
struct ProdSmem<false, kListWords> {
    static constexpr int kCols = kListWords * 32;
    static constexpr int kWarps = 4;
    static constexpr int kBlocksPerSm = 6;
    uint2 pm[kListIds];  // by id: set bits before the word, bitmap
    double acc[kAccCap];
    int kb[32];
    int kl[32];
    unsigned short colbuf[kAccCap];
    unsigned short word[kListIds];  // id -> window word
    unsigned char id[kListWords];   // window word -> id (kNoId: no entry)
};

template <bool TAB, int W = kBmWords>
size_t prod_smem_bytes() {
    return sizeof(ProdSmem<TAB, W>) * ProdSmem<TAB, W>::kWarps + sizeof(AddTerm) * kMaxAdd;
}

// first position in [s, e) with col >= c (col ascending).  Pool positions
// reach 2^31 - 2^20, so the midpoint is s + (e - s) / 2: s + e would overflow.
__device__ __forceinline__ int lower_bound_col(const int* col, int s, int e, int c) {
    while (s < e) {
        const int mid = s + ((e - s) >> 1);
        if (col[mid] < c) s = mid + 1;
        else e = mid;
    }
    return s;
}

// slot of column offset o (o inside the current chunk's pattern)
__device__ __forceinline__ int slot_lookup(const ProdSmem<true>& S, int o) { return S.tab[o]; }
// (o's own bit is set: the set bits at or below it, shifted to the top,
// count one more than the bits below it)
template <int W>
__device__ __forceinline__ int slot_lookup(const ProdSmem<false, W>& S, int o) {
    const uint2 e = S.pm[o >> 5];
    return (int)e.x + __popc(e.y << (~o & 31)) - 1;
}

__device__ __forceinline__ int slot_lookup(const ProdSmem<false, kListWords>& S, int o) {
    const uint2 e = S.pm[S.id[o >> 5]];
    return (int)e.x + __popc(e.y << (~o & 31)) - 1;
}

// where a segment's a_rk are kept
__device__ __forceinline__ double* ka_of(ProdSmem<true>& S) { return S.ka; }
template <int W>
__device__ __forceinline__ double* ka_of(ProdSmem<false, W>& S) { return S.acc + (kAccCap - 32); }

// Load the segment [seg, seg + cnt) of A's row: a_rk (unless `store_a` is
// false) and the range of B's row k restricted to columns [c0, c1) (the
// whole row when `whole`).
template <bool TAB, int W>
__device__ __forceinline__ void load_segment(const ProductArgs& P, int seg, int cnt, bool whole, int c0, int c1,
                                             int lane, ProdSmem<TAB, W>& S, bool store_a, bool a_holes,
                                             unsigned long long* fma = nullptr, int* kwn = nullptr) {
    if (lane < cnt) {
        int k = P.A.col[seg + lane];
        const RowDesc d = P.B.rd[k];
        int b = d.rb, e = d.re;
        if (fma && !(a_holes && P.A.val[seg + lane] == 0.0)) *fma += (unsigned long long)rd_nnz(d);
        if (kwn) {
            // B row k's bitmap: its first word's offset in the window (c0 is a
            // multiple of 32 and the window holds the whole row) and its words
            const int2 h = P.bhdr[k];
            kwn[lane] = h.y > 0 ? ((h.x - (c0 >> 5)) << 16) | h.y : 0;
        }
        if (!whole) {
            int b2 = lower_bound_col(P.B.col, b, e, c0);
            e = lower_bound_col(P.B.col, b2, e, c1);
            b = b2;
        }
        if (store_a) ka_of(S)[lane] = P.A.val[seg + lane];
        S.kb[lane] = b;
        S.kl[lane] = e - b;
    }
    __syncwarp();
}

// ---- symbolic pass, table map: plain flag stores, four pieces per step
__device__ __forceinline__ void mark_row(const int* col, int s, int e, int c0, int cend, int lane,
                                         ProdSmem<true>& S) {
    for (int q0 = s; q0 < e; q0 += 128) {
        int cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u * 32 + lane;
            cs[u] = q < e ? col[q] : INT_MIN;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (cs[u] >= c0 && cs[u] < cend) S.tab[cs[u] - c0] = 1;
    }
}
__device__ __forceinline__ void mark_one(int o, ProdSmem<true>& S) { S.tab[o] = 1; }
__device__ __forceinline__ void clear_map(int wlen, int lane, ProdSmem<true>& S) {
    uint4* t4 = reinterpret_cast<uint4*>(S.tab);
    const int n16 = (wlen + 7) >> 3;
    for (int i = lane; i < n16; i += 32) t4[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ---- symbolic pass, bitmap map: lane l walks a contiguous slice of the row
// and ORs whole runs of columns into a bitmap word at a time.  CHK: test
// each column against [c0, cend); a B row needs no test, since
// load_segment has already clipped it to that range (or, for a row that
// takes one chunk, the range spans every B column of the row).
template <bool CHK, int W>
__device__ __forceinline__ void mark_row(const int* col, int s, int e, int c0, int cend, int lane,
                                         ProdSmem<false, W>& S) {
    const int m = (e - s + 31) >> 5;
    const int q0 = s + lane * m, q1 = min(e, q0 + m);
    unsigned curw = 0xffffffffu, mask = 0u;
    for (int q = q0; q < q1; q += 4) {
        int cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cs[u] = q + u < q1 ? col[q + u] : INT_MIN;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int c = cs[u];
            if (CHK ? (c < c0 || c >= cend) : (q + u >= q1)) continue;
            unsigned off = (unsigned)(c - c0), w = off >> 5;
            if (w != curw) {
                if (mask) atomicOr(&S.pm[curw].y, mask);
                curw = w;
                mask = 0u;
            }
            mask |= 1u << (off & 31);
        }
    }
    if (mask) atomicOr(&S.pm[curw].y, mask);
}
// Two B rows at once, each as mark_row<false> marks it (lane l walks its
// contiguous slice of each row): the column loads of both rows are issued
// before either row's columns are ORed in, so the second row's loads do not
// wait for the first row's marking.  The rows are clipped to the window.
template <int W>
__device__ __forceinline__ void mark_row_pair(const int* col, int sa, int ea, int sb, int eb, int c0,
                                              int lane, ProdSmem<false, W>& S) {
    const int ma = (ea - sa + 31) >> 5, mb = (eb - sb + 31) >> 5;
    int qa = sa + lane * ma, qb = sb + lane * mb;
    const int qa1 = min(ea, qa + ma), qb1 = min(eb, qb + mb);
    unsigned wa = 0xffffffffu, ka = 0u, wb = 0xffffffffu, kb = 0u;
    while (qa < qa1 || qb < qb1) {
        int cs[2][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            cs[0][u] = qa + u < qa1 ? col[qa + u] : 0;
            cs[1][u] = qb + u < qb1 ? col[qb + u] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (qa + u >= qa1) continue;
            const unsigned off = (unsigned)(cs[0][u] - c0), w = off >> 5;
            if (w != wa) {
                if (ka) atomicOr(&S.pm[wa].y, ka);
                wa = w;
                ka = 0u;
            }
            ka |= 1u << (off & 31);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (qb + u >= qb1) continue;
            const unsigned off = (unsigned)(cs[1][u] - c0), w = off >> 5;
            if (w != wb) {
                if (kb) atomicOr(&S.pm[wb].y, kb);
                wb = w;
                kb = 0u;
            }
            kb |= 1u << (off & 31);
        }
        qa += 4;
        qb += 4;
    }
    if (ka) atomicOr(&S.pm[wa].y, ka);
    if (kb) atomicOr(&S.pm[wb].y, kb);
}
// Short B rows (at most 32 entries each): lane i marks the segment's B row i,
// so the rows' column loads are in flight together instead of one row after
// the other.  The rows are clipped to [c0, cend) (see mark_row).
template <int W>
__device__ __forceinline__ void mark_rows_short(const int* col, int cnt, int c0, int cend, int lane,
                                                ProdSmem<false, W>& S, bool active = true) {
    if (lane >= cnt || !active) return;
    const int s = S.kb[lane], e = s + S.kl[lane];
    unsigned curw = 0xffffffffu, mask = 0u;
#pragma unroll 2
    for (int q = s; q < e; q += 4) {
        int cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cs[u] = q + u < e ? col[q + u] : INT_MIN;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = cs[u];
            if (q + u >= e) continue;
            const unsigned off = (unsigned)(c - c0), w = off >> 5;
            if (w != curw) {
                if (mask) atomicOr(&S.pm[curw].y, mask);
                curw = w;
                mask = 0u;
            }
            mask |= 1u << (off & 31);
        }
    }
    if (mask) atomicOr(&S.pm[curw].y, mask);
}
template <int W>
__device__ __forceinline__ void mark_one(int o, ProdSmem<false, W>& S) { atomicOr(&S.pm[o >> 5].y, 1u << (o & 31)); }
template <int W>
__device__ __forceinline__ void clear_map(int wlen, int lane, ProdSmem<false, W>& S) {
    const int nw = (wlen + 31) >> 5;
    for (int w = lane; w < nw; w += 32) S.pm[w].y = 0u;
}

// The B rows of A's row [pa0, pa1) into the bitmap, for a row that takes one
// chunk whose first column c0 is a multiple of 32: a B row with a bitmap
// (bhdr) is ORed in a word at a time, lane l collecting the window words
// l, l + 32, ... in registers (coalesced loads, no shared-memory traffic
// until the end); the others are marked column by column as in build_map.
template <int W>
__device__ __forceinline__ void mark_from_bitmaps(const ProductArgs& P, int pa0, int pa1, int c0, int cend, int lane,
                                                  ProdSmem<false, W>& S, bool store_a, bool a_holes,
                                                  unsigned long long* fma) {
    constexpr int R = (W + 31) / 32;
    unsigned reg[R];
#pragma unroll
    for (int u = 0; u < R; ++u) reg[u] = 0u;
    int* kwn = reinterpret_cast<int*>(S.colbuf);  // free until the slots are assigned
    const unsigned* bits = P.bbits;
    for (int seg = pa0; seg < pa1; seg += 32) {
        const int cnt = min(32, pa1 - seg);
        load_segment<false>(P, seg, cnt, true, c0, cend, lane, S, store_a, a_holes, fma, kwn);
        // rows without a bitmap: short ones one per lane, long ones by the warp
        const int my = lane < cnt && kwn[lane] == 0 ? S.kl[lane] : 0;
        mark_rows_short(P.B.col, cnt, c0, cend, lane, S, my > 0 && my <= 32);
        unsigned longm = __ballot_sync(kFull, my > 32);
        while (longm) {
            const int i = __ffs(longm) - 1;
            longm &= longm - 1u;
            mark_row<false>(P.B.col, S.kb[i], S.kb[i] + S.kl[i], c0, cend, lane, S);
        }
        // U B rows at a time (4; 2 for the wide window's 16 words per lane):
        // their words are loaded before any is ORed in, so the loads of
        // consecutive rows are in flight together
        constexpr int U = R <= 5 ? 4 : 2;
        for (int i = 0; i < cnt; i += U) {
            unsigned t[U][R];
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int h = i + j < cnt ? kwn[i + j] : 0;
                const int kw = h >> 16, kn = h & 0xffff;
                const int base = S.kb[i + j < cnt ? i + j : i] - kw;  // bits[base + w]: window word w
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    const int w = lane + 32 * u;
                    t[j][u] = h != 0 && w >= kw && w < kw + kn ? bits[base + w] : 0u;
                }
            }
#pragma unroll
            for (int j = 0; j < U; ++j)
#pragma unroll
                for (int u = 0; u < R; ++u) reg[u] |= t[j][u];
        }
        __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int w = lane + 32 * u;
        if (w < W && reg[u]) S.pm[w].y |= reg[u];
    }
    __syncwarp();
}

// Mark every output column of row r in [c0, cend) (cend - c0 <= kCols).
// BMP: B row bitmaps may be used (not in the batch kernel's wide window).
// PAIR: long B rows are marked two at a time (not in the batch kernel, which
// runs at its register limit).
template <bool TAB, bool BMP = false, bool PAIR = false, int W>
__device__ __forceinline__ void build_map(const ProductArgs& P, const AddTerm* add, int nadd, unsigned tmask, int r,
                                          int c0, int cend, int pa0, int pa1, bool whole, int lane, ProdSmem<TAB, W>& S,
                                          bool store_a, int ab, int ae, bool a_holes = false,
                                          unsigned long long* fma = nullptr) {
    clear_map(cend - c0, lane, S);
    __syncwarp();
    for (int t = 0; t < nadd; ++t) {
        if (!((tmask >> t) & 1u)) continue;
        const AddTerm& T = add[t];
        if (!T.rd) {
            if (lane == 0 && r >= c0 && r < cend) mark_one(r - c0, S);
        } else {
            // (term t's row range is in lane t)
            const int s = __shfl_sync(kFull, ab, t), e = __shfl_sync(kFull, ae, t);
            if constexpr (TAB) mark_row(P.pool_col, s, e, c0, cend, lane, S);
            else mark_row<true>(P.pool_col, s, e, c0, cend, lane, S);
        }
    }
    if constexpr (!TAB && BMP) {
        if (whole && P.bhdr) {
            mark_from_bitmaps(P, pa0, pa1, c0, cend, lane, S, store_a, a_holes, fma);
            return;
        }
    }
    for (int seg = pa0; seg < pa1; seg += 32) {
        const int cnt = min(32, pa1 - seg);
        load_segment<TAB>(P, seg, cnt, whole, c0, cend, lane, S, store_a, a_holes, fma);
        if constexpr (!TAB) {
            if (warp_max(lane < cnt ? S.kl[lane] : 0) <= 32) {
                mark_rows_short(P.B.col, cnt, c0, cend, lane, S);
                __syncwarp();
                continue;
            }
        }
        if constexpr (TAB) {
            for (int i = 0; i < cnt; ++i) mark_row(P.B.col, S.kb[i], S.kb[i] + S.kl[i], c0, cend, lane, S);
        } else {
            int i = 0;
            if constexpr (PAIR)
                for (; i + 1 < cnt; i += 2)
                    mark_row_pair(P.B.col, S.kb[i], S.kb[i] + S.kl[i], S.kb[i + 1], S.kb[i + 1] + S.kl[i + 1], c0,
                                  lane, S);
            for (; i < cnt; ++i) mark_row<false>(P.B.col, S.kb[i], S.kb[i] + S.kl[i], c0, cend, lane, S);
        }
        __syncwarp();
    }
    __syncwarp();
}

// number of marked columns in [0, wlen)
__device__ __forceinline__ int count_marks(int wlen, int lane, const ProdSmem<true>& S, int& /*words*/) {
    int total = 0;
    for (int i0 = 0; i0 < wlen; i0 += 32) {
        int i = i0 + lane;
        total += __popc(__ballot_sync(kFull, i < wlen && S.tab[i] != 0));
    }
    return total;
}
// (the upper half: words with a mark, for the map's choice)
template <int W>
__device__ __forceinline__ int count_marks(int wlen, int lane, const ProdSmem<false, W>& S, int& words) {
    int s = 0;
    for (int w = lane; w < ((wlen + 31) >> 5); w += 32) {
        const unsigned b = S.pm[w].y;
        s += __popc(b) + (b ? 1 << 16 : 0);
    }
    s = warp_sum(s);
    words += s >> 16;
    return s & 0xffff;
}

// Number the marked columns of [0, wlen) in ascending order and fill
// colbuf.  Only the first kAccCap get a slot; returns their count and sets
// *cut to the offset of the first column without one (wlen if all fit).
__device__ __forceinline__ int assign_slots(int wlen, int cap, int lane, ProdSmem<true>& S, int* cut) {
    int run = 0, cutoff = wlen;
    for (int i0 = 0; i0 < wlen; i0 += 32) {
        const int i = i0 + lane;
        const bool f = i < wlen && S.tab[i] != 0;
        const unsigned m = __ballot_sync(kFull, f);
        const int slot = run + __popc(m & lanemask_lt());
        if (f && slot < cap) {
            S.tab[i] = (unsigned short)slot;
            S.colbuf[slot] = (unsigned short)i;
        }
        if (run <= cap && run + __popc(m) > cap) {
            const unsigned fo = __ballot_sync(kFull, f && slot == cap);
            cutoff = i0 + __ffs(fo) - 1;
        }
        run += __popc(m);
        if (cutoff < wlen) break;
    }
    __syncwarp();
    *cut = cutoff;
    return min(run, cap);
}
template <int W>
__device__ __forceinline__ int assign_slots(int wlen, int cap, int lane, ProdSmem<false, W>& S, int* cut) {
    constexpr int per = (W + 31) / 32;  // words per lane (the last lanes' partly past nw)
    const int nw = (wlen + 31) >> 5;
    const int base = lane * per;
    int s = 0;
#pragma unroll
    for (int i = 0; i < per; ++i) s += base + i < nw ? __popc(S.pm[base + i].y) : 0;
    int run = warp_excl_scan(s, lane);
    const int total = __shfl_sync(kFull, run + s, 31);
#pragma unroll
    for (int i = 0; i < per; ++i) {
        if (base + i < nw) {
            S.pm[base + i].x = (unsigned)run;
            run += __popc(S.pm[base + i].y);
        }
    }
    __syncwarp();
    int cutoff = wlen;
    if (total > cap) {
        int found = INT_MAX;
        for (int w = lane; w < nw; w += 32) {
            const int pc = __popc(S.pm[w].y), pre = (int)S.pm[w].x;
            if (pre <= cap && cap < pre + pc) {
                unsigned bits = S.pm[w].y;
                for (int i = 0; i < cap - pre; ++i) bits &= bits - 1u;  // drop the lowest ones
                found = w * 32 + (__ffs(bits) - 1);
            }
        }
        cutoff = warp_min(found);
    }
    if (nw <= 8) {
        // a few words: lane l takes bit l of one word at a time (no lane
        // walks a word's set bits alone)
        for (int w = 0; w < nw; ++w) {
            const unsigned bits = S.pm[w].y;
            if ((bits >> lane) & 1u) {
                const int o = w * 32 + lane;
                if (o < cutoff) S.colbuf[(int)S.pm[w].x + __popc(bits & lanemask_lt())] = (unsigned short)o;
            }
        }
    } else {
        for (int w = lane; w < nw; w += 32) {
            unsigned bits = S.pm[w].y;
            int idx = (int)S.pm[w].x;
            while (bits) {
                const int o = w * 32 + __ffs(bits) - 1;
                if (o < cutoff) S.colbuf[idx] = (unsigned short)o;
                ++idx;
                bits &= bits - 1u;
            }
        }
    }
    __syncwarp();
    *cut = cutoff;
    return min(total, cap);
}

// The 128 entries [off, off + 128) of B row kk of the segment, four 32-entry
// pieces, one element of each per lane (column -1: no element).
struct Chunk {
    int c[4];
    double v[4];
};

template <bool TAB, int W>
__device__ __forceinline__ void chunk_load(const int* bcol, const double* bval,
                                           const ProdSmem<TAB, W>& S, int kk, int off, int lane, Chunk& ch) {
    const int len = S.kl[kk];
    const int* rc = bcol + S.kb[kk] + lane;
    const double* rv = bval + S.kb[kk] + lane;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int q = off + u * 32;
        ch.c[u] = -1;
        if (q + lane < len) {
            ch.c[u] = rc[q];
            ch.v[u] = rv[q];
        }
    }
}

template <bool TAB, int W>
__device__ __forceinline__ void chunk_next(const ProdSmem<TAB, W>& S, int cnt, int& kk, int& off) {
    off += 128;
    if (off >= S.kl[kk]) {
        off = 0;
        do {
            ++kk;
        } while (kk < cnt && S.kl[kk] == 0);
    }
}

// Fold a chunk in: its columns are distinct, so the four read-modify-writes
// are independent and are interleaved.  `np` (the same in every lane) is the
// number of pieces holding entries: a DFMA occupies the FP64 pipe for the
// whole warp, so the empty pieces at a row's end are branched over.
template <bool TAB, int W>
__device__ __forceinline__ void chunk_fold(ProdSmem<TAB, W>& S, const Chunk& ch, double a, int c0, int np = 4) {
    int i[4];
    double x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) i[u] = ch.c[u] >= 0 ? slot_lookup(S, ch.c[u] - c0) : -1;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (i[u] >= 0) x[u] = S.acc[i[u]];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (u >= np) break;
        if (i[u] >= 0) S.acc[i[u]] = __fma_rn(a, ch.v[u], x[u]);
    }
}

// acc[slot(j)] = fma(a_rk, b_kj, acc[slot(j)]) for the segment's k in order.
// Table map: chunks stream through three register sets (the loads of the
// next two are in flight while one is folded in).  Bitmap map (more warps,
// fewer registers): one chunk at a time.  A warp barrier separates
// consecutive B rows (the order of the fma chain).
template <bool WIDE>
__device__ __forceinline__ void accumulate_segment(const ProductArgs& P, int /*seg*/, int cnt, int c0, int lane,
                                                   ProdSmem<true>& S, bool /*wide_row*/) {
    const int* bcol = P.B.col;
    const double* bval = P.B.val;
    int k0 = 0, o0 = 0;
    while (k0 < cnt && S.kl[k0] == 0) ++k0;
    if (k0 >= cnt) return;
    Chunk A, B, C;
    chunk_load<true>(bcol, bval, S, k0, o0, lane, A);
    int k1 = k0, o1 = o0;
    chunk_next<true>(S, cnt, k1, o1);
    int k2 = k1, o2 = o1;
    if (k1 < cnt) {
        chunk_load<true>(bcol, bval, S, k1, o1, lane, B);
        chunk_next<true>(S, cnt, k2, o2);
    }
    auto step = [&](Chunk& X, Chunk& Z) -> bool {
        if (k2 < cnt) chunk_load<true>(bcol, bval, S, k2, o2, lane, Z);
        chunk_fold<true>(S, X, S.ka[k0], c0);
        if (k1 >= cnt) return false;
        if (k1 != k0) __syncwarp();
        k0 = k1;
        o0 = o1;
        k1 = k2;
        o1 = o2;
        if (k2 < cnt) chunk_next<true>(S, cnt, k2, o2);
        return true;
    };
    for (;;) {
        if (!step(A, C)) break;
        if (!step(B, A)) break;
        if (!step(C, B)) break;
    }
    __syncwarp();
}
// One 32-lane piece of short B row kk (at most 32 entries): column -1 where
// there is none.
template <int W>
__device__ __forceinline__ void short_load(const int* bcol, const double* bval,
                                           const ProdSmem<false, W>& S, int cnt, int kk, int lane, int& c, double& v) {
    c = -1;
    v = 0.0;
    if (kk < cnt && lane < S.kl[kk]) {
        const int q = S.kb[kk] + lane;
        c = bcol[q];
        v = bval[q];
    }
}
template <int W>
__device__ __forceinline__ void short_fold(ProdSmem<false, W>& S, int c, double v, double a, int c0) {
    if (c >= 0) {
        const int i = slot_lookup(S, c - c0);
        S.acc[i] = __fma_rn(a, v, S.acc[i]);
    }
}

template <bool WIDE, int W>
__device__ __forceinline__ void accumulate_segment(const ProductArgs& P, int seg, int cnt, int c0, int lane,
                                                   ProdSmem<false, W>& S, bool wide_row) {
    const int* bcol = P.B.col;
    const double* bval = P.B.val;
    const double* ka = ka_of(S);
    // a_rk of row kk: kept in the accumulator's last slots, or (WIDE, or a
    // row that takes every slot) read from A's row (the same address in
    // every lane)
    const bool a_global = WIDE || wide_row;
    auto a_of = [&](int kk) { return a_global ? P.A.val[seg + kk] : ka[kk]; };
    if (warp_max(lane < cnt ? S.kl[lane] : 0) <= 32) {
        // every B row is one piece: the pieces of the next three rows are
        // loaded while one is folded (rows in k order, a warp barrier between)
        int ca, cb, cc, cd;
        double va, vb, vc, vd;
        short_load(bcol, bval, S, cnt, 0, lane, ca, va);
        short_load(bcol, bval, S, cnt, 1, lane, cb, vb);
        short_load(bcol, bval, S, cnt, 2, lane, cc, vc);
        for (int kk = 0; kk < cnt; kk += 4) {
            short_load(bcol, bval, S, cnt, kk + 3, lane, cd, vd);
            short_fold(S, ca, va, a_of(kk), c0);
            __syncwarp();
            if (kk + 1 >= cnt) break;
            short_load(bcol, bval, S, cnt, kk + 4, lane, ca, va);
            short_fold(S, cb, vb, a_of(kk + 1), c0);
            __syncwarp();
            if (kk + 2 >= cnt) break;
            short_load(bcol, bval, S, cnt, kk + 5, lane, cb, vb);
            short_fold(S, cc, vc, a_of(kk + 2), c0);
            __syncwarp();
            if (kk + 3 >= cnt) break;
            short_load(bcol, bval, S, cnt, kk + 6, lane, cc, vc);
            short_fold(S, cd, vd, a_of(kk + 3), c0);
            __syncwarp();
        }
        return;
    }
    for (int kk = 0; kk < cnt; ++kk) {
        const int len = S.kl[kk];
        if (len == 0) continue;
        const double a = a_of(kk);
        if (len <= 32) {
            // a short B row fills one piece: fold only that one (a DFMA
            // occupies the FP64 pipe for the whole warp, active lanes or not)
            if (lane < len) {
                const int q = S.kb[kk] + lane;
                const int i = slot_lookup(S, bcol[q] - c0);
                S.acc[i] = __fma_rn(a, bval[q], S.acc[i]);
            }
        } else {
            // whole 128-entry chunks: four full pieces, no per-lane tests
            const int* rc = bcol + S.kb[kk] + lane;
            const double* rv = bval + S.kb[kk] + lane;
            int off = 0;
            for (; off + 128 <= len; off += 128) {
                int j[4];
                double v[4], x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    j[u] = rc[off + 32 * u];
                    v[u] = rv[off + 32 * u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) j[u] = slot_lookup(S, j[u] - c0);
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = S.acc[j[u]];
#pragma unroll
                for (int u = 0; u < 4; ++u) S.acc[j[u]] = __fma_rn(a, v[u], x[u]);
            }
            // the rest (up to four pieces, the last one partial), two pieces
            // at a time with their read-modify-writes interleaved
            for (; off < len; off += 64) {
                const bool in0 = off + lane < len;
                const bool two = off + 32 < len;  // (the same in every lane)
                const bool in1 = two && off + 32 + lane < len;
                int j0 = 0, j1 = 0;
                double v0 = 0.0, v1 = 0.0, x0 = 0.0, x1 = 0.0;
                if (in0) {
                    j0 = rc[off];
                    v0 = rv[off];
                }
                if (in1) {
                    j1 = rc[off + 32];
                    v1 = rv[off + 32];
                }
                if (in0) j0 = slot_lookup(S, j0 - c0);
                if (in1) j1 = slot_lookup(S, j1 - c0);
                if (in0) x0 = S.acc[j0];
                if (in1) x1 = S.acc[j1];
                if (in0) S.acc[j0] = __fma_rn(a, v0, x0);
                if (two && in1) S.acc[j1] = __fma_rn(a, v1, x1);
            }
        }
        __syncwarp();
    }
}

// ---- the list map
__device__ __forceinline__ void clear_map(int wlen, int lane, ProdSmem<false, kListWords>& S) {
    unsigned* id4 = reinterpret_cast<unsigned*>(S.id);
    for (int i = lane; i < (wlen + 127) >> 7; i += 32) id4[i] = 0xffffffffu;
}
// OR `bits` into window word w for the active lanes, whose words are
// distinct; nid: words in use so far (past kListIds: the map is full, and the
// mark is dropped).
__device__ __forceinline__ void list_or(ProdSmem<false, kListWords>& S, bool active, int w, unsigned bits, int& nid) {
    const unsigned i = active ? S.id[w] : 0u;
    const bool fresh = active && i == kNoId;
    const unsigned m = __ballot_sync(kFull, fresh);
    if (fresh) {
        const int j = nid + __popc(m & lanemask_lt());
        if (j < kListIds) {
            S.id[w] = (unsigned char)j;
            S.word[j] = (unsigned short)w;
            S.pm[j] = make_uint2(0u, bits);
        }
    } else if (active) {
        S.pm[i].y |= bits;
    }
    nid += __popc(m);
    __syncwarp();
}
// The columns of [c0, cend) among the row [s, e) (ascending), 32 at a time:
// the lanes of one word form a run, whose bits a segmented OR collects.
__device__ __forceinline__ void list_mark_row(const int* col, int s, int e, int c0, int cend, int lane,
                                              ProdSmem<false, kListWords>& S, int& nid) {
    for (int q0 = s; q0 < e; q0 += 32) {
        const int q = q0 + lane;
        const int c = q < e ? col[q] : INT_MAX;
        const bool in = c >= c0 && c < cend;
        const int w = in ? (c - c0) >> 5 : -1 - lane;
        unsigned v = in ? 1u << ((c - c0) & 31) : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned v2 = __shfl_down_sync(kFull, v, d);
            const int w2 = __shfl_down_sync(kFull, w, d);
            if (lane + d < 32 && w2 == w) v |= v2;
        }
        const int wp = __shfl_up_sync(kFull, w, 1);
        list_or(S, in && (lane == 0 || wp != w), w, v, nid);
    }
}
// Mark every output column of row r in [c0, cend), c0 a multiple of 32;
// returns the words in use (more than kListIds: the window is too wide).
__device__ __forceinline__ int list_build(const ProductArgs& P, const AddTerm* add, int nadd, int r, int c0, int cend,
                                          int pa0, int pa1, int lane, ProdSmem<false, kListWords>& S, int ab, int ae) {
    int nid = 0;
    clear_map(cend - c0, lane, S);
    __syncwarp();
    for (int t = 0; t < nadd; ++t) {
        if (!add[t].rd) {
            list_or(S, lane == 0 && r >= c0 && r < cend, (r - c0) >> 5, 1u << ((r - c0) & 31), nid);
        } else {
            list_mark_row(P.pool_col, __shfl_sync(kFull, ab, t), __shfl_sync(kFull, ae, t), c0, cend, lane, S, nid);
        }
    }
    const int wb = c0 >> 5;
    const unsigned nw = (unsigned)((cend - c0 + 31) >> 5);
    for (int seg = pa0; seg < pa1 && nid <= kListIds; seg += 32) {
        const int cnt = min(32, pa1 - seg);
        if (lane < cnt) {
            const int k = P.A.col[seg + lane];
            S.kb[lane] = P.B.rb[k];
            S.kl[lane] = P.bhdr[k].y;
        }
        __syncwarp();
        // four B rows' first words are loaded before any is marked
        for (int i0 = 0; i0 < cnt; i0 += 4) {
            uint2 t[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                t[j] = make_uint2(0xffffffffu, 0u);
                if (i0 + j < cnt && lane < S.kl[i0 + j]) t[j] = P.blists[S.kb[i0 + j] + lane];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (i0 + j >= cnt) break;
                const int m = S.kl[i0 + j];
                const unsigned w = t[j].x - (unsigned)wb;
                list_or(S, lane < m && w < nw, (int)w, t[j].y, nid);
                for (int l0 = 32; l0 < m; l0 += 32) {
                    uint2 x = make_uint2(0xffffffffu, 0u);
                    if (l0 + lane < m) x = P.blists[S.kb[i0 + j] + l0 + lane];
                    const unsigned w2 = x.x - (unsigned)wb;
                    list_or(S, l0 + lane < m && w2 < nw, (int)w2, x.y, nid);
                }
            }
        }
        __syncwarp();
    }
    return nid;
}
// The same for the widest window from c0 on that the map holds (cend is cut,
// to a multiple of 32); returns the columns marked (ids: the words in use).
__device__ __forceinline__ int list_chunk(const ProductArgs& P, const AddTerm* add, int nadd, int r, int c0, int& cend,
                                          int pa0, int pa1, int lane, ProdSmem<false, kListWords>& S, int ab, int ae,
                                          int& words, int& ids) {
    for (;;) {
        const int nid = list_build(P, add, nadd, r, c0, cend, pa0, pa1, lane, S, ab, ae);
        if (nid <= kListIds) {
            int s = 0;
            for (int i = lane; i < nid; i += 32) s += __popc(S.pm[i].y);
            words += nid;
            ids = nid;
            return warp_sum(s);
        }
        words = max(words, kListIds + 1);
        cend = c0 + max(32, ((cend - c0) / 2) & ~31);
    }
}
// Number the columns from window word `from` on in ascending order and fill
// colbuf, whole words of them while they fit `cap` slots; returns their count, *cut: the offset of the
// first word without slots (wlen if all fit).
__device__ __forceinline__ int assign_slots(int wlen, int cap, int lane, ProdSmem<false, kListWords>& S, int* cut,
                                            int from, int ids) {
    const int nw = (wlen + 31) >> 5, per = (nw - from + 31) >> 5;
    const int b = min(nw, from + lane * per), e = min(nw, b + per);
    int s = 0;
    for (int w = b; w < e; ++w) {
        const unsigned i = S.id[w];
        if (i != kNoId) s += __popc(S.pm[i].y);
    }
    int run = warp_excl_scan(s, lane);
    const int total = __shfl_sync(kFull, run + s, 31);
    int cw = nw;  // first word that does not fit
    int cs = total;
    for (int w = b; w < e; ++w) {
        const unsigned i = S.id[w];
        if (i == kNoId) continue;
        const unsigned bits = S.pm[i].y;
        S.pm[i].x = (unsigned)run;
        if (run + __popc(bits) > cap && cw == nw) {
            cw = w;
            cs = run;
        }
        run += __popc(bits);
    }
    int cutoff = wlen, cnt = total;
    if (total > cap) {
        const int w = warp_min(cw);
        cnt = warp_min(cw == w ? cs : INT_MAX);
        cutoff = w * 32;
    }
    __syncwarp();
    // the words in use, one a turn: lane l takes bit l
    for (int i = 0; i < ids; ++i) {
        const uint2 p = S.pm[i];
        const int o = S.word[i] * 32 + lane;
        if ((p.y >> lane & 1u) && o >= from * 32 && o < cutoff) S.colbuf[p.x + __popc(p.y & lanemask_lt())] = (unsigned short)o;
    }
    __syncwarp();
    *cut = cutoff;
    return cnt;
}

// Statistics of one row of a batched step, added to its instance's record:
// multiply-adds (per-lane partial counts), Algorithm 1 candidates (per lane),
// entries written and the largest |x| (per lane).
__device__ __forceinline__ void row_stats_batch(const ProductArgs& P, int inst, unsigned long long fma,
                                                unsigned long long cand, int written, unsigned long long absmax,
                                                int lane, int span = 0) {
    for (int o = 16; o; o >>= 1) {
        fma += __shfl_xor_sync(kFull, fma, o);
        cand += __shfl_xor_sync(kFull, cand, o);
    }
    absmax = warp_max_u64(absmax);
    if (lane == 0) {
        if (P.stat_tab) {
            StepStat* st = P.stat_tab + inst;
            if (fma) atomicAdd(&st->fma, fma);
            if (written) atomicAdd(&st->nnz_pre, (unsigned long long)written);
            if (cand) atomicAdd(&st->ncand, cand);
            if (span > 0) atomicMax(&st->span_max, (unsigned)span);
        }
        if (P.absmax_slot && absmax) atomicMax(&(P.absmax_slot + (size_t)inst * P.absmax_stride)->absmax, absmax);
    }
}

__device__ __forceinline__ void write_desc(const ProductArgs& P, int r, const RowDesc& d) {
    P.out_rb[r] = d.rb;
    P.out_re[r] = d.re;
    P.out_rd[r] = d;
}
// step_done of a product step
__device__ __forceinline__ void product_done(const ProductArgs& P) {
    step_done(P.ctl, P.mark, P.stat ? &P.stat->pool_start : nullptr, P.start_out, P.cslot, P.ncslot);
}
// The descriptor of the entries written at [base, base + n), one per column
// that has an entry (read back by a lane of the warp that wrote them).
__device__ __forceinline__ RowDesc stored_row(const ProductArgs& P, long long base, int n) {
    if (n <= 0) return RowDesc{0, 0, 0, 0};
    return rd_row((int)base, (int)base + n, P.pool_col[base], P.pool_col[base + n - 1]);
}

// Per-warp state of the product kernel across the rows a warp processes.
struct RowState {
    unsigned long long written = 0ull, cand = 0ull, absmax = 0ull, fma = 0ull;
    int span = 0;   // widest column window of this warp's rows
    int words = 0;  // most words that one of them has entries in
    Arena arena;
    CandArena carena;
};

// One output row r of C = sum_t alpha_t M_t + A B (see k_product), processed
// by one warp with the slot map S.
template <bool TAB, bool BATCH, bool WIDE, int W>
__device__ __forceinline__ void product_row(const ProductArgs& P, const AddTerm* add, ProdSmem<TAB, W>& S,
                                            RowState& st, int r, int lane) {
    using Smem = ProdSmem<TAB, W>;
    // columns and slots of one chunk (lowered only to exercise chunking)
    const int kCols = P.chunk_cols > 0 && P.chunk_cols < Smem::kCols ? P.chunk_cols : Smem::kCols;
    constexpr int kCapN = (TAB || WIDE) ? kAccCap : kAccCap - 32;  // a row's slots
    const int kSlots = P.chunk_slots > 0 && P.chunk_slots < kCapN ? P.chunk_slots : kCapN;
    const int nadd = P.nadd;
    const unsigned long long eps_bits = (unsigned long long)__double_as_longlong(P.eps_g);
    unsigned long long& my_written = st.written;
    unsigned long long& my_cand = st.cand;
    unsigned long long& my_absmax = st.absmax;
    unsigned long long& my_fma = st.fma;
    int& my_span = st.span;
    Arena& arena = st.arena;
    CandArena& carena = st.carena;


    // ---- the row's terms: single instance, every term and the product;
    // batch, what the row's instance does in this step
    bool prod = P.A.rb != nullptr;
    unsigned tmask = kFull;  // terms present in this row (batch: coefficient != 0)
    int r_inst = 0;
    if constexpr (BATCH) {
        r_inst = P.inst[r];
        const BatchStep bs = P.bstep[r_inst];
        // the row equals the norm phase's power: k_reuse_copy_batch writes it
        if (bs.reuse && __ldcg(P.inst_dropped + r_inst) == 0) return;
        if (bs.mode == kBatchSkip || bs.mode == kBatchPass) {
            if (lane == 0) write_desc(P, r, bs.mode == kBatchPass ? P.B.rd[r] : RowDesc{0, 0, 0, 0});
            return;
        }
        prod = bs.mode == kBatchProduct;
        const double a_lane = lane < nadd ? P.alpha_tab[(size_t)lane * P.ninst + r_inst] : 0.0;
        tmask = __ballot_sync(kFull, __double_as_longlong(a_lane) != 0ll);
    }
    // batch: the counters are per row (reported per instance after each
    // row); single: running totals, reported per block at the end
    if constexpr (BATCH) {
        my_fma = 0ull;
        my_cand = 0ull;
    }
    const unsigned long long fma0 = BATCH ? 0ull : my_fma, cand0 = BATCH ? 0ull : my_cand;
    // ---- column window of row r and the row's multiply-add count.  A
    // matrix (or a batch instance) of at most one map's columns is its own
    // window: no loads to find the row's, and the B row lengths are counted
    // while the map is built
    int lo = INT_MAX, hi = -1;
    bool fixed = false;
    int fixed_span = 0;
    constexpr bool LIST = !TAB && W == kListWords;
    if constexpr (!TAB && !LIST) {
        int w0 = 0, w1 = P.n;
        if constexpr (BATCH) {
            w1 = -1;
            if (P.inst_off) {
                w0 = P.inst_off[r_inst];
                w1 = P.inst_off[r_inst + 1];
            }
        }
        // with B row bitmaps the window starts at a multiple of 32 columns
        const int a0 = P.bhdr ? (w0 & ~31) : w0;
        if (w1 > w0 && w1 - a0 <= kCols) {
            lo = a0;
            hi = w1 - 1;
            fixed = true;
            fixed_span = w1 - w0;
        }
    }
    // addend term t's row range, in lane t (the terms' loads in parallel;
    // the loops over the terms below take it with a shuffle)
    RowDesc ad{0, 0, 0, 0};
    const bool my_term = lane < nadd && ((tmask >> lane) & 1u);
    if (my_term && add[lane].rd) ad = add[lane].rd[r];
    const int ab = ad.rb, ae = ad.re;
    if (!fixed && my_term) {
        if (!add[lane].rd) {
            lo = min(lo, r);
            hi = max(hi, r);
        } else if (ab < ae) {
            lo = min(lo, rd_first(ad));
            hi = max(hi, rd_last(ad));
        }
    }
    int pa0 = 0, pa1 = 0;
    bool a_holes = false;  // A's row stores exact zeros, which are no terms
    if (prod) {
        pa0 = P.A.rb[r];
        pa1 = P.A.re[r];
        a_holes = P.A.rd && pa1 - pa0 != rd_nnz(P.A.rd[r]);
    }
    for (int p = pa0 + lane; p < pa1 && !fixed; p += 32) {
        const RowDesc d = P.B.rd[P.A.col[p]];
        if (!(a_holes && P.A.val[p] == 0.0)) my_fma += (unsigned long long)rd_nnz(d);
        if (d.rb < d.re) {
            lo = min(lo, rd_first(d));
            hi = max(hi, rd_last(d));
        }
    }
    if (my_term) my_fma += add[lane].rd ? (unsigned long long)rd_nnz(ad) : 1ull;
    lo = warp_min(lo);
    hi = warp_max(hi);
    const int row_span = fixed ? fixed_span : hi - lo + 1;  // the statistic: before any alignment
    my_span = max(my_span, row_span);
    if (hi < lo) {
        if (lane == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
        if constexpr (BATCH) row_stats_batch(P, r_inst, my_fma - fma0, 0ull, 0, 0ull, lane);
        return;
    }
    if constexpr (!TAB) {
        if (P.bhdr) lo &= ~31;
    }

    // ---- exact entry count of the row, reserve it in the pool
    long long total = 0;
    bool reuse = false;
    int words = 0, ids = 0;
    if constexpr (LIST) {
        for (long long c0 = lo; c0 <= hi;) {
            int cend = (int)min((long long)hi + 1, c0 + kCols);
            total += list_chunk(P, add, nadd, r, (int)c0, cend, pa0, pa1, lane, S, ab, ae, words, ids);
            reuse = c0 == lo && cend == hi + 1;
            c0 = cend;
        }
    } else if (hi - lo + 1 <= kCols) {
        build_map<TAB, (!BATCH || W == kBmWords), !BATCH>(P, add, nadd, tmask, r, lo, hi + 1, pa0, pa1, true, lane, S,
                                                   !WIDE, ab, ae, a_holes, fixed ? &my_fma : nullptr);
        total = count_marks(hi - lo + 1, lane, S, words);
        reuse = true;
    } else {
        for (long long c0 = lo; c0 <= hi; c0 += kCols) {
            int cend = (int)min((long long)hi + 1, c0 + kCols);
            build_map<TAB, false, !BATCH>(P, add, nadd, tmask, r, (int)c0, cend, pa0, pa1, false, lane, S, !WIDE, ab,
                                          ae);
            total += count_marks(cend - (int)c0, lane, S, words);
        }
    }
    st.words = max(st.words, words);
    const long long base = arena_take(arena, (unsigned long long)((total + 3) & ~3LL), P.arena, P.ctl, P.pool_val, lane);
    if (base < 0) {
        if (lane == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
        return;
    }
    // a row of the narrow accumulator that fits every slot (kAccCap) in one
    // chunk takes them all and reads a_rk from A's row, as WIDE does,
    // instead of two column chunks (single-matrix kernels: the batch kernel
    // runs at its register limit)
    bool wide_row = WIDE;
    int slots = kSlots;
    if constexpr (!TAB && !WIDE && !BATCH) {
        if (reuse && total > kSlots && total <= kAccCap && P.chunk_slots <= 0) {
            wide_row = true;
            slots = kAccCap;
        }
    }
    const bool single = reuse && total <= slots;
    int written = 0;
    int c0 = lo;
    // the map's columns are [m0, mend): a chunk's, but the list map's serves
    // every chunk of slots inside them
    int m0 = lo, mend = LIST && reuse ? hi + 1 : lo;
    while (c0 <= hi) {
        int cend = (int)min((long long)hi + 1, (long long)c0 + kCols);
        if constexpr (LIST) {
            if (c0 >= mend) {
                int w = 0;
                list_chunk(P, add, nadd, r, c0, cend, pa0, pa1, lane, S, ab, ae, w, ids);
                m0 = c0;
                mend = cend;
            }
            cend = mend;
        } else if (!reuse) {
            build_map<TAB, false, !BATCH>(P, add, nadd, tmask, r, c0, cend, pa0, pa1, false, lane, S, !WIDE, ab, ae);
        }
        if constexpr (!LIST) m0 = c0;
        reuse = false;
        int cut, cnt;
        if constexpr (LIST)
            cnt = assign_slots(cend - m0, slots, lane, S, &cut, (c0 - m0) >> 5, ids);
        else
            cnt = assign_slots(cend - m0, slots, lane, S, &cut);
        const int c1 = m0 + cut;
        for (int i = lane; i < cnt; i += 32) S.acc[i] = 0.0;
        __syncwarp();

        // ---- weighted sum of the addends, t ascending
        for (int t = 0; t < nadd; ++t) {
            if (!((tmask >> t) & 1u)) continue;
            const AddTerm& T = add[t];
            // batch: the row's instance's coefficient (a small, cached table)
            const double alpha = BATCH ? P.alpha_tab[(size_t)t * P.ninst + r_inst] : T.alpha;
            if (!T.rd) {
                if (lane == 0 && r >= c0 && r < c1) {
                    int i = slot_lookup(S, r - m0);
                    S.acc[i] = __fma_rn(alpha, 1.0, S.acc[i]);
                }
            } else {
                const int s = __shfl_sync(kFull, ab, t), e = __shfl_sync(kFull, ae, t);
                for (int q = s + lane; q < e; q += 32) {
                    int c = P.pool_col[q];
                    if (c >= c0 && c < c1) {
                        int i = slot_lookup(S, c - m0);
                        S.acc[i] = __fma_rn(alpha, P.pool_val[q], S.acc[i]);
                    }
                }
            }
            __syncwarp();
        }

        // ---- product A B: k of row r ascending
        for (int seg = pa0; seg < pa1; seg += 32) {
            const int cnt_seg = min(32, pa1 - seg);
            load_segment<TAB>(P, seg, cnt_seg, single, c0, c1, lane, S, !wide_row, false);
            accumulate_segment<WIDE>(P, seg, cnt_seg, m0, lane, S, wide_row);
        }

        // ---- write back the nonzero entries in column order; the entries
        // with |x| <= eps_g enter the column sums of Algorithm 1's first pass
        // (batch: the filter of the row's instance, read here rather than
        // held in registers through the row)
        unsigned long long r_eps = eps_bits;
        int r_lsb = P.e_lsb;
        bool r_filt = P.filtering != 0;
        if constexpr (BATCH) {
            const BatchStep& bs = P.bstep[r_inst];
            r_filt = bs.eps_g > 0.0;
            r_eps = (unsigned long long)__double_as_longlong(bs.eps_g);
            r_lsb = bs.e_lsb;
        }
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            int i = i0 + lane;
            double x = 0.0;
            int c = 0;
            if (i < cnt) {
                x = S.acc[i];
                c = m0 + (int)S.colbuf[i];
            }
            unsigned long long xb = mag_bits(x);
            bool nz = i < cnt && xb != 0ull;
            unsigned m = __ballot_sync(kFull, nz);
            const bool cand = nz && r_filt && xb <= r_eps;
            if (nz) {
                long long pos = (long long)base + written + __popc(m & lanemask_lt());
                P.pool_col[pos] = c;
                P.pool_val[pos] = x;
                my_absmax = xb > my_absmax ? xb : my_absmax;
                if (cand) {
                    exact_add(P.words + c, (size_t)P.n, P.sticky + c, xb, r_lsb);
                    ++my_cand;
                }
            }
            if (P.cand_col)
                cand_push(carena, cand, c, xb, P.cand_col, P.cand_x, &P.ctl->cand_cnt[0], P.cand_cap,
                          P.cand_chunk, &P.ctl->cand_over, lane);
            written += __popc(m);
        }
        __syncwarp();
        c0 = c1;
    }
    // the row's unused reserved slots read as exact zeros (never candidates)
    const long long rend = base + ((total + 3) & ~3LL);
    for (long long q = base + written + lane; q < rend; q += 32) P.pool_val[q] = 0.0;
    __syncwarp();
    if (lane == 0) write_desc(P, r, stored_row(P, base, written));
    if constexpr (BATCH) {
        row_stats_batch(P, r_inst, my_fma - fma0, my_cand - cand0, written, my_absmax, lane, row_span);
        my_absmax = 0ull;
    } else if (lane == 0) {
        my_written += (unsigned long long)written;
    }
}

template <bool TAB, bool BATCH, bool WIDE, int W = kBmWords>
__global__ void __launch_bounds__(ProdSmem<TAB, W>::kWarps * 32, ProdSmem<TAB, W>::kBlocksPerSm)
    k_product(const __grid_constant__ ProductArgs P) {
    pdl_enter();
    // a baby step whose product equals an already computed power (no entry
    // dropped so far) is done by k_reuse_pass1 instead (same value in all blocks)
    if (P.skip_unless && __ldcg(P.skip_unless) == 0) return;
    using Smem = ProdSmem<TAB, W>;
    constexpr int kWarps = Smem::kWarps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AddTerm* add = reinterpret_cast<AddTerm*>(smem_raw);
    Smem* warps = reinterpret_cast<Smem*>(smem_raw + sizeof(AddTerm) * kMaxAdd);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nadd = P.nadd;
    for (int t = threadIdx.x; t < nadd; t += blockDim.x) add[t] = P.add[t];
    __shared__ unsigned long long blk_written, blk_cand, blk_absmax, blk_fma, blk_arena;
    __shared__ int blk_span, blk_words;
    if (threadIdx.x == 0) {
        // the block's warps take their first pool arenas with one atomic: at
        // the launch every warp wants one at once, on the same counter
        // (beside k_band a warp takes its first with its first row: it may have none)
        blk_arena = BATCH && P.pair ? ~0ull >> 1 : atomicAdd(&P.ctl->pool_used, (unsigned long long)kWarps * P.arena);
        blk_span = blk_words = 0;
        blk_fma = 0ull;
        blk_written = 0ull;
        blk_cand = 0ull;
        blk_absmax = 0ull;
    }
    __syncthreads();
    Smem& S = warps[wib];
    RowState st;
    // (past the pool's capacity the first row's arena_take reports the overflow)
    if (blk_arena + (unsigned long long)kWarps * P.arena <= P.ctl->pool_cap) {
        st.arena.next = blk_arena + (unsigned long long)wib * P.arena;
        st.arena.end = st.arena.next + P.arena;
    }
    for (int r = blockIdx.x * kWarps + wib; r < P.n; r += gridDim.x * kWarps) {
        if constexpr (BATCH)
            if (P.band && P.band[P.inst[r]]) continue;  // k_band's rows
        product_row<TAB, BATCH, WIDE, W>(P, add, S, st, r, lane);
    }
    // the unused end of this warp's arena reads as exact zeros too, and the
    // unused end of its candidate chunk as holes
    arena_close(st.arena, P.pool_val, lane);
    if (P.cand_col) cand_close(st.carena, P.cand_x, lane);
    if constexpr (BATCH) {
        if (!P.pair) product_done(P);
        return;
    }
    product_done(P);
    // ---- block totals for the step statistics
    st.cand = (unsigned long long)warp_sum((int)st.cand);
    st.absmax = warp_max_u64(st.absmax);
    for (int o = 16; o; o >>= 1) st.fma += __shfl_xor_sync(kFull, st.fma, o);
    if (lane == 0) {
        atomicAdd(&blk_fma, st.fma);
        atomicAdd(&blk_written, st.written);
        atomicAdd(&blk_cand, st.cand);
        atomicMax(&blk_absmax, st.absmax);
        atomicMax(&blk_span, st.span);
        atomicMax(&blk_words, st.words);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blk_fma) atomicAdd(&P.ctl->fma_total, blk_fma);
        if (P.stat) {
            if (blk_span > 0) atomicMax(&P.stat->span_max, (unsigned)blk_span);
            if (blk_words > 0) atomicMax(&P.stat->words_max, (unsigned)blk_words);
            if (blk_fma) atomicAdd(&P.stat->fma, blk_fma);
            if (blk_written) atomicAdd(&P.stat->nnz_pre, blk_written);
            if (blk_cand) atomicAdd(&P.stat->ncand, blk_cand);
        }
        if (P.absmax_slot && blk_absmax) atomicMax(&P.absmax_slot->absmax, blk_absmax);
    }
}


// Keep the entries of row [s, e) with |x| > fb (bits), in place and in
// column order; the dropped tail is cleared to exact zeros.  Returns the new
// end.  Rounds of 128 entries, software-pipelined: the loads of round i + 1
// are issued before the writes of round i.  Entries only move left, so the
// writes of round i stay below its end and never reach round i + 1's
// entries, which were read before the warp barrier that ends round i.
__device__ __forceinline__ void compact_load(const int* col, const double* val, int q0, int e, int lane, int c[4],
                                             double x[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int q = q0 + u * 32 + lane;
        c[u] = 0;
        x[u] = 0.0;
        if (q < e) {
            c[u] = col[q];
            x[u] = val[q];
        }
    }
}

__device__ __forceinline__ int compact_row(int* col, double* val, int s, int e, unsigned long long fb, int lane) {
    int w = s;
    int c[4];
    double x[4];
    compact_load(col, val, s, e, lane, c, x);
    for (int q0 = s; q0 < e; q0 += 128) {
        int cn[4];
        double xn[4];
        compact_load(col, val, q0 + 128, e, lane, cn, xn);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool keep = q0 + u * 32 + lane < e && mag_bits(x[u]) > fb;
            const unsigned m = __ballot_sync(kFull, keep);
            if (keep) {
                const int pos = w + __popc(m & lanemask_lt());
                col[pos] = c[u];
                val[pos] = x[u];
            }
            w += __popc(m);
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            c[u] = cn[u];
            x[u] = xn[u];
        }
    }
    for (int q = w + lane; q < e; q += 32) val[q] = 0.0;
    return w;
}

// Keep the entries of row r (descriptor d) with |x| > fb, in place; returns
// how many.  A full row stays full while at least three quarters of its
// columns between the first and the last kept entry keep theirs: the others
// become holes (exact zeros: they add nothing to any sum, fold or candidate
// list), so nothing moves and a product finds an entry at its column's place.
// Measured where rows are bands (half-bandwidth 5, n = 65536): the entries
// near the threshold are dropped one here, one there, and 0.9 and more stay.
__device__ __forceinline__ int filter_row(int* col, double* val, int* rb, int* re, RowDesc* rd, int r,
                                          unsigned long long fb, int lane) {
    const RowDesc d = rd[r];
    int s = d.rb, e = d.re;
    if (rd_full(d)) {
        int kept = 0, first = -1, last = -1;
        for (int q0 = s; q0 < e; q0 += 128) {
            double x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = q0 + u * 32 + lane;
                x[u] = q < e ? val[q] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q1 = q0 + u * 32;
                if (q1 >= e) break;
                const unsigned long long xb = mag_bits(x[u]);
                const unsigned m = __ballot_sync(kFull, xb > fb);
                if (xb != 0ull && xb <= fb) val[q1 + lane] = 0.0;
                if (m) {
                    if (first < 0) first = q1 + __ffs(m) - 1;
                    last = q1 + 31 - __clz(m);
                    kept += __popc(m);
                }
            }
        }
        if (kept == rd_nnz(d)) return kept;  // nothing dropped
        if (kept == 0) {
            if (lane == 0) {
                rb[r] = re[r] = 0;
                rd[r] = RowDesc{0, 0, 0, 0};
            }
            return 0;
        }
        const int c0 = rd_first(d) + (first - s);
        s = first;
        e = last + 1;
        if (4ll * kept >= 3ll * (e - s)) {
            if (lane == 0) {
                rb[r] = s;
                re[r] = e;
                rd[r] = rd_full_row(s, e, c0, kept);
            }
            return kept;
        }
        __syncwarp();
        fb = 0ull;  // too many holes: the kept entries alone
    }
    const int w = compact_row(col, val, s, e, fb, lane);
    if (w != d.re || s != d.rb) {
        __syncwarp();
        if (lane == 0) {
            const RowDesc n = w > s ? rd_row(s, w, col[s], col[w - 1]) : RowDesc{0, 0, 0, 0};
            rb[r] = n.rb;
            re[r] = n.re;
            rd[r] = n;
        }
    }
    return w - s;
}

// ---------------------------------------------------------------- k_product_cta
// One output row per block of four warps: for matrices with fewer rows than
// the warp-per-row kernel has resident warps, whose B rows are long.  The
// block's warps share one bitmap slot map over the row's window (up to 4608
// columns) and kCtaCap accumulator slots:
//  - symbolic pass: each warp marks the B rows of every fourth 32-entry
//    segment of A's row (from their bitmaps when the step has them), ORing
//    into the shared map; a block-wide scan numbers the columns;
//  - numeric pass: the addends in order, then the B rows in k order, each B
//    row's entries spread over the block's 128 threads (four independent
//    read-modify-writes per thread: a B row's entries have distinct
//    columns), with a block barrier after each B row, so that every slot is
//    folded in the order of k_product (addends t ascending, then k
//    ascending) and the results are bitwise the same;
//  - write-back: each warp takes a quarter of the slots in column order,
//    positions from a block-wide count, Algorithm 1's first pass as in
//    k_product.
// A row whose window or pattern does not fit is computed by the block's
// first warp with the warp-per-row code (bitmap map, every accumulator
// slot) in the same shared memory, the other warps waiting.
constexpr int kCtaWarps = 4;
constexpr int kCtaCap = 2560;

struct CtaSmem {
    uint2 pm[kBmWords];  // the first member, as in ProdSmem<false, kBmWords> (mark_row uses only pm)
    double acc[kCtaCap];
    unsigned short colbuf[kCtaCap];
    int kb[kCtaWarps][32];
    int kl[kCtaWarps][32];
    int kwn[kCtaWarps][32];
    double ka[32];
    int wcnt[kCtaWarps];
    int lo, hi, total, fits;
    long long base;
};
static_assert(sizeof(ProdSmem<false, kBmWords>) <= sizeof(CtaSmem), "the warp-per-row fallback fits");

size_t cta_smem_bytes() { return sizeof(CtaSmem) + sizeof(AddTerm) * kMaxAdd; }

// block-wide exclusive scan of one int per thread; *total gets the sum
__device__ __forceinline__ int cta_excl_scan(int v, int tid, int* wsum, int* total) {
    const int lane = tid & 31, wib = tid >> 5;
    const int x = warp_excl_scan(v, lane);
    if (lane == 31) wsum[wib] = x + v;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kCtaWarps; ++w) {
        before += w < wib ? wsum[w] : 0;
        all += wsum[w];
    }
    *total = all;
    __syncthreads();
    return before + x;
}

__device__ __forceinline__ void cta_row(const ProductArgs& P, const AddTerm* add, CtaSmem& S, RowState& st, int r,
                                        int tid) {
    const int lane = tid & 31, wib = tid >> 5;
    constexpr int kT = kCtaWarps * 32;
    const int nadd = P.nadd;
    const bool prod = P.A.rb != nullptr;
    int pa0 = 0, pa1 = 0;
    bool a_holes = false;
    if (prod) {
        pa0 = P.A.rb[r];
        pa1 = P.A.re[r];
        a_holes = P.A.rd && pa1 - pa0 != rd_nnz(P.A.rd[r]);
    }
    // ---- column window: the matrix itself when it is at most one map wide
    int lo = INT_MAX, hi = -1;
    int row_span = 0;
    if (P.n <= kBmBits) {
        lo = 0;
        hi = P.n - 1;
        row_span = P.n;
    } else {
        if (tid == 0)
            for (int t = 0; t < nadd; ++t) {
                const AddTerm& T = add[t];
                if (!T.rd) {
                    lo = min(lo, r);
                    hi = max(hi, r);
                } else {
                    const RowDesc d = T.rd[r];
                    if (d.rb < d.re) {
                        lo = min(lo, rd_first(d));
                        hi = max(hi, rd_last(d));
                    }
                }
            }
        for (int p = pa0 + tid; p < pa1; p += kT) {
            const RowDesc d = P.B.rd[P.A.col[p]];
            if (d.rb < d.re) {
                lo = min(lo, rd_first(d));
                hi = max(hi, rd_last(d));
            }
        }
        lo = warp_min(lo);
        hi = warp_max(hi);
        if (lane == 0) {
            S.kb[wib][0] = lo;
            S.kl[wib][0] = hi;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kCtaWarps; ++w) {
            lo = min(lo, S.kb[w][0]);
            hi = max(hi, S.kl[w][0]);
        }
        __syncthreads();
        row_span = hi - lo + 1;
    }
    if (hi < lo) {  // no entry at all
        if (tid == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
        return;
    }
    st.span = max(st.span, row_span);
    if (P.bhdr) lo &= ~31;
    const int wlen = hi - lo + 1;
    const int nw = (wlen + 31) >> 5;
    if (wlen > kBmBits) {
        // wider than the map: the first warp computes the row alone
        if (wib == 0)
            product_row<false, false, true, kBmWords>(P, add, *reinterpret_cast<ProdSmem<false, kBmWords>*>(&S), st,
                                                      r, lane);
        __syncthreads();
        return;
    }
    // ---- symbolic pass
    for (int w = tid; w < nw; w += kT) S.pm[w].y = 0u;
    __syncthreads();
    ProdSmem<false, kBmWords>& M = *reinterpret_cast<ProdSmem<false, kBmWords>*>(&S);  // its pm is S.pm
    if (wib == 0) {
        for (int t = 0; t < nadd; ++t) {
            const AddTerm& T = add[t];
            if (!T.rd) {
                if (lane == 0 && r >= lo && r <= hi) mark_one(r - lo, M);
            } else {
                const RowDesc d = T.rd[r];
                mark_row<true>(P.pool_col, d.rb, d.re, lo, hi + 1, lane, M);
            }
        }
    }
    unsigned long long rf = 0ull;  // this thread's share of the row's multiply-adds
    constexpr int R = (kBmWords + 31) / 32;
    unsigned reg[R];
#pragma unroll
    for (int u = 0; u < R; ++u) reg[u] = 0u;
    for (int seg = pa0 + 32 * wib; seg < pa1; seg += 32 * kCtaWarps) {
        const int cnt = min(32, pa1 - seg);
        if (lane < cnt) {
            const int k = P.A.col[seg + lane];
            const RowDesc d = P.B.rd[k];
            const int b = d.rb, e = d.re;
            if (!(a_holes && P.A.val[seg + lane] == 0.0)) rf += (unsigned long long)rd_nnz(d);
            S.kb[wib][lane] = b;
            S.kl[wib][lane] = e - b;
            int h = 0;
            if (P.bbits) {  // (the headers of lists are not a bitmap's)
                const int2 bh = P.bhdr[k];
                h = bh.y > 0 ? ((bh.x - (lo >> 5)) << 16) | bh.y : 0;
            }
            S.kwn[wib][lane] = h;
        }
        __syncwarp();
        // rows without a bitmap: short ones one per lane, long ones by the warp
        const int my = lane < cnt && S.kwn[wib][lane] == 0 ? S.kl[wib][lane] : 0;
        if (my > 0 && my <= 32) {
            const int s0 = S.kb[wib][lane];
            unsigned curw = 0xffffffffu, mask = 0u;
            for (int q = s0; q < s0 + my; ++q) {
                const unsigned off = (unsigned)(P.B.col[q] - lo), w = off >> 5;
                if (w != curw) {
                    if (mask) atomicOr(&S.pm[curw].y, mask);
                    curw = w;
                    mask = 0u;
                }
                mask |= 1u << (off & 31);
            }
            if (mask) atomicOr(&S.pm[curw].y, mask);
        }
        unsigned longm = __ballot_sync(kFull, my > 32);
        while (longm) {
            const int i = __ffs(longm) - 1;
            longm &= longm - 1u;
            mark_row<false>(P.B.col, S.kb[wib][i], S.kb[wib][i] + S.kl[wib][i], lo, hi + 1, lane, M);
        }
        for (int i = 0; i < cnt; ++i) {
            const int h = S.kwn[wib][i];
            if (h == 0) continue;
            const int kw = h >> 16, kn = h & 0xffff;
            const int base = S.kb[wib][i] - kw;  // bits[base + w]: window word w
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int w = lane + 32 * u;
                if (w >= kw && w < kw + kn) reg[u] |= P.bbits[base + w];
            }
        }
        __syncwarp();
    }
    if (wib == 0 && lane == 0)
        for (int t = 0; t < nadd; ++t) rf += add[t].rd ? (unsigned long long)rd_nnz(add[t].rd[r]) : 1ull;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int w = lane + 32 * u;
        if (w < kBmWords && reg[u]) atomicOr(&S.pm[w].y, reg[u]);
    }
    __syncthreads();
    // ---- number the columns: thread t takes words 2t and 2t + 1 (in order)
    static_assert(2 * kCtaWarps * 32 >= kBmWords, "two words per thread cover the map");
    int total = 0;
    {
        const int w0 = 2 * tid, w1 = 2 * tid + 1;
        const int c0 = w0 < nw ? __popc(S.pm[w0].y) : 0;
        const int c1 = w1 < nw ? __popc(S.pm[w1].y) : 0;
        const int ex = cta_excl_scan(c0 + c1, tid, S.wcnt, &total);
        if (w0 < nw) S.pm[w0].x = (unsigned)ex;
        if (w1 < nw) S.pm[w1].x = (unsigned)(ex + c0);
    }
    if (total > kCtaCap) {
        // more entries than slots: the first warp computes the row alone
        // (with its own counts; this pass's are dropped), once every thread
        // is done with the map
        __syncthreads();
        if (wib == 0)
            product_row<false, false, true, kBmWords>(P, add, *reinterpret_cast<ProdSmem<false, kBmWords>*>(&S), st,
                                                      r, lane);
        __syncthreads();
        return;
    }
    st.fma += rf;
    if (wib == 0) {
        const long long b = arena_take(st.arena, (unsigned long long)((total + 3) & ~3), P.arena, P.ctl, P.pool_val,
                                       lane);
        if (lane == 0) S.base = b;
    }
    // the column list: each thread fills the two words whose prefixes it wrote
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int w = 2 * tid + k;
        if (w < nw) {
            unsigned bits = S.pm[w].y;
            int idx = (int)S.pm[w].x;
            while (bits) {
                S.colbuf[idx++] = (unsigned short)(w * 32 + __ffs(bits) - 1);
                bits &= bits - 1u;
            }
        }
    }
    for (int i = tid; i < total; i += kT) S.acc[i] = 0.0;
    __syncthreads();
    const long long base = S.base;
    if (base < 0) {
        if (tid == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
        return;
    }
    // ---- numeric pass: the addends, t ascending
    for (int t = 0; t < nadd; ++t) {
        const AddTerm& T = add[t];
        if (!T.rd) {
            if (tid == 0) {
                const int i = slot_lookup(M, r - lo);
                S.acc[i] = __fma_rn(T.alpha, 1.0, S.acc[i]);
            }
        } else {
            const RowDesc d = T.rd[r];
            for (int q = d.rb + tid; q < d.re; q += kT) {
                const int i = slot_lookup(M, P.pool_col[q] - lo);
                S.acc[i] = __fma_rn(T.alpha, P.pool_val[q], S.acc[i]);
            }
        }
        __syncthreads();
    }
    // ---- the B rows, k ascending, a block barrier after each
    const int* bcol = P.B.col;
    const double* bval = P.B.val;
    for (int seg = pa0; seg < pa1; seg += 32) {
        const int cnt = min(32, pa1 - seg);
        __syncthreads();  // every thread is done with the last segment (its last rows may be empty)
        if (wib == 0 && lane < cnt) {
            const int k = P.A.col[seg + lane];
            const int b = P.B.rb[k];
            S.kb[0][lane] = b;
            S.kl[0][lane] = P.B.re[k] - b;
            S.ka[lane] = P.A.val[seg + lane];
        }
        __syncthreads();
        for (int kk = 0; kk < cnt; ++kk) {
            const int len = S.kl[0][kk];
            if (len == 0) continue;
            const double a = S.ka[kk];
            const int* rc = bcol + S.kb[0][kk];
            const double* rv = bval + S.kb[0][kk];
            int off = tid;
            for (; off + 3 * kT < len; off += 4 * kT) {
                int j[4];
                double v[4], x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    j[u] = rc[off + u * kT];
                    v[u] = rv[off + u * kT];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) j[u] = slot_lookup(M, j[u] - lo);
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = S.acc[j[u]];
#pragma unroll
                for (int u = 0; u < 4; ++u) S.acc[j[u]] = __fma_rn(a, v[u], x[u]);
            }
            for (; off < len; off += kT) {
                const int j = slot_lookup(M, rc[off] - lo);
                S.acc[j] = __fma_rn(a, rv[off], S.acc[j]);
            }
            __syncthreads();
        }
    }
    // ---- write-back: warp w takes slots [w Q, (w + 1) Q) in column order
    const int Q = ((total + kCtaWarps - 1) / kCtaWarps + 31) & ~31;
    const int s0 = min(total, wib * Q), s1 = min(total, s0 + Q);
    int mine = 0;
    for (int i0 = s0; i0 < s1; i0 += 32) {
        const int i = i0 + lane;
        mine += __popc(__ballot_sync(kFull, i < s1 && mag_bits(S.acc[i]) != 0ull));
    }
    int written = 0;
    const int before = cta_excl_scan(lane == 0 ? mine : 0, tid, S.wcnt, &written);
    const long long wbase = base + __shfl_sync(kFull, before, 0);
    const bool filt = P.filtering != 0;
    const unsigned long long r_eps = (unsigned long long)__double_as_longlong(P.eps_g);
    int w_off = 0;
    for (int i0 = s0; i0 < s1; i0 += 32) {
        const int i = i0 + lane;
        double x = 0.0;
        int c = 0;
        if (i < s1) {
            x = S.acc[i];
            c = lo + (int)S.colbuf[i];
        }
        const unsigned long long xb = mag_bits(x);
        const bool nz = i < s1 && xb != 0ull;
        const unsigned m = __ballot_sync(kFull, nz);
        const bool cand = nz && filt && xb <= r_eps;
        if (nz) {
            const long long pos = wbase + w_off + __popc(m & lanemask_lt());
            P.pool_col[pos] = c;
            P.pool_val[pos] = x;
            st.absmax = xb > st.absmax ? xb : st.absmax;
            if (cand) {
                exact_add(P.words + c, (size_t)P.n, P.sticky + c, xb, P.e_lsb);
                ++st.cand;
            }
        }
        if (P.cand_col)
            cand_push(st.carena, cand, c, xb, P.cand_col, P.cand_x, &P.ctl->cand_cnt[0], P.cand_cap, P.cand_chunk,
                      &P.ctl->cand_over, lane);
        w_off += __popc(m);
    }
    // the row's unused reserved slots read as exact zeros (never candidates)
    const long long rend = base + ((total + 3) & ~3);
    for (long long q = base + written + tid; q < rend; q += kT) P.pool_val[q] = 0.0;
    __syncthreads();  // the map and the accumulator are free for the next row
    if (tid == 0) {
        write_desc(P, r, stored_row(P, base, written));
        st.written += (unsigned long long)written;
    }
}

__global__ void __launch_bounds__(kCtaWarps * 32, 7) k_product_cta(const __grid_constant__ ProductArgs P) {
    pdl_enter();
    if (P.skip_unless && __ldcg(P.skip_unless) == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AddTerm* add = reinterpret_cast<AddTerm*>(smem_raw);
    CtaSmem& S = *reinterpret_cast<CtaSmem*>(smem_raw + sizeof(AddTerm) * kMaxAdd);
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    for (int t = tid; t < P.nadd; t += blockDim.x) add[t] = P.add[t];
    __syncthreads();
    RowState st;
    for (int r = blockIdx.x; r < P.n; r += gridDim.x) cta_row(P, add, S, st, r, tid);
    if (wib == 0) arena_close(st.arena, P.pool_val, lane);
    if (P.cand_col) cand_close(st.carena, P.cand_x, lane);
    product_done(P);
    st.cand = (unsigned long long)warp_sum((int)st.cand);
    st.absmax = warp_max_u64(st.absmax);
    for (int o = 16; o; o >>= 1) st.fma += __shfl_xor_sync(kFull, st.fma, o);
    st.written = __shfl_sync(kFull, st.written, 0);
    st.span = warp_max(st.span);
    if (lane == 0) {
        if (st.fma) atomicAdd(&P.ctl->fma_total, st.fma);
        if (P.stat) {
            if (st.span > 0) atomicMax(&P.stat->span_max, (unsigned)st.span);
            if (st.fma) atomicAdd(&P.stat->fma, st.fma);
            if (st.written) atomicAdd(&P.stat->nnz_pre, st.written);
            if (st.cand) atomicAdd(&P.stat->ncand, st.cand);
        }
        if (P.absmax_slot && st.absmax) atomicMax(&P.absmax_slot->absmax, st.absmax);
    }
}

// ---------------------------------------------------------------- k_band
// The product step for matrices whose rows span consecutive columns (banded
// and 1D operators, their powers and the filtered sums of those).  Where
// every term of an output row is full (RowDesc) the row is folded output by
// output in registers: no symbolic pass, slot map, shared-memory
// read-modify-write or barrier between B rows.  A tile is R consecutive output
// rows by 64 columns; a lane owns the columns c and c + 32 of the tile's rows.
// The addends are folded in order, then k ascending over the union of the
// rows' ranges of A: B row k's entry of column c is at position c - first, is
// loaded once and folded into every row of the tile that has k
// (acc = fma(a_rk, b_kc, acc)).  Every output's fold is k_product's, in its
// order, and the results are bitwise the same.
//
// Bound by the FP64 pipe: one instruction per (row, k, 32 columns that B row k
// meets).  R = 4 rows share a load, so that loads are a quarter of them (with
// one row per tile the same fold waited on L2: L1 holds 15-40 % of what
// neighbouring rows, in other warps, read again).  Measured against the
// accumulator kernel, whose slot lookups and read-modify-writes it saves:
// banded n = 65536, half-bandwidth 5: Z Z^9 361 -> 200 us, the giant steps
// 470-527 -> 324-423 us (77-81 % of the pipe); banded N(0, 1) n = 20000,
// w = 15: giant steps 2.31-6.22 -> 1.92-4.59 ms (93-98 %).
//
// All instances are held to 72 registers, so that seven blocks fit an SM, and
// spill (bytes of stores / loads, -Xptxas -v): one row a tile 30-34 / 32-40,
// shared by the block 8-30 / 4-28; four rows 106-130 / 184-208, shared 70-94 /
// 100-128; in a batch one row 30-82 / 28-72, four 238-294 / 360-448.  The batch's
// four rows pay for it (launch_band); elsewhere they are faster all the same.
//
// TEAM: the block's four warps share a tile and take its column groups in
// turn (long rows, or few).  A row with a term that is not full, or whose
// range from its first to its last column is longer than its terms together,
// is computed by the accumulator's code (product_row) in the same memory (a
// shared tile's four by a warp each: first evaluation of a band in pieces, n =
// 65536, 25.7 -> 16.8 ms with the lengths bounded by the bandwidth); rows whose
// ranges lie apart are folded one by one.
constexpr int kBandWarps = 4;
using BandMap = ProdSmem<false, kBmWords>;
template <int R, bool TEAM>
struct BandStage {  // terms k of the tile's rows
    static constexpr int kBytes = TEAM ? (int)sizeof(BandMap) * kBandWarps : (int)sizeof(BandMap);
    static constexpr int N = (kBytes / (8 * R + 16)) & ~7;
    int4 d[N];  // {pool position of column 0, first, last column, the tile's rows that have k}
    double a[N][R];
};

// acc[r][u] = fma(a[r], x[u], acc[r][u]) for the rows [R0, R1] and the pieces
// [U0, U1], the columns this lane has (in[u])
template <int R, int U0, int U1, int R0, int R1>
__device__ __forceinline__ void fold_rows(const double* a, const double (&x)[2], const bool (&in)[2],
                                          double (&acc)[R][2]) {
#pragma unroll
    for (int r = R0; r <= R1; ++r) {
        const double ar = a[r];
#pragma unroll
        for (int u = U0; u <= U1; ++u)
            if (in[u]) acc[r][u] = __fma_rn(ar, x[u], acc[r][u]);
    }
}
// ... for the rows that have k (a bit each).  They are chosen by a jump, not
// by an `if` around each: the compiler turns those into predicates, and an
// FP64 instruction holds its pipe for 64 cycles a warp even when no lane takes
// part (a chain with every lane predicated off measured the time of a full
// one).
template <int R, int U0, int U1>
__device__ __forceinline__ void fold_term(int rows, const double* a, const double (&x)[2],
                                          const bool (&in)[2], double (&acc)[R][2]) {
    if constexpr (R == 1) {
        fold_rows<R, U0, U1, 0, 0>(a, x, in, acc);
    } else {
        static_assert(R == 4);
        switch (rows) {
            case 15: fold_rows<R, U0, U1, 0, 3>(a, x, in, acc); break;
            case 1: fold_rows<R, U0, U1, 0, 0>(a, x, in, acc); break;
            case 3: fold_rows<R, U0, U1, 0, 1>(a, x, in, acc); break;
            case 7: fold_rows<R, U0, U1, 0, 2>(a, x, in, acc); break;
            case 8: fold_rows<R, U0, U1, 3, 3>(a, x, in, acc); break;
            case 12: fold_rows<R, U0, U1, 2, 3>(a, x, in, acc); break;
            case 14: fold_rows<R, U0, U1, 1, 3>(a, x, in, acc); break;
            case 2: fold_rows<R, U0, U1, 1, 1>(a, x, in, acc); break;
            case 4: fold_rows<R, U0, U1, 2, 2>(a, x, in, acc); break;
            case 6: fold_rows<R, U0, U1, 1, 2>(a, x, in, acc); break;
            case 0: break;
            default:  // rows with gaps between them
                if (rows & 1) fold_rows<R, U0, U1, 0, 0>(a, x, in, acc);
                if (rows & 2) fold_rows<R, U0, U1, 1, 1>(a, x, in, acc);
                if (rows & 4) fold_rows<R, U0, U1, 2, 2>(a, x, in, acc);
                if (rows & 8) fold_rows<R, U0, U1, 3, 3>(a, x, in, acc);
                break;
        }
    }
}

// The columns gmin + lane + 32 u <= gmax of a group over the staged terms
// [0, nt) in order, the pieces that B row k meets.
template <int R, bool TEAM>
__device__ __forceinline__ void fold_group(const BandStage<R, TEAM>& G, int nt, const double* val,
                                           int gmin, int gmax, int lane, double (&acc)[R][2]) {
    const double* const v = val + gmin + lane;
#pragma unroll 1
    for (int q = 0; q < nt; ++q) {
        const int4 d = G.d[q];
        if (d.y > gmax || d.z < gmin) continue;
        double x[2];
        bool in[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = gmin + lane + 32 * u;
            in[u] = c >= d.y && c <= d.z;
            if (in[u]) x[u] = v[(long long)d.x + 32 * u];
        }
        const double* a = G.a[q];
        switch ((d.y < gmin + 32 ? 1 : 0) | (d.z >= gmin + 32 && gmax >= gmin + 32 ? 2 : 0)) {
            case 3: fold_term<R, 0, 1>(d.w, a, x, in, acc); break;
            case 1: fold_term<R, 0, 0>(d.w, a, x, in, acc); break;
            case 2: fold_term<R, 1, 1>(d.w, a, x, in, acc); break;
            default: break;
        }
    }
}

constexpr int kBandMaxRow = 1 << 20;   // columns of a row folded here
constexpr int kBandMaxWork = 1 << 24;  // and entries of its terms

// (the accumulator that keeps a_rk in shared memory: the wide one reads it from
// global memory before each B row, 8.85 -> 8.62 ms on a first evaluation whose
// rows are mostly in pieces, banded n = 65536)
template <bool BATCH>
__device__ __noinline__ void general_row(const ProductArgs& P, const AddTerm* add, BandMap& S, RowState& st, int r,
                                         int lane) {
    product_row<false, BATCH, false, kBmWords>(P, add, S, st, r, lane);
}

// One row's columns gmin + lane + 32 u within [lo, hi] to pool positions
// base + (column - lo), holes as exact zeros; FILT: Algorithm 1's first pass
// as in k_product.  Returns the true entries.  (The pieces are a loop and not
// two copies: with a copy for each of the tile's rows and pieces the kernel's
// code outgrew its instruction cache.)
template <bool FILT>
__device__ __forceinline__ int write_group(const ProductArgs& P, CandArena& carena, long long base, int lo, int hi,
                                           int gmin, const double (&acc)[2], unsigned long long r_eps, int r_lsb,
                                           int lane, int& cand_n, unsigned long long& absmax) {
    int nnz = 0;
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        if (gmin + 32 * u > hi || gmin + 32 * u + 31 < lo) continue;
        const int c = gmin + 32 * u + lane;
        const bool in = c >= lo && c <= hi;
        const double x = u ? acc[1] : acc[0];
        const unsigned long long xb = mag_bits(x);
        const bool nz = in && xb != 0ull;
        if (in) {
            P.pool_col[base + (c - lo)] = c;
            P.pool_val[base + (c - lo)] = nz ? x : 0.0;
        }
        if (nz && xb > absmax) absmax = xb;
        if constexpr (FILT) {
            const bool cand = nz && xb <= r_eps;  // (r_eps 0: the row is not filtered)
            if (cand) {
                exact_add(P.words + c, (size_t)P.n, P.sticky + c, xb, r_lsb);
                ++cand_n;
            }
            cand_push(carena, cand, c, xb, P.cand_col, P.cand_x, &P.ctl->cand_cnt[0], P.cand_cap, P.cand_chunk,
                      &P.ctl->cand_over, lane);
        }
        nnz += __popc(__ballot_sync(kFull, nz));
    }
    return nnz;
}

// The descriptor of the row written at [base, base + total) with nnz true
// entries: full while at least three quarters of its columns have one, else
// its entries alone (by one warp).
__device__ __forceinline__ void band_desc(const ProductArgs& P, int r, long long base, int total, int lo, int nnz,
                                          int lane) {
    // the row's unused reserved slots read as exact zeros (never candidates)
    if (lane < (-total & 3)) P.pool_val[base + total + lane] = 0.0;
    if (nnz == 0) {
        if (lane == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
    } else if (4ll * nnz >= 3ll * total) {
        if (lane == 0) write_desc(P, r, rd_full_row((int)base, (int)base + total, lo, nnz));
    } else {
        __syncwarp();
        compact_row(P.pool_col, P.pool_val, (int)base, (int)base + total, 0ull, lane);
        __syncwarp();
        if (lane == 0) write_desc(P, r, stored_row(P, base, nnz));
    }
}

template <bool BATCH, bool TEAM, int R, bool FILT>
__global__ void __launch_bounds__(kBandWarps * 32, 7) k_band(const __grid_constant__ ProductArgs P) {
    // (a batch's k_band works beside k_product and waits for it at its end)
    if (BATCH && P.pair) pdl_release();
    else pdl_enter();
    if (P.skip_unless && __ldcg(P.skip_unless) == 0) return;
    using Stage = BandStage<R, TEAM>;
    constexpr int N = Stage::N;
    constexpr int NT = TEAM ? kBandWarps * 32 : 32;  // threads of a tile
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AddTerm* add = reinterpret_cast<AddTerm*>(smem_raw);
    unsigned char* const mem = smem_raw + sizeof(AddTerm) * kMaxAdd;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int tid = TEAM ? (int)threadIdx.x : lane;
    const bool lead = !TEAM || wib == 0;
    BandMap& S = reinterpret_cast<BandMap*>(mem)[TEAM ? 0 : wib];
    Stage& G = *reinterpret_cast<Stage*>(&S);
    __shared__ long long s_base;
    __shared__ int s_lo[R], s_hi[R], s_nnz[R], s_ok;
    __shared__ unsigned s_sum[R];
    __shared__ int s_late;  // the block's rows left to the accumulator
    const int nadd = P.nadd;
    for (int t = threadIdx.x; t < nadd; t += blockDim.x) add[t] = P.add[t];
    if (threadIdx.x == 0) s_late = 0;
    __syncthreads();
    auto sync = [] {
        if constexpr (TEAM) __syncthreads();
        else __syncwarp();
    };
    RowState st;
    // tiles are handed out as warps (blocks) come free: their work differs by
    // an order of magnitude in a batch, and a matrix has a few per warp.  The
    // next one's number is fetched while this one is computed.
    const int tiles = (P.n + R - 1) / R;
    const int first = TEAM ? gridDim.x : gridDim.x * kBandWarps;
    __shared__ int s_next;
    int tile = TEAM ? blockIdx.x : blockIdx.x * kBandWarps + wib;
    while (tile < tiles) {
        int next = 0;
        if (lead && lane == 0) next = first + (int)atomicAdd(&P.ctl->ticket, 1u);
        const int r0 = tile * R;
        // ---- lane i < R: row r0 + i's part of A, and what becomes of it (1:
        // folded here, 2: by the accumulator, 0: done)
        int my_kind = 0, my_inst = 0, my_pa = 0, my_k = 0, my_na = 0;
        bool my_holes = false;
        if (lane < R && r0 + lane < P.n) {
            const int r = r0 + lane;
            my_kind = 1;
            bool prod = P.A.rb != nullptr;
            if constexpr (BATCH) {
                my_inst = P.inst[r];
                if (!P.band[my_inst]) {
                    my_kind = 0;
                } else {
                    const BatchStep& bs = P.bstep[my_inst];
                    if (bs.reuse && __ldcg(P.inst_dropped + my_inst) == 0) {
                        my_kind = 0;  // k_reuse_copy_batch writes it
                    } else if (bs.mode == kBatchSkip || bs.mode == kBatchPass) {
                        if (lead) write_desc(P, r, bs.mode == kBatchPass ? P.B.rd[r] : RowDesc{0, 0, 0, 0});
                        my_kind = 0;
                    }
                    prod = bs.mode == kBatchProduct;
                }
            }
            if (my_kind && prod) {
                my_pa = P.A.rb[r];
                my_na = P.A.re[r] - my_pa;
                if (my_na > 0) {
                    if (P.A.rd) {
                        const RowDesc d = P.A.rd[r];
                        my_k = rd_first(d);
                        my_holes = my_na != rd_nnz(d);
                        if (!rd_full(d)) my_kind = 2;
                    } else {
                        my_k = P.A.col[my_pa];  // (a caller's row: consecutive, checked on input)
                    }
                }
            }
        }
        unsigned todo = __ballot_sync(kFull, my_kind == 1), late = __ballot_sync(kFull, my_kind == 2);
        bool joint = true;
        while (todo) {
            const unsigned m = joint ? todo : todo & (0u - todo);  // rows folded together
            const bool mine = lane < R && ((m >> lane) & 1u);
            const bool many = (m & (m - 1u)) != 0u;
            const int kb = warp_min(mine && my_na > 0 ? my_k : INT_MAX);
            const int ke = max(kb, warp_max(mine && my_na > 0 ? my_k + my_na : 0));
            const int nk = kb == INT_MAX ? 0 : ke - kb;
            if (many && nk > warp_sum(mine ? min(my_na, 1 << 24) : 0) + 32) {
                joint = false;  // ranges of A far apart
                continue;
            }
            // ---- the terms: stage them; the rows' column ranges and work
            int kf[R], kn[R], pa[R];
            unsigned holes = __ballot_sync(kFull, my_holes);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                kf[i] = __shfl_sync(kFull, my_k, i);
                kn[i] = (m >> i) & 1u ? __shfl_sync(kFull, my_na, i) : (__shfl_sync(kFull, my_na, i), 0);
                pa[i] = __shfl_sync(kFull, my_pa, i);
            }
            // (entries of the terms, holes included, saturating at 2^24 a thread;
            // multiply-adds, exact below that)
            int lo[R], hi[R];
            unsigned sum[R], fma[R];
            unsigned bad = 0u;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                lo[i] = INT_MAX;
                hi[i] = -1;
                sum[i] = fma[i] = 0u;
            }
            auto stage = [&](int q0, int q1, bool count) {  // k of [kb + q0, kb + q1)
                for (int q = q0 + tid; q < q1; q += NT) {
                    const int k = kb + q;
                    const RowDesc d = P.B.rd[k];
                    const int f = rd_first(d), len = d.re - d.rb;
                    unsigned rows = 0u;
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int at = k - kf[i];
                        const bool in = (unsigned)at < (unsigned)kn[i];
                        const double a = in ? P.A.val[pa[i] + at] : 0.0;
                        G.a[q - q0][i] = a;
                        if (in && !((holes >> i & 1u) && a == 0.0) && len > 0) {
                            rows |= 1u << i;
                            if (count) {
                                lo[i] = min(lo[i], f);
                                hi[i] = max(hi[i], f + len - 1);
                                sum[i] = min(sum[i] + (unsigned)min(len, kBandMaxWork), (unsigned)kBandMaxWork);
                                fma[i] += (unsigned)rd_nnz(d);
                                if (!rd_full(d)) bad |= 1u << i;
                            }
                        }
                    }
                    G.d[q - q0] = make_int4(d.rb - f, len > 0 ? f : INT_MAX, f + len - 1, (int)rows);
                }
            };
            if constexpr (TEAM) {
                __syncthreads();
                if (threadIdx.x < R) {
                    s_lo[threadIdx.x] = INT_MAX;
                    s_hi[threadIdx.x] = -1;
                    s_sum[threadIdx.x] = s_nnz[threadIdx.x] = 0;
                    if (threadIdx.x == 0) s_ok = 0;
                }
            }
            for (int q0 = 0; q0 < nk; q0 += N) {
                sync();
                stage(q0, min(nk, q0 + N), true);
            }
            if (lead)
                for (int x = lane; x < nadd * R; x += 32) {
                    const int t = x / R, i = x - t * R;
                    if (!((m >> i) & 1u)) continue;
                    if (BATCH && __double_as_longlong(P.alpha_tab[(size_t)t * P.ninst + P.inst[r0 + i]]) == 0ll) continue;
                    int f = r0 + i, l = f, len = 1, nnz = 1;
                    bool full = true;
                    if (add[t].rd) {
                        const RowDesc d = add[t].rd[r0 + i];
                        len = d.re - d.rb;
                        if (len <= 0) continue;
                        f = rd_first(d);
                        l = rd_last(d);
                        nnz = rd_nnz(d);
                        full = rd_full(d);
                    }
#pragma unroll
                    for (int e = 0; e < R; ++e)
                        if (e == i) {
                            lo[e] = min(lo[e], f);
                            hi[e] = max(hi[e], l);
                            sum[e] = min(sum[e] + (unsigned)min(len, kBandMaxWork), (unsigned)kBandMaxWork);
                            fma[e] += (unsigned)nnz;
                            if (!full) bad |= 1u << e;
                        }
                }
            bad = __reduce_or_sync(kFull, bad);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                lo[i] = warp_min(lo[i]);
                hi[i] = warp_max(hi[i]);
                sum[i] = __reduce_add_sync(kFull, sum[i]);
            }
            if constexpr (TEAM) {
                __syncthreads();
                if (lane == 0) {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        atomicMin(&s_lo[i], lo[i]);
                        atomicMax(&s_hi[i], hi[i]);
                        atomicAdd(&s_sum[i], sum[i]);
                    }
                    if (bad) atomicOr(&s_ok, (int)bad);
                }
                __syncthreads();
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    lo[i] = s_lo[i];
                    hi[i] = s_hi[i];
                    sum[i] = s_sum[i];
                }
                bad = (unsigned)s_ok;
            }
            unsigned fold = 0u;
            int glo = INT_MAX, ghi = -1;
            long long width = 0;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (!((m >> i) & 1u) || hi[i] < lo[i]) continue;
                const int total = hi[i] - lo[i] + 1;
                if ((bad >> i & 1u) || total > kBandMaxRow || (unsigned)total > sum[i] || sum[i] >= (unsigned)kBandMaxWork) {
                    bad |= 1u << i;
                    continue;
                }
                fold |= 1u << i;
                glo = min(glo, lo[i]);
                ghi = max(ghi, hi[i]);
                width += total;
            }
            if (many && ghi - glo + 1 > width) {
                joint = false;  // columns far apart
                continue;
            }
            // ---- settled: the empty rows, the accumulator's rows
            int need = 0, at[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                at[i] = need;
                if (!((m >> i) & 1u)) continue;
                if (hi[i] < lo[i]) {
                    if (lead && lane == 0) write_desc(P, r0 + i, RowDesc{0, 0, 0, 0});
                    if constexpr (!BATCH) st.fma += fma[i];
                } else if (bad >> i & 1u) {
                    late |= 1u << i;
                } else {
                    need += (hi[i] - lo[i] + 4) & ~3;
                    if constexpr (!BATCH) st.fma += fma[i];
                    st.span = max(st.span, hi[i] - lo[i] + 1);
                }
            }
            long long base = 0;
            if (fold) {
                if (lead) base = arena_take(st.arena, (unsigned long long)need, P.arena, P.ctl, P.pool_val, lane);
                if constexpr (TEAM) {
                    if (threadIdx.x == 0) s_base = base;
                    __syncthreads();
                    base = s_base;
                }
                if (base < 0) {  // the pool is full (recorded): the phase is run again
                    if (lead && lane < R && (fold >> lane & 1u)) write_desc(P, r0 + lane, RowDesc{0, 0, 0, 0});
                    fold = 0u;
                }
            }
            if (fold) {
                sync();
                int nnz[R], cand[BATCH ? R : 1];
                unsigned long long amax[BATCH ? R : 1];  // per row in a batch, else the thread's totals
                if constexpr (!BATCH) {
                    cand[0] = (int)st.cand;
                    amax[0] = st.absmax;
                }
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    nnz[i] = 0;
                    if constexpr (BATCH) {
                        cand[i] = 0;
                        amax[i] = 0ull;
                    }
                }
                const int groups = (ghi - glo + 64) >> 6;
                for (int g0 = 0; g0 < groups; g0 += TEAM ? kBandWarps : 1) {
                    const int gmin = glo + 64 * (g0 + (TEAM ? wib : 0)), gmax = min(ghi, gmin + 63);
                    double acc[R][2];
#pragma unroll
                    for (int i = 0; i < R; ++i) acc[i][0] = acc[i][1] = 0.0;
                    if (gmin <= gmax) {
                        // the addends, t ascending
                        for (int t = 0; t < nadd; ++t) {
#pragma unroll
                            for (int i = 0; i < R; ++i) {
                                if (!(fold >> i & 1u)) continue;
                                const int r = r0 + i;
                                const double alpha = BATCH ? P.alpha_tab[(size_t)t * P.ninst + __shfl_sync(kFull, my_inst, i)]
                                                           : add[t].alpha;
                                if (BATCH && __double_as_longlong(alpha) == 0ll) continue;
                                if (!add[t].rd) {
#pragma unroll
                                    for (int u = 0; u < 2; ++u)
                                        if (gmin + lane + 32 * u == r) acc[i][u] = __fma_rn(alpha, 1.0, acc[i][u]);
                                    continue;
                                }
                                const RowDesc d = add[t].rd[r];
                                const int f = rd_first(d), l = f + (d.re - d.rb) - 1;
                                if (f > gmax || l < gmin) continue;
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    const int c = gmin + lane + 32 * u;
                                    if (c >= f && c <= l) acc[i][u] = __fma_rn(alpha, P.pool_val[d.rb + (c - f)], acc[i][u]);
                                }
                            }
                        }
                    }
                    // the product, k ascending
                    for (int q0 = 0; q0 < nk; q0 += N) {
                        if (nk > N) {
                            sync();
                            stage(q0, min(nk, q0 + N), false);
                            sync();
                        }
                        if (gmin > gmax) continue;
                        fold_group<R, TEAM>(G, min(nk - q0, N), P.pool_val, gmin, gmax, lane, acc);
                    }
                    if (gmin > gmax) continue;
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if (!(fold >> i & 1u)) continue;
                        unsigned long long r_eps = (unsigned long long)__double_as_longlong(P.eps_g);
                        int r_lsb = P.e_lsb;
                        if constexpr (BATCH && FILT) {
                            const BatchStep& bs = P.bstep[__shfl_sync(kFull, my_inst, i)];
                            r_eps = (unsigned long long)__double_as_longlong(bs.eps_g);
                            r_lsb = bs.e_lsb;
                        }
                        nnz[i] += write_group<FILT>(P, st.carena, base + at[i], lo[i], hi[i], gmin, acc[i], r_eps, r_lsb,
                                                    lane, cand[BATCH ? i : 0], amax[BATCH ? i : 0]);
                    }
                }
                if constexpr (!BATCH) {
                    st.cand = (unsigned long long)cand[0];
                    st.absmax = amax[0];
                }
                if constexpr (TEAM) {
                    if (lane == 0) {
#pragma unroll
                        for (int i = 0; i < R; ++i)
                            if (nnz[i]) atomicAdd(&s_nnz[i], nnz[i]);
                    }
                    __syncthreads();
#pragma unroll
                    for (int i = 0; i < R; ++i) nnz[i] = s_nnz[i];
                }
                if (lead) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if (!(fold >> i & 1u)) continue;
                        band_desc(P, r0 + i, base + at[i], hi[i] - lo[i] + 1, lo[i], nnz[i], lane);
                        if (!BATCH && lane == 0) st.written += (unsigned long long)nnz[i];
                    }
                }
                if constexpr (BATCH) {
                    // lane i adds row i's candidates, entries and largest |x|
                    // to its instance's record
                    int my_cand = 0, my_nnz = 0, my_span = 0;
                    unsigned long long my_max = 0ull;
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int ci = FILT ? warp_sum(cand[i]) : 0;
                        const unsigned long long mi = P.absmax_slot ? warp_max_u64(amax[i]) : 0ull;
                        if (lane == i && (fold >> i & 1u)) {
                            my_cand = ci;
                            my_max = mi;
                            my_nnz = nnz[i];
                            my_span = hi[i] - lo[i] + 1;
                        }
                    }
                    if (my_nnz > 0) {
                        if (P.stat_tab) {
                            StepStat* rec = P.stat_tab + my_inst;
                            atomicAdd(&rec->nnz_pre, (unsigned long long)my_nnz);
                            if (my_cand) atomicAdd(&rec->ncand, (unsigned long long)my_cand);
                            atomicMax(&rec->span_max, (unsigned)my_span);
                        }
                        if (my_max) atomicMax(&(P.absmax_slot + (size_t)my_inst * P.absmax_stride)->absmax, my_max);
                    }
                }
            }
            if constexpr (BATCH) {  // the multiply-adds of the rows settled here
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const unsigned f = __reduce_add_sync(kFull, fma[i]);
                    if (lane == i && ((m & ~bad) >> i & 1u) && f && P.stat_tab)
                        atomicAdd(&P.stat_tab[my_inst].fma, (unsigned long long)f);
                }
            }
            todo &= ~m;
        }
        if (late) {
            sync();
            if (!BATCH && lead && lane == 0) atomicAdd(&s_late, __popc(late));
            // (one by one; a shared tile's row i by warp i)
            BandMap& M = reinterpret_cast<BandMap*>(mem)[wib];
            while (late) {
                const int i = __ffs(late) - 1;
                late &= late - 1u;
                if (TEAM && i != wib) continue;
                general_row<BATCH>(P, add, M, st, r0 + i, lane);
                __syncwarp();
            }
        }
        if constexpr (TEAM) {
            if (threadIdx.x == 0) s_next = next;
            __syncthreads();  // the tile's memory is free
            tile = s_next;
            __syncthreads();
        } else {
            tile = __shfl_sync(kFull, next, 0);
        }
    }
    arena_close(st.arena, P.pool_val, lane);
    if (P.cand_col) cand_close(st.carena, P.cand_x, lane);
    if constexpr (BATCH)
        if (P.pair) pdl_wait();
    product_done(P);
    if constexpr (BATCH) return;
    // ---- the step statistics, once per block
    __shared__ unsigned long long blk_written, blk_cand, blk_absmax, blk_fma;
    __shared__ int blk_span;
    if (threadIdx.x == 0) {
        blk_written = blk_cand = blk_absmax = blk_fma = 0ull;
        blk_span = 0;
    }
    __syncthreads();
    st.cand = (unsigned long long)warp_sum((int)st.cand);
    st.absmax = warp_max_u64(st.absmax);
    st.written = __shfl_sync(kFull, st.written, 0);
    for (int o = 16; o; o >>= 1) st.fma += __shfl_xor_sync(kFull, st.fma, o);
    if (lane == 0) {
        atomicAdd(&blk_fma, st.fma);
        atomicAdd(&blk_written, st.written);
        atomicAdd(&blk_cand, st.cand);
        atomicMax(&blk_absmax, st.absmax);
        atomicMax(&blk_span, st.span);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blk_fma) atomicAdd(&P.ctl->fma_total, blk_fma);
        if (P.stat) {
            if (blk_span > 0) atomicMax(&P.stat->span_max, (unsigned)blk_span);
            if (s_late > 0) atomicAdd(&P.stat->general, (unsigned)s_late);
            if (blk_fma) atomicAdd(&P.stat->fma, blk_fma);
            if (blk_written) atomicAdd(&P.stat->nnz_pre, blk_written);
            if (blk_cand) atomicAdd(&P.stat->ncand, blk_cand);
        }
        if (P.absmax_slot && blk_absmax) atomicMax(&P.absmax_slot->absmax, blk_absmax);
    }
}
size_t band_smem_bytes() { return sizeof(AddTerm) * kMaxAdd + sizeof(BandMap) * kBandWarps; }

// ---------------------------------------------------------------- k_reuse_pass1
// A baby step Z-hat_(k) = filter(Z Z-hat_(k-1)) while no earlier step has
// dropped an entry: Z-hat_(k-1) is then the power Z^(k-1) of the norm phase,
// so the product is that phase's Z^k, entry for entry, and its rows are kept
// as they are.  What the product's write-back would have done remains:
// Algorithm 1's first pass (exact column sums and the candidate list of the
// entries 0 < |x| <= eps_g) and the step statistics.  The power's pool range
// is [mark[k-1], mark[k]).  Does nothing once an entry has been dropped (the
// product kernel then runs instead).

__global__ void __launch_bounds__(256) k_reuse_pass1(ReuseArgs R) {
    pdl_enter();
    if (__ldcg(&R.ctl->dropped) != 0) return;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const unsigned long long eb = (unsigned long long)__double_as_longlong(R.eps_g);
    unsigned long long nnz = 0ull, cand = 0ull;
    CandArena ca;
    for (int r = gw; r < R.n; r += nwarps) {
        const int s = R.rb[r], e = R.re[r];
        for (int q0 = s; q0 < e; q0 += 32) {
            const int q = q0 + lane;
            const bool in = q < e;
            const unsigned long long xb = in ? mag_bits(R.val[q]) : 0ull;
            const int c = in ? R.col[q] : 0;
            const bool is_cand = xb != 0ull && xb <= eb;
            if (is_cand) {
                exact_add_checked(R.words, R.sticky, c, R.n, xb, R.e_lsb, R.ctl);
                ++cand;
            }
            if (xb) ++nnz;
            cand_push(ca, is_cand, c, xb, R.cand_col, R.cand_x, &R.ctl->cand_cnt[0], R.cand_cap, R.cand_chunk,
                      &R.ctl->cand_over, lane);
        }
    }
    cand_close(ca, R.cand_x, lane);
    // the counts go to the step's record once per block: one atomic per warp
    // on the same two words queued behind one another at the launch's end
    __shared__ unsigned long long blk_nnz, blk_cand;
    if (threadIdx.x == 0) {
        blk_nnz = 0ull;
        blk_cand = 0ull;
    }
    __syncthreads();
    nnz = (unsigned long long)warp_sum((int)nnz);
    cand = (unsigned long long)warp_sum((int)cand);
    if (lane == 0) {
        if (nnz) atomicAdd(&blk_nnz, nnz);
        if (cand) atomicAdd(&blk_cand, cand);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blk_nnz) atomicAdd(&R.stat->nnz_pre, blk_nnz);
        if (blk_cand) atomicAdd(&R.stat->ncand, blk_cand);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        R.ctl->cslot[0] = R.ctl->cslot[1] = 0ull;  // (Algorithm 1 starts from 0)
        R.stat->fma = R.fma;
        R.stat->pool_start = R.ctl->mark[R.k - 1];
        R.stat->pool_end = R.ctl->mark[R.k];
    }
}

// ---------------------------------------------------------------- k_reuse_copy_batch
// Batched baby step k for the instances that have dropped no entry so far:
// their Z-hat_(k-1) is the norm phase's Z^(k-1), so the product Z Z-hat_(k-1)
// is that phase's Z^k, entry for entry (the same terms in the same order).
// Each such row is copied from the norm phase's pool (P.power) into the
// step's own pool range, and what the product's write-back does besides is
// done on the way: Algorithm 1's first pass (column sums and candidate list
// of the entries 0 < |x| <= eps_g) and the row statistics, with the
// product's multiply-add count (the B row lengths summed over row r of A).
// The product kernel skips these rows.
__global__ void __launch_bounds__(256) k_reuse_copy_batch(ProductArgs P) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    Arena arena;
    CandArena carena;
    for (int r = gw; r < P.n; r += nwarps) {
        const int i = P.inst[r];
        const BatchStep bs = P.bstep[i];
        if (!bs.reuse || __ldcg(P.inst_dropped + i) != 0) continue;
        unsigned long long fma = 0ull;
        const int pa0 = P.A.rb[r], pa1 = P.A.re[r];
        const bool a_holes = pa1 - pa0 != rd_nnz(P.A.rd[r]);
        for (int p = pa0 + lane; p < pa1; p += 32)
            if (!(a_holes && P.A.val[p] == 0.0)) fma += (unsigned long long)rd_nnz(P.B.rd[P.A.col[p]]);
        const int s = P.power.rb[r], len = P.power.re[r] - s;
        if (len <= 0) {
            if (lane == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
            row_stats_batch(P, i, fma, 0ull, 0, 0ull, lane);
            continue;
        }
        const unsigned long long span = ((unsigned long long)len + 3ull) & ~3ull;
        const long long base = arena_take(arena, span, P.arena, P.ctl, P.pool_val, lane);
        if (base < 0) {
            if (lane == 0) write_desc(P, r, RowDesc{0, 0, 0, 0});
            continue;
        }
        const bool filt = bs.eps_g > 0.0;
        const unsigned long long eb = (unsigned long long)__double_as_longlong(bs.eps_g);
        unsigned long long cand = 0ull;
        for (int q0 = 0; q0 < len; q0 += 32) {
            const int q = q0 + lane;
            const bool in = q < len;
            const double x = in ? P.power.val[s + q] : 0.0;
            const int c = in ? P.power.col[s + q] : 0;
            const unsigned long long xb = mag_bits(x);
            const bool is_cand = filt && xb != 0ull && xb <= eb;
            if (in) {
                P.pool_col[base + q] = c;
                P.pool_val[base + q] = x;
            }
            if (is_cand) {
                exact_add(P.words + c, (size_t)P.n, P.sticky + c, xb, bs.e_lsb);
                ++cand;
            }
            if (P.cand_col)
                cand_push(carena, is_cand, c, xb, P.cand_col, P.cand_x, &P.ctl->cand_cnt[0], P.cand_cap, P.cand_chunk,
                          &P.ctl->cand_over, lane);
        }
        for (long long q = base + len + lane; q < base + (long long)span; q += 32) P.pool_val[q] = 0.0;
        RowDesc d = P.power.rd[r];
        d.rb = (int)base;
        d.re = (int)(base + len);
        if (lane == 0) write_desc(P, r, d);
        row_stats_batch(P, i, fma, cand, rd_nnz(d), 0ull, lane);
    }
    arena_close(arena, P.pool_val, lane);
    if (P.cand_col) cand_close(carena, P.cand_x, lane);
    step_done(P.ctl, 0, nullptr, nullptr, nullptr, 0);
}

// ---------------------------------------------------------------- k_alg1
// Passes 2, 3, ... of Algorithm 1 and the compaction, as one cooperative
// launch.  On entry the column sums of pass 1 (entries |x| <= eps_g) are in
// the chunk words and both cslot words are 0.  Every block evaluates the same
// scalar recurrence from the same global values, so all blocks take the same
// decisions without further communication.  Bound by the latency of a pass
// (finalize: eight words a column; the list; a barrier after each), not by
// bytes or instructions, up to a few hundred thousand candidates: with the
// barrier's one atomic per block (it was two, and sleeps between polls)
// cos of banded N(0, 1), n = 1000, w = 8, took 1153 us before and 1048 after.
constexpr int kAlg1Threads = 1024;  // one block per SM: few grid-barrier arrivals
constexpr int kAlg1BlocksPerSm = 1;
// Small steps run as one cluster of 16 blocks: the passes of a step are two
// barriers each, and the cluster's cost less than the grid's, which is most
// of the time while the candidates are few.  Measured as whole evaluations
// (us, grid / cluster): 1D n = 256 445 / 430, n = 2000 (50 k entries a step)
// 520 / 505, 16 x 16 grid (51 k) 910 / 853, banded n = 1000 (74 k) 675 / 655;
// n = 2000 (148 k) 744 / 769, 32 x 32 grid (318 k) 996 / 995, 48 x 48 (808 k)
// 1188 / 1279: the line lies at 100 k entries.
constexpr int kClusterColumns = 4096;
constexpr double kClusterEntries = 1e5;

template <bool CLUSTER>
__device__ __forceinline__ bool alg1_barrier(const Alg1Args& A) {
    if constexpr (CLUSTER) {
        cluster_barrier();
        return true;
    }
    return grid_barrier(A.ctl, A.budget_ns);
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kAlg1Threads, kAlg1BlocksPerSm) k_alg1(Alg1Args A) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int nthreads = gridDim.x * blockDim.x;
    const size_t n = (size_t)A.n;
    __shared__ unsigned long long red[kAlg1Threads / 32];

    double eps_f = A.eps_g, c = 0.0;
    int it = 0;
    bool alive = true;
    // the step's pool range; the counter runs past the capacity on overflow
    const unsigned long long p0 = min(__ldcg(&A.stat->pool_start), A.ctl->pool_cap);
    const unsigned long long pe = __ldcg(&A.stat->pool_end);
    const unsigned long long p1 = min(pe ? pe : __ldcg(&A.ctl->pool_used), A.ctl->pool_cap);
    // a phase whose pool overflowed is discarded: its pool range is not
    // complete, so there is nothing to filter (every block reads the same
    // status, set by an earlier launch)
    if (__ldcg(&A.ctl->status) & kDevPoolFull) return;
    bool over = __ldcg(&A.ctl->cand_over) != 0 || A.cand_col == nullptr;
    const unsigned long long ccap = A.ctl->cand_cap;
    const unsigned cchunk = A.ctl->cand_chunk;
    const unsigned long long split = far_split(A.eps_g, A.far_shift);
    if (__ldcg(&A.stat->ncand) == 0ull) {
        // the product left no entry with |x| <= eps_g: the first pass finds an
        // empty candidate matrix (c = 0), nothing is dropped
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            A.stat->eps_f = eps_f;
            A.stat->iters = 1;
            A.stat->dropped = 0.0;
            A.stat->nnz_post = A.stat->nnz_pre;
        }
        return;
    }
    bool dirty = false;  // the column sums were left in place by the last finalize
    for (;;) {
        // finalize: round each column sum, take the max.  The sums are kept
        // for an incremental (list) pass and cleared for a full pool scan.
        unsigned long long local = 0ull;
        dirty = !over;
        for (int j = gt; j < A.n; j += nthreads) {
            double s = chunk_round(A.words + j, n, A.sticky + j, A.e_lsb, over);
            unsigned long long sb = (unsigned long long)__double_as_longlong(s);
            local = sb > local ? sb : local;
        }
        local = warp_max_u64(local);
        if (lane == 0) red[threadIdx.x >> 5] = local;
        __syncthreads();
        if (threadIdx.x < 32) {
            unsigned long long v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0ull;
            v = warp_max_u64(v);
            if (threadIdx.x == 0) {
                if (v) atomicMax(&A.ctl->cslot[it & 1], v);
                if (blockIdx.x == 0) {
                    A.ctl->cslot[(it + 1) & 1] = 0ull;
                    if (it == 0) A.ctl->cand_cnt[1] = 0ull;  // the first rescan's output list
                }
            }
        }
        if (!alg1_barrier<CLUSTER>(A)) {
            alive = false;
            break;
        }
        c = __longlong_as_double((long long)__ldcg(&A.ctl->cslot[it & 1]));
        double m = c / eps_f;
        ++it;
        if (!(c > A.bound)) break;
        if (it >= A.maxit) {
            if (gt == 0) atomicOr(&A.ctl->status, kDevNotConv);
            break;
        }
        eps_f = A.eps_g / m;
        const unsigned long long fb = (unsigned long long)__double_as_longlong(eps_f);
        if (!over) {
            // The first rescan reads the product's candidates (list 0) and
            // writes those still at or below eps_f to list 1: the near ones
            // (above eps_g / 2^far_shift, default 2^6) to its front half, the
            // far ones to its back half.  The far ones cannot leave while
            // eps_f stays above that bound; later rescans read the near
            // ones in place, subtracting and clearing (|x| = 0: a hole) those
            // that leave, and read the far half (in place) only once eps_f
            // falls below the bound.
            const bool first = it == 1;
            const unsigned long long half = ccap / 2;
            int* fcol = A.cand_col + ccap + half;
            unsigned long long* fx = A.cand_x + ccap + half;
            const unsigned long long nt = (unsigned long long)nthreads;
            if (!first) {
                const unsigned long long cnt = min(__ldcg(&A.ctl->cand_cnt[1]), half);
                const int* ic = A.cand_col + ccap;
                unsigned long long* ix = A.cand_x + ccap;
                for (unsigned long long q0 = (unsigned long long)gt; q0 < cnt; q0 += 4ull * nt) {
                    unsigned long long xb[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const unsigned long long q = q0 + (unsigned long long)u * nt;
                        xb[u] = q < cnt ? __ldcg(ix + q) : 0ull;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (xb[u] > fb) {  // 0 (a hole) never
                            const unsigned long long q = q0 + (unsigned long long)u * nt;
                            exact_sub_checked(A.words, A.sticky, __ldcg(ic + q), A.n, xb[u], A.e_lsb, A.ctl);
                            ix[q] = 0ull;
                        }
                    }
                }
            }
            const unsigned long long cnt = first ? min(__ldcg(&A.ctl->cand_cnt[0]), ccap) : 0ull;
            const int* ic = A.cand_col;
            const unsigned long long* ix = A.cand_x;
            const int bo = 1;
            CandArena ca, cf;
            // four candidates per thread at a time, all loads issued first
            for (unsigned long long q0 = (unsigned long long)(gt & ~31); q0 < cnt; q0 += 4ull * nt) {
                unsigned long long xb[4];
                int col[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long q = q0 + (unsigned long long)u * nt + (unsigned long long)lane;
                    xb[u] = q < cnt ? __ldcg(ix + q) : 0ull;
                    col[u] = q < cnt ? __ldcg(ic + q) : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool keep = xb[u] != 0ull && xb[u] <= fb;
                    // an entry that leaves the list leaves the column sums
                    if (xb[u] != 0ull && !keep)
                        exact_sub_checked(A.words, A.sticky, col[u], A.n, xb[u], A.e_lsb, A.ctl);
                    const bool far = first && keep && xb[u] <= split;
                    cand_push(ca, keep && !far, col[u], xb[u], A.cand_col + (size_t)bo * ccap,
                              A.cand_x + (size_t)bo * ccap, &A.ctl->cand_cnt[bo], half, cchunk, &A.ctl->cand_over,
                              lane);
                    if (first)
                        cand_push(cf, far, col[u], xb[u], fcol, fx, &A.ctl->cand_far, half, cchunk, &A.ctl->cand_over,
                                  lane);
                }
            }
            cand_close(ca, A.cand_x + (size_t)bo * ccap, lane);
            if (first) cand_close(cf, fx, lane);
            if (!first && fb < split) {
                // eps_f is below the far candidates' bound: those above it leave
                const unsigned long long nf = min(__ldcg(&A.ctl->cand_far), half);
                for (unsigned long long q = (unsigned long long)gt; q < nf; q += nt) {
                    const unsigned long long xb = __ldcg(fx + q);
                    if (xb > fb) {
                        exact_sub_checked(A.words, A.sticky, __ldcg(fcol + q), A.n, xb, A.e_lsb, A.ctl);
                        fx[q] = 0ull;
                    }
                }
            }
            if (!alg1_barrier<CLUSTER>(A)) {
                alive = false;
                break;
            }
            // a list that overflowed is incomplete: scan the pool from now on
            // (the flag is read after the barrier, so every block agrees)
            over = __ldcg(&A.ctl->cand_over) != 0;
            continue;
        }
        // accumulate the entries still below the threshold: one streaming
        // pass over the step's pool range (its gaps hold exact zeros)
        for (unsigned long long q0 = p0 + (unsigned long long)gt; q0 < p1; q0 += 4ull * nthreads) {
            unsigned long long xb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long q = q0 + (unsigned long long)u * nthreads;
                xb[u] = q < p1 ? mag_bits(__ldcg(A.val + q)) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (xb[u] != 0ull && xb[u] <= fb) {
                    const int col = A.col[q0 + (unsigned long long)u * nthreads];
                    exact_add_checked(A.words, A.sticky, col, A.n, xb[u], A.e_lsb, A.ctl);
                }
            }
        }
        if (!alg1_barrier<CLUSTER>(A)) {
            alive = false;
            break;
        }
    }
    if (!alive) return;
    if (gt == 0) {  // the lists are empty for the next step
        A.ctl->cand_cnt[0] = A.ctl->cand_cnt[1] = A.ctl->cand_far = 0ull;
        A.ctl->cand_over = 0;
    }
    if (dirty) clear_sums(A.words, A.sticky, A.n, gt, nthreads);  // zero for the next step
    if (!sum_is_exact(c, A.e_lsb)) {
        // every candidate is tiny against eps_g and c may have lost bits
        // below the LSB: count the final candidates again with the LSB of
        // the largest one.  cslot[it & 1] is 0 (cleared by the last
        // finalize), cslot[(it - 1) & 1] holds the c every block has read
        // once all blocks reach the first barrier.
        const unsigned long long fb = (unsigned long long)__double_as_longlong(eps_f);
        const int sx = it & 1, sc = (it - 1) & 1;
        if (!alg1_barrier<CLUSTER>(A)) return;
        if (gt == 0) A.ctl->cslot[sc] = 0ull;
        unsigned long long mx = 0ull;
        for (unsigned long long q = p0 + (unsigned long long)gt; q < p1; q += (unsigned long long)nthreads) {
            const unsigned long long xb = mag_bits(__ldcg(A.val + q));
            if (xb <= fb && xb > mx) mx = xb;
        }
        mx = warp_max_u64(mx);
        if (lane == 0 && mx) atomicMax(&A.ctl->cslot[sx], mx);
        if (!alg1_barrier<CLUSTER>(A)) return;
        const int lsb = lsb_for_bound(__ldcg(&A.ctl->cslot[sx]));
        for (unsigned long long q = p0 + (unsigned long long)gt; q < p1; q += (unsigned long long)nthreads) {
            const unsigned long long xb = mag_bits(__ldcg(A.val + q));
            if (xb != 0ull && xb <= fb) exact_add_checked(A.words, A.sticky, A.col[q], A.n, xb, lsb, A.ctl);
        }
        if (!alg1_barrier<CLUSTER>(A)) return;
        unsigned long long local = 0ull;
        for (int j = gt; j < A.n; j += nthreads) {
            const double s = chunk_round(A.words + j, n, A.sticky + j, lsb, true);
            const unsigned long long sb = (unsigned long long)__double_as_longlong(s);
            local = sb > local ? sb : local;
        }
        local = warp_max_u64(local);
        if (lane == 0 && local) atomicMax(&A.ctl->cslot[sc], local);
        if (!alg1_barrier<CLUSTER>(A)) return;
        c = __longlong_as_double((long long)__ldcg(&A.ctl->cslot[sc]));
    }
    if (!(c > 0.0)) {
        // nothing was dropped: the matrix stays as the product wrote it
        if (gt == 0) {
            A.stat->eps_f = eps_f;
            A.stat->iters = it;
            A.stat->dropped = c;
            A.stat->nnz_post = __ldcg(&A.stat->nnz_pre);
        }
        return;
    }

    if (gt == 0) A.ctl->dropped = 1;
    // compaction: keep |x| > eps_f, in place, column order preserved
    const unsigned long long fb = (unsigned long long)__double_as_longlong(eps_f);
    unsigned long long kept = 0ull;
    for (int r = gw; r < A.n; r += nwarps) {
        const int k = filter_row(A.col, A.val, A.rb, A.re, A.rd, r, fb, lane);
        if (lane == 0) kept += (unsigned long long)k;
    }
    if (lane == 0 && kept) atomicAdd(&A.stat->nnz_post, kept);
    if (gt == 0) {
        A.stat->eps_f = eps_f;
        A.stat->iters = it;
        A.stat->dropped = c;
    }
}

// ---------------------------------------------------------------- k_alg1_batch
// Algorithm 1 for every filtered instance of a batched step, one cooperative
// launch.  The instances run the recurrence of k_alg1 side by side: column
// sums belong to the instance owning the column, each instance has its own
// c, eps_f and pass count, and a pass streams the step's whole pool range
// once for all instances still iterating.  Every block keeps the per-instance
// state in shared memory and updates it from the same global column-sum
// maxima, so all blocks take the same decisions.
constexpr int kMaxBatch = 1024;  // instances of one batched launch

__global__ void __launch_bounds__(kAlg1Threads, kAlg1BlocksPerSm) k_alg1_batch(Alg1BatchArgs A) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int nthreads = gridDim.x * blockDim.x;
    const size_t n = (size_t)A.n;
    __shared__ double s_eps[kMaxBatch];  // eps_f
    __shared__ double s_c[kMaxBatch];    // last column-sum maximum c
    __shared__ int s_it[kMaxBatch];
    // 0 iterating, 1 finished, 2 not filtered here, 3 finished without
    // candidates, 4 finished with a c to count again (see below)
    __shared__ unsigned char s_state[kMaxBatch];
    __shared__ int s_left;
    if (__ldcg(&A.ctl->status) & kDevPoolFull) return;  // discarded phase (same for all blocks)
    if (threadIdx.x == 0) s_left = 0;
    __syncthreads();
    int left = 0;
    for (int i = threadIdx.x; i < A.ninst; i += blockDim.x) {
        const BatchStep bs = A.bstep[i];
        const bool filt = (bs.mode == kBatchProduct || bs.mode == kBatchAddOnly) && bs.eps_g > 0.0;
        s_eps[i] = bs.eps_g;
        s_c[i] = 0.0;
        s_it[i] = 0;
        // an instance without candidates finds c = 0 in its first pass
        const bool empty = filt && __ldcg(&A.stat_tab[i].ncand) == 0ull;
        s_state[i] = !filt ? 2 : (empty ? 3 : 0);
        if (empty) s_it[i] = 1;
        left += (filt && !empty) ? 1 : 0;
    }
    atomicAdd(&s_left, left);
    __syncthreads();
    const unsigned long long cap = A.ctl->pool_cap;
    const unsigned long long p0 = min(__ldcg(A.pool_start), cap);
    const unsigned long long p1 = min(__ldcg(&A.ctl->pool_used), cap);
    bool over = __ldcg(&A.ctl->cand_over) != 0 || A.cand_col == nullptr;
    const unsigned long long ccap = A.ctl->cand_cap;
    const unsigned cchunk = A.ctl->cand_chunk;
    bool alive = true;
    bool dirty = false;  // some column sums were left in place
    int pass = 0;
    while (s_left > 0) {
        // finalize the column sums of the iterating instances (kept for an
        // incremental list pass, cleared for a full pool scan)
        if (!over) dirty = true;
        for (int j = gt; j < A.n; j += nthreads) {
            const int i = A.inst[j];
            if (s_state[i] != 0) continue;
            double v = chunk_round(A.words + j, n, A.sticky + j, A.bstep[i].e_lsb, over);
            unsigned long long vb = (unsigned long long)__double_as_longlong(v);
            if (vb) atomicMax(&A.cslot[2 * i + (pass & 1)], vb);
        }
        if (blockIdx.x == 0) {
            for (int i = threadIdx.x; i < A.ninst; i += blockDim.x) A.cslot[2 * i + ((pass + 1) & 1)] = 0ull;
            if (threadIdx.x == 0 && pass == 0) A.ctl->cand_cnt[1] = 0ull;  // the first rescan's output list
        }
        if (!grid_barrier(A.ctl, A.budget_ns)) {
            alive = false;
            break;
        }
        // the recurrence of every iterating instance (identical in all blocks)
        __syncthreads();
        if (threadIdx.x == 0) s_left = 0;
        __syncthreads();
        left = 0;
        for (int i = threadIdx.x; i < A.ninst; i += blockDim.x) {
            if (s_state[i] != 0) continue;
            const BatchStep bs = A.bstep[i];
            const double c = __longlong_as_double((long long)__ldcg(&A.cslot[2 * i + (pass & 1)]));
            const double m = c / s_eps[i];
            const int it = ++s_it[i];
            s_c[i] = c;
            if (!(c > bs.bound)) {
                s_state[i] = 1;
            } else if (it >= bs.maxit) {
                s_state[i] = 1;
                if (blockIdx.x == 0) atomicOr(&A.ctl->status, kDevNotConv);
            } else {
                s_eps[i] = bs.eps_g / m;
                ++left;
            }
        }
        atomicAdd(&s_left, left);
        __syncthreads();
        if (s_left == 0) break;
        if (!over) {
            // the first rescan reads the product's candidates (list 0) into
            // list 1, each instance's candidates at or below its eps_g /
            // 2^far_shift in its back half; later rescans read the front half
            // in place (as in k_alg1), clearing the entries that leave and
            // those of instances that have finished
            const bool first = pass == 0;
            const unsigned long long half = ccap / 2;
            int* fcol = A.cand_col + ccap + half;
            unsigned long long* fx = A.cand_x + ccap + half;
            const unsigned long long nt = (unsigned long long)nthreads;
            if (!first) {
                const unsigned long long cnt = min(__ldcg(&A.ctl->cand_cnt[1]), half);
                const int* ic = A.cand_col + ccap;
                unsigned long long* ix = A.cand_x + ccap;
                for (unsigned long long q0 = (unsigned long long)gt; q0 < cnt; q0 += 4ull * nt) {
                    unsigned long long xb[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const unsigned long long q = q0 + (unsigned long long)u * nt;
                        xb[u] = q < cnt ? __ldcg(ix + q) : 0ull;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (!xb[u]) continue;
                        const unsigned long long q = q0 + (unsigned long long)u * nt;
                        const int cq = __ldcg(ic + q);
                        if ((unsigned)cq >= (unsigned)A.n) {
                            atomicOr(&A.ctl->status, kDevInternal);
                            continue;
                        }
                        const int i = A.inst[cq];
                        if (s_state[i] != 0) {
                            ix[q] = 0ull;
                        } else if (xb[u] > (unsigned long long)__double_as_longlong(s_eps[i])) {
                            // an entry that leaves the list leaves the column sums
                            exact_sub(A.words + cq, n, A.sticky + cq, xb[u], A.bstep[i].e_lsb);
                            ix[q] = 0ull;
                        }
                    }
                }
            }
            const unsigned long long cnt = first ? min(__ldcg(&A.ctl->cand_cnt[0]), ccap) : 0ull;
            const int* ic = A.cand_col;
            const unsigned long long* ix = A.cand_x;
            const int bo = 1;
            CandArena ca, cf;
            // four candidates per thread at a time, all loads issued first
            for (unsigned long long q0 = (unsigned long long)(gt & ~31); q0 < cnt; q0 += 4ull * nt) {
                unsigned long long xb[4];
                int col[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long q = q0 + (unsigned long long)u * nt + (unsigned long long)lane;
                    xb[u] = q < cnt ? __ldcg(ix + q) : 0ull;
                    col[u] = q < cnt ? __ldcg(ic + q) : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    bool keep = false, far = false;
                    if (xb[u]) {
                        if ((unsigned)col[u] >= (unsigned)A.n) {
                            atomicOr(&A.ctl->status, kDevInternal);
                        } else {
                            const int i = A.inst[col[u]];
                            if (s_state[i] == 0) {
                                keep = xb[u] <= (unsigned long long)__double_as_longlong(s_eps[i]);
                                // an entry that leaves the list leaves the column sums
                                if (!keep) exact_sub(A.words + col[u], n, A.sticky + col[u], xb[u], A.bstep[i].e_lsb);
                                far = first && keep && xb[u] <= far_split(A.bstep[i].eps_g, A.far_shift);
                            }
                        }
                    }
                    cand_push(ca, keep && !far, col[u], xb[u], A.cand_col + (size_t)bo * ccap,
                              A.cand_x + (size_t)bo * ccap, &A.ctl->cand_cnt[bo], half, cchunk, &A.ctl->cand_over,
                              lane);
                    if (first)
                        cand_push(cf, far, col[u], xb[u], fcol, fx, &A.ctl->cand_far, half, cchunk, &A.ctl->cand_over,
                                  lane);
                }
            }
            cand_close(ca, A.cand_x + (size_t)bo * ccap, lane);
            if (first) cand_close(cf, fx, lane);
            // an instance whose eps_f fell below its far bound: its far
            // candidates above eps_f leave, in place (the same test in all blocks)
            int below = 0;
            if (!first)
                for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
                    if (s_state[i] == 0 &&
                        (unsigned long long)__double_as_longlong(s_eps[i]) < far_split(A.bstep[i].eps_g, A.far_shift))
                        below = 1;
            if (__syncthreads_or(below)) {
                const unsigned long long nf = min(__ldcg(&A.ctl->cand_far), half);
                for (unsigned long long q = (unsigned long long)gt; q < nf; q += nt) {
                    const unsigned long long xq = __ldcg(fx + q);
                    if (xq == 0ull) continue;
                    const int cq = __ldcg(fcol + q);
                    if ((unsigned)cq >= (unsigned)A.n) continue;
                    const int i = A.inst[cq];
                    if (s_state[i] == 0 && xq > (unsigned long long)__double_as_longlong(s_eps[i])) {
                        exact_sub(A.words + cq, n, A.sticky + cq, xq, A.bstep[i].e_lsb);
                        fx[q] = 0ull;
                    }
                }
            }
            if (!grid_barrier(A.ctl, A.budget_ns)) {
                alive = false;
                break;
            }
            over = __ldcg(&A.ctl->cand_over) != 0;  // read after the barrier: every block agrees
            ++pass;
            continue;
        }
        // accumulate the entries still below their instance's threshold
        for (unsigned long long q0 = p0 + (unsigned long long)gt; q0 < p1; q0 += 4ull * nthreads) {
            unsigned long long xb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long q = q0 + (unsigned long long)u * nthreads;
                xb[u] = q < p1 ? mag_bits(__ldcg(A.val + q)) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (xb[u] == 0ull) continue;
                const int col = A.col[q0 + (unsigned long long)u * nthreads];
                if ((unsigned)col >= (unsigned)A.n) {
                    atomicOr(&A.ctl->status, kDevInternal);
                    continue;
                }
                const int i = A.inst[col];
                if (s_state[i] != 0) continue;
                if (xb[u] <= (unsigned long long)__double_as_longlong(s_eps[i]))
                    exact_add(A.words + col, n, A.sticky + col, xb[u], A.bstep[i].e_lsb);
            }
        }
        if (!grid_barrier(A.ctl, A.budget_ns)) {
            alive = false;
            break;
        }
        ++pass;
    }
    if (!alive) return;
    if (gt == 0) {  // the lists are empty for the next step
        A.ctl->cand_cnt[0] = A.ctl->cand_cnt[1] = A.ctl->cand_far = 0ull;
        A.ctl->cand_over = 0;
    }
    if (dirty) clear_sums(A.words, A.sticky, A.n, gt, nthreads);  // zero for the next step
    // an instance whose candidates are all tiny against its eps_g may have
    // lost bits of c below the LSB: its final candidates are counted again
    // with the LSB of its largest one (the same instances in every block)
    int nfix = 0;
    for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
        if (s_state[i] == 1 && !sum_is_exact(s_c[i], A.bstep[i].e_lsb)) {
            s_state[i] = 4;
            ++nfix;
        }
    if (__syncthreads_or(nfix)) {
        __shared__ int s_lsb[kMaxBatch];
        // every block has read the maxima: slot 2i takes the largest
        // candidate, slot 2i + 1 the new c
        if (!grid_barrier(A.ctl, A.budget_ns)) return;
        if (blockIdx.x == 0)
            for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
                if (s_state[i] == 4) A.cslot[2 * i] = A.cslot[2 * i + 1] = 0ull;
        if (!grid_barrier(A.ctl, A.budget_ns)) return;
        for (unsigned long long q = p0 + (unsigned long long)gt; q < p1; q += (unsigned long long)nthreads) {
            const unsigned long long xb = mag_bits(__ldcg(A.val + q));
            if (xb == 0ull) continue;
            const int col = A.col[q];
            if ((unsigned)col >= (unsigned)A.n) continue;
            const int i = A.inst[col];
            if (s_state[i] == 4 && xb <= (unsigned long long)__double_as_longlong(s_eps[i]))
                atomicMax(&A.cslot[2 * i], xb);
        }
        if (!grid_barrier(A.ctl, A.budget_ns)) return;
        for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
            if (s_state[i] == 4) s_lsb[i] = lsb_for_bound(__ldcg(&A.cslot[2 * i]));
        __syncthreads();
        for (unsigned long long q = p0 + (unsigned long long)gt; q < p1; q += (unsigned long long)nthreads) {
            const unsigned long long xb = mag_bits(__ldcg(A.val + q));
            if (xb == 0ull) continue;
            const int col = A.col[q];
            if ((unsigned)col >= (unsigned)A.n) continue;
            const int i = A.inst[col];
            if (s_state[i] == 4 && xb <= (unsigned long long)__double_as_longlong(s_eps[i]))
                exact_add(A.words + col, n, A.sticky + col, xb, s_lsb[i]);
        }
        if (!grid_barrier(A.ctl, A.budget_ns)) return;
        for (int j = gt; j < A.n; j += nthreads) {
            const int i = A.inst[j];
            if (s_state[i] != 4) continue;
            const double v = chunk_round(A.words + j, n, A.sticky + j, s_lsb[i], true);
            const unsigned long long vb = (unsigned long long)__double_as_longlong(v);
            if (vb) atomicMax(&A.cslot[2 * i + 1], vb);
        }
        if (!grid_barrier(A.ctl, A.budget_ns)) return;
        for (int i = threadIdx.x; i < A.ninst; i += blockDim.x)
            if (s_state[i] == 4) {
                s_c[i] = __longlong_as_double((long long)__ldcg(&A.cslot[2 * i + 1]));
                s_state[i] = 1;
            }
        __syncthreads();
    }
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < A.ninst; i += blockDim.x) {
            if (s_state[i] == 2) continue;
            A.stat_tab[i].eps_f = s_eps[i];
            A.stat_tab[i].iters = s_it[i];
            A.stat_tab[i].dropped = s_c[i];
            if (!(s_c[i] > 0.0)) A.stat_tab[i].nnz_post = __ldcg(&A.stat_tab[i].nnz_pre);  // nothing dropped
            else if (A.inst_dropped) A.inst_dropped[i] = 1;
        }
    // compaction of the instances that dropped entries: keep |x| > eps_f of
    // the row's instance, in place
    for (int r = gw; r < A.n; r += nwarps) {
        const int i = A.inst[r];
        if (s_state[i] != 1 || !(s_c[i] > 0.0)) continue;
        const unsigned long long fb = (unsigned long long)__double_as_longlong(s_eps[i]);
        const int k = filter_row(A.col, A.val, A.rb, A.re, A.rd, r, fb, lane);
        if (lane == 0 && k) atomicAdd(&A.stat_tab[i].nnz_post, (unsigned long long)k);
    }
}

// ---------------------------------------------------------------- k_norms
// Exact ||M||_1 of up to kMaxNorms matrices whose max |x| is already in
// slots[i].absmax: accumulate every |x| into per-column fixed-point sums,
// barrier, round and take the maximum into slots[i].result.
constexpr int kNormThreads = 256;

__global__ void __launch_bounds__(kNormThreads) k_norms(NormArgs A) {
    pdl_enter();
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int nthreads = gridDim.x * blockDim.x;
    const size_t n = (size_t)A.n;
    // a phase whose pool overflowed is discarded, and a caller's matrix that
    // failed its check is not read: only the check has bounded its entry count
    // (all blocks read the same status, set by an earlier launch)
    if (__ldcg(&A.ctl->status) & (kDevPoolFull | kDevBadInput)) return;
    // every |x| of every matrix into per-column fixed-point sums: streaming
    // passes over the matrices' pool ranges
    for (int mi = 0; mi < A.count; ++mi) {
        // the counter keeps counting past the capacity when the pool overflows
        const unsigned long long cap = A.ctl->pool_cap;
        const unsigned long long p0 = min(__ldcg(&A.ctl->mark[mi]), cap);
        const unsigned long long p1 = min(__ldcg(&A.ctl->mark[mi + 1]), cap);
        unsigned long long* words = A.words + (size_t)mi * kChunks * n;
        unsigned* sticky = A.sticky + (size_t)mi * n;
        if (A.inst) {
            // batch: the fixed point of each column follows its instance's max
            // |x|; four entries per thread at a time, so that their dependent
            // loads (column, instance, max) overlap
            for (unsigned long long q0 = p0 + (unsigned long long)gt; q0 < p1; q0 += 4ull * nthreads) {
                unsigned long long xb[4];
                int c[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned long long q = q0 + (unsigned long long)u * nthreads;
                    xb[u] = q < p1 ? mag_bits(A.pool_val[q]) : 0ull;
                    c[u] = xb[u] ? A.pool_col[q] : 0;
                }
                int lsb[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    lsb[u] = 0;
                    if (xb[u] && (unsigned)c[u] < (unsigned)A.n)
                        lsb[u] = lsb_for_bound(A.slots[(size_t)A.inst[c[u]] * A.slot_stride + mi].absmax);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (!xb[u]) continue;
                    if ((unsigned)c[u] >= (unsigned)A.n) {
                        atomicOr(&A.ctl->status, kDevInternal);
                        continue;
                    }
                    exact_add(words + c[u], n, sticky + c[u], xb[u], lsb[u]);
                }
            }
            continue;
        }
        const int lsb = lsb_for_bound(A.slots[mi].absmax);
        for (unsigned long long q0 = p0 + (unsigned long long)gt; q0 < p1; q0 += 4ull * nthreads) {
            unsigned long long xb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long q = q0 + (unsigned long long)u * nthreads;
                xb[u] = q < p1 ? mag_bits(A.pool_val[q]) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (xb[u] != 0ull) {
                    const int c = A.pool_col[q0 + (unsigned long long)u * nthreads];
                    exact_add_checked(words, sticky, c, A.n, xb[u], lsb, A.ctl);
                }
            }
        }
    }
    if (!grid_barrier(A.ctl, A.budget_ns)) return;
    const int lane = threadIdx.x & 31;
    for (int mi = 0; mi < A.count; ++mi) {
        unsigned long long* words = A.words + (size_t)mi * kChunks * n;
        unsigned long long mx = 0ull;
        for (int j = gt; j < A.n; j += nthreads) {
            NormSlot* slot = A.inst ? A.slots + (size_t)A.inst[j] * A.slot_stride + mi : A.slots + mi;
            const int lsb = lsb_for_bound(slot->absmax);
            const double sum = chunk_round(words + j, n, A.sticky + (size_t)mi * n + j, lsb);
            const unsigned long long sb = (unsigned long long)__double_as_longlong(sum);
            if (A.inst) {
                if (sb) atomicMax(&slot->result, sb);  // columns of one warp may belong to several instances
            } else {
                mx = sb > mx ? sb : mx;
            }
        }
        if (!A.inst) {
            mx = warp_max_u64(mx);  // one reduction per warp, not per column
            if (lane == 0 && mx) atomicMax(&A.slots[mi].result, mx);
        }
    }
}

// ---------------------------------------------------------------- k_norms_rows
// The same norms, by tiles of consecutive rows: for banded and grid matrices
// a tile's entries fall in a narrow window of columns, so a block sums its
// tile exactly in shared memory (24-bit pieces in 32-bit words: a tile of at
// most 255 rows cannot overflow them) and adds the window to the global sums
// once, instead of one global reduction per piece of every entry.  A tile
// whose window is wider than kNormWin takes the global path entry by entry.
// One block per (tile, matrix); k_norms_finish rounds and takes the maxima.
// Bound by instructions (51 % of the issue slots, one block of 32 warps an SM):
// Z^1..Z^10 of a 128 x 128 grid, 14.6 M entries, 114 -> 103 us with the split
// written out in 32-bit shifts; exp banded n = 65536 3800 -> 3770 us a call.
constexpr int kNormTile = 128;
constexpr int kNormWin = 3072;
constexpr int kNormRowsThreads = 1024;
static_assert(kNormTile <= 255, "shared 24-bit pieces of a tile must not overflow");

size_t norms_rows_smem_bytes() { return sizeof(unsigned) * (size_t)(kNormPieces + 1) * kNormWin; }

__global__ void __launch_bounds__(kNormRowsThreads) k_norms_rows(NormRowsArgs A) {
    pdl_enter();
    extern __shared__ unsigned nsm[];  // [kNormPieces][kNormWin] pieces, then [kNormWin] sticky counts
    __shared__ int s_lo[kNormRowsThreads / 32], s_hi[kNormRowsThreads / 32];
    if (__ldcg(&A.ctl->status) & kDevPoolFull) return;  // discarded phase
    const int mi = blockIdx.y;
    const int n = A.n;
    const int r0 = blockIdx.x * kNormTile, r1 = min(n, r0 + kNormTile);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int* rb = A.rb[mi];
    const int* re = A.re[mi];
    const int lsb0 = A.inst ? 0 : lsb_for_bound(A.slots[mi].absmax);
    unsigned long long* words = A.words + (size_t)mi * kNormPieces * n;
    unsigned* sticky = A.sticky + (size_t)mi * n;
    // the tile's column window (rows are sorted)
    int lo = INT_MAX, hi = -1;
    for (int r = r0 + (int)threadIdx.x; r < r1; r += blockDim.x) {
        const int s = rb[r], e = re[r];
        if (s < e) {
            lo = min(lo, A.col[s]);
            hi = max(hi, A.col[e - 1]);
        }
    }
    lo = warp_min(lo);
    hi = warp_max(hi);
    if (lane == 0) {
        s_lo[wid] = lo;
        s_hi[wid] = hi;
    }
    __syncthreads();
    lo = INT_MAX;
    hi = -1;
    for (int i = 0; i < nw; ++i) {
        lo = min(lo, s_lo[i]);
        hi = max(hi, s_hi[i]);
    }
    if (hi < lo) return;  // an empty tile (same in all threads)
    if (lo < 0 || hi >= n) {
        if (threadIdx.x == 0) atomicOr(&A.ctl->status, kDevInternal);
        return;
    }
    const int wlen = hi - lo + 1;
    const bool local = wlen <= kNormWin;
    unsigned* wst = nsm + (size_t)kNormPieces * kNormWin;
    if (local) {
        for (int i = threadIdx.x; i < wlen; i += blockDim.x) {
#pragma unroll
            for (int p = 0; p < kNormPieces; ++p) nsm[p * kNormWin + i] = 0u;
            wst[i] = 0u;
        }
        __syncthreads();
    }
    for (int r = r0 + wid; r < r1; r += nw) {
        const int s = rb[r], e = re[r];
        // batch: the fixed point of a column follows its instance's max |x|;
        // a row's columns all belong to the row's instance (block diagonal)
        const int lsb = A.inst ? lsb_for_bound(A.slots[(size_t)A.inst[r] * A.slot_stride + mi].absmax) : lsb0;
        // 128 entries per round, all loads issued first
        for (int q0 = s; q0 < e; q0 += 128) {
            unsigned long long xs[4];
            int cs[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = q0 + u * 32 + lane;
                xs[u] = q < e ? mag_bits(A.val[q]) : 0ull;
                cs[u] = q < e ? A.col[q] : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned long long xb = xs[u];
                if (xb == 0ull) continue;
                const int c = cs[u], o = c - lo;
                if ((unsigned)o >= (unsigned)wlen) {  // (rows are sorted: never)
                    atomicOr(&A.ctl->status, kDevInternal);
                    continue;
                }
                // split24, without its cases for values below the fixed
                // point's last bit (32-bit words of the shifted mantissa, cut
                // into the same pieces)
                unsigned p0, p1, p2, p3;
                int L;
                const unsigned xh = (unsigned)(xb >> 32), xl = (unsigned)xb, E = xh >> 20;
                const int sh = (int)E - 1075 - lsb;
                bool lost = false;
                if (E != 0u && sh >= 0) {
                    const unsigned mh = (xh & 0xfffffu) | 0x100000u, q24 = (unsigned)sh / 24u, t = (unsigned)sh - q24 * 24u;
                    const unsigned w0 = xl << t, w1 = __funnelshift_l(xl, mh, t), w2 = __funnelshift_l(mh, 0u, t);
                    L = (int)q24;
                    p0 = w0 & 0xffffffu;
                    p1 = __funnelshift_r(w0, w1, 24) & 0xffffffu;
                    p2 = __funnelshift_r(w1, w2, 16) & 0xffffffu;
                    p3 = w2 >> 8;
                } else {
                    unsigned pc[4];
                    L = split24(xb, lsb, pc, lost);
                    p0 = pc[0];
                    p1 = pc[1];
                    p2 = pc[2];
                    p3 = pc[3];
                }
                if (local) {
                    unsigned* const w = nsm + L * kNormWin + o;
                    atomicAdd(w, p0);
                    atomicAdd(w + kNormWin, p1);
                    atomicAdd(w + 2 * kNormWin, p2);
                    if (p3) atomicAdd(w + 3 * kNormWin, p3);
                    if (lost) atomicAdd(&wst[o], 1u);
                } else {
                    unsigned long long* const w = words + (size_t)L * n + c;
                    if (p0) atomicAdd(w, (unsigned long long)p0);
                    if (p1) atomicAdd(w + n, (unsigned long long)p1);
                    if (p2) atomicAdd(w + 2 * (size_t)n, (unsigned long long)p2);
                    if (p3) atomicAdd(w + 3 * (size_t)n, (unsigned long long)p3);
                    if (lost) atomicAdd(&sticky[c], 1u);
                }
            }
        }
    }
    if (!local) return;
    __syncthreads();
    for (int i = threadIdx.x; i < wlen; i += blockDim.x) {
#pragma unroll
        for (int p = 0; p < kNormPieces; ++p) {
            const unsigned v = nsm[p * kNormWin + i];
            if (v) atomicAdd(&words[(size_t)p * n + lo + i], (unsigned long long)v);
        }
        if (wst[i]) atomicAdd(&sticky[lo + i], wst[i]);
    }
}

__global__ void k_norms_finish(int n, int count, NormSlot* slots, unsigned long long* words, unsigned* sticky,
                               const Ctl* ctl, const int* inst, int slot_stride) {
    pdl_enter();
    if (__ldcg(&ctl->status) & kDevPoolFull) return;
    // one thread per (matrix, column); the column count is padded to whole
    // warps so that a warp's columns belong to one matrix and it reduces
    // them before the single atomic
    const long long npad = ((long long)n + 31) & ~31LL;
    const long long nt = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < (long long)count * npad; u += nt) {
        const int mi = (int)(u / npad), j = (int)(u % npad);
        unsigned long long vb = 0ull;
        NormSlot* slot = slots + mi;
        if (j < n) {
            if (inst) slot = slots + (size_t)inst[j] * slot_stride + mi;
            const int lsb = lsb_for_bound(slot->absmax);
            const double v = round24(words + (size_t)mi * kNormPieces * n + j, (size_t)n, sticky + (size_t)mi * n + j, lsb);
            vb = (unsigned long long)__double_as_longlong(v);
        }
        if (inst) {
            // a warp's columns are consecutive, so their instances form
            // contiguous runs: a segmented reduction leaves each run's
            // maximum in its first lane
            const int ti = j < n ? inst[j] : -1;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long w = __shfl_down_sync(kFull, vb, o);
                const int tj = __shfl_down_sync(kFull, ti, o);
                if (lane + o < 32 && tj == ti) vb = w > vb ? w : vb;
            }
            const int tp = __shfl_up_sync(kFull, ti, 1);
            const bool first = lane == 0 || tp != ti;
            if (first && ti >= 0 && vb) atomicMax(&slot->result, vb);
        } else {
            vb = warp_max_u64(vb);
            if (lane == 0 && vb) atomicMax(&slot->result, vb);
        }
    }
}

// ---------------------------------------------------------------- k_export
// Copy nwords 32-bit words of a device record (the control block, norm slots,
// step records) into pinned host memory mapped into the device's address
// space.  The host reads the words after synchronising with the stream.  A
// kernel's stores take no copy engine, so these small read-backs do not
// queue behind a large device-to-host copy that another stream has in
// flight (a result being copied out while the next evaluation runs).
__global__ void k_export(const unsigned* src, unsigned* dst, int nwords) {
    pdl_enter();
    for (int i = threadIdx.x; i < nwords; i += blockDim.x) dst[i] = __ldcg(src + i);
}

// ---------------------------------------------------------------- k_row_bitmaps
// Column bitmap of every row of B for the product's symbolic pass: hdr[r] =
// {first column / 32, words}, the words at bits[rb[r]] on.  A row gets one
// only if it needs no more words than it has entries (so they fit its own
// pool range) and no more than one window's; otherwise words = 0.  One warp
// per row: each 32-entry piece ORs runs of lanes with the same word (the
// columns ascend) and the first lane of a run adds it to the word.
__global__ void k_row_bitmaps(int n, RowView B, int2* hdr, unsigned* bits) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += nwarps) {
        const int s = B.rb[r], e = B.re[r];
        int2 h = make_int2(0, 0);
        if (e > s) {
            const int w0 = B.col[s] >> 5;
            const int nw = (B.col[e - 1] >> 5) - w0 + 1;
            h.x = w0;
            if (nw <= e - s && nw <= kBmWordsBig) {
                h.y = nw;
                for (int j = lane; j < nw; j += 32) bits[s + j] = 0u;
                __syncwarp();
                for (int q0 = s; q0 < e; q0 += 32) {
                    const int q = q0 + lane;
                    const bool in = q < e;
                    const int c = in ? B.col[q] : 0;
                    const int wi = in ? (c >> 5) - w0 : -1 - lane;
                    unsigned v = in ? 1u << (c & 31) : 0u;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const unsigned v2 = __shfl_down_sync(kFull, v, d);
                        const int w2 = __shfl_down_sync(kFull, wi, d);
                        if (lane + d < 32 && w2 == wi) v |= v2;
                    }
                    const int wp = __shfl_up_sync(kFull, wi, 1);
                    if (in && (lane == 0 || wp != wi)) atomicOr(bits + s + wi, v);
                }
            }
        }
        if (lane == 0) hdr[r] = h;
    }
}

// ---------------------------------------------------------------- k_copy_result
// A result's arrays into the caller's, in one launch instead of three copies:
// each copy cost about 5 us of the host's time and 2 us on the stream, more
// than the bytes of a small result (a batch of 128 hands over 384 arrays).
// 16 bytes a thread and access, four in flight, where source and destination
// are aligned alike; the arrays of a batch's results start anywhere and go by
// words.
// A batch call of 128 instances 17.05 -> 16.25 ms, one banded product
// (n = 30001, 4 MB of result) 281 -> 259 us.
struct CopyArgs {
    const unsigned* src[3];
    unsigned* dst[3];
    long long words[3];
};
__global__ void __launch_bounds__(256) k_copy_result(const __grid_constant__ CopyArgs C) {
    pdl_enter();
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        const unsigned* s = C.src[a];
        unsigned* d = C.dst[a];
        const long long n = C.words[a];
        const long long head = ((16 - ((unsigned long long)d & 15)) & 15) >> 2;
        if ((((unsigned long long)s ^ (unsigned long long)d) & 15) == 0 && n > head) {
            const long long q = (n - head) >> 2;  // 16-byte pieces
            const uint4* s4 = reinterpret_cast<const uint4*>(s + head);
            uint4* d4 = reinterpret_cast<uint4*>(d + head);
            long long i = t0;
            for (; i + 3 * step < q; i += 4 * step) {
                const uint4 x0 = s4[i], x1 = s4[i + step], x2 = s4[i + 2 * step], x3 = s4[i + 3 * step];
                d4[i] = x0;
                d4[i + step] = x1;
                d4[i + 2 * step] = x2;
                d4[i + 3 * step] = x3;
            }
            for (; i < q; i += step) d4[i] = s4[i];
            if (t0 < head) d[t0] = s[t0];
            const long long tail = head + 4 * q + t0;
            if (tail < n) d[tail] = s[tail];
        } else {
            long long i = t0;
            for (; i + 3 * step < n; i += 4 * step) {
                const unsigned x0 = s[i], x1 = s[i + step], x2 = s[i + 2 * step], x3 = s[i + 3 * step];
                d[i] = x0;
                d[i + step] = x1;
                d[i + 2 * step] = x2;
                d[i + 3 * step] = x3;
            }
            for (; i < n; i += step) d[i] = s[i];
        }
    }
}

// ---------------------------------------------------------------- k_row_lists
// The words of every row of B that hold entries, as {column / 32, bitmap} at
// the row's own positions of `lists`, columns ascending; hdr[r].y = how many
// (never more than the row's entries).  One warp per row; a 32-entry piece's
// last run of columns may go on in the next piece and is carried over.
__global__ void k_row_lists(int n, RowView B, int2* hdr, uint2* lists) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += nwarps) {
        const int s = B.rb[r], e = B.re[r];
        int m = 0;               // words written
        int cw = -1;             // the carried run's word
        unsigned cb = 0u;        // and bits
        for (int q0 = s; q0 < e; q0 += 32) {
            const int q = q0 + lane;
            const bool in = q < e;
            const int c = in ? B.col[q] : 0;
            const int w = in ? c >> 5 : -2 - lane;
            unsigned v = in ? 1u << (c & 31) : 0u;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned v2 = __shfl_down_sync(kFull, v, d);
                const int w2 = __shfl_down_sync(kFull, w, d);
                if (lane + d < 32 && w2 == w) v |= v2;
            }
            const int wp = __shfl_up_sync(kFull, w, 1);
            const unsigned lead = __ballot_sync(kFull, in && (lane == 0 || wp != w));
            const bool joins = __shfl_sync(kFull, w, 0) == cw;  // the first run continues the carried one
            if (joins) {
                if (lane == 0) v |= cb;
            } else if (cw >= 0) {
                if (lane == 0) lists[s + m] = make_uint2((unsigned)cw, cb);
                ++m;
            }
            const int ll = 31 - __clz(lead);  // the last run's first lane: carried
            if ((lead >> lane & 1u) && lane != ll)
                lists[s + m + __popc(lead & lanemask_lt())] = make_uint2((unsigned)w, v);
            m += __popc(lead) - 1;
            cw = __shfl_sync(kFull, w, ll);
            cb = __shfl_sync(kFull, v, ll);
        }
        if (lane == 0) {
            if (cw >= 0) lists[s + m] = make_uint2((unsigned)cw, cb);
            hdr[r] = make_int2(0, cw >= 0 ? m + 1 : 0);
        }
    }
}

// ---------------------------------------------------------------- plumbing
// An empty pool of `cap` entries and empty candidate lists (the barrier's and
// the counters' fields from bar_count on keep their values).
__global__ void k_reset(Ctl* ctl, unsigned long long cap, unsigned long long cand_cap, unsigned cand_chunk) {
    pdl_enter();
    if (threadIdx.x) return;
    ctl->pool_used = ctl->pool_mark = 0ull;
    ctl->pool_cap = cap;
    ctl->cslot[0] = ctl->cslot[1] = ctl->nnz_total = 0ull;
    ctl->status = 0;
    ctl->cand_cnt[0] = ctl->cand_cnt[1] = ctl->cand_far = 0ull;
    ctl->cand_cap = cand_cap;
    ctl->cand_over = 0;
    ctl->cand_chunk = cand_chunk;
    ctl->dropped = 0;
}

// max |x| over the pool entries [mark[i], mark[i+1])
__global__ void k_absmax(const double* pool_val, const Ctl* ctl, int i, NormSlot* slot) {
    pdl_enter();
    if (__ldcg(&ctl->status) & kDevBadInput) return;  // (as k_norms)
    const int lane = threadIdx.x & 31;
    const unsigned long long cap = ctl->pool_cap;  // counters may run past it on overflow
    const unsigned long long p0 = min(__ldcg(&ctl->mark[i]), cap), p1 = min(__ldcg(&ctl->mark[i + 1]), cap);
    unsigned long long mx = 0ull;
    for (unsigned long long q = p0 + blockIdx.x * blockDim.x + threadIdx.x; q < p1;
         q += (unsigned long long)gridDim.x * blockDim.x) {
        unsigned long long b = mag_bits(pool_val[q]);
        mx = b > mx ? b : mx;
    }
    mx = warp_max_u64(mx);
    if (lane == 0 && mx) atomicMax(&slot->absmax, mx);
}

// Where the rows of B are runs of consecutive columns, a row of A B is one too
// if the B rows that it takes meet one another (share a column, or lie side by
// side), and a sum of powers of Z is if they lie about the diagonal.  Bands do;
// runs at unrelated places (permuted blocks, gathers) don't, and k_band would
// leave every row of their products to the accumulator's narrow map.
// Row r of length len, columns [first, last] of [0, n), is further from the
// diagonal than it is long (and not the rest of one that the edge cuts off).
__device__ __forceinline__ bool far_from_diagonal(int n, int r, int first, int last, int len) {
    const int gap = max(first - r, r - last);
    return gap > len + 1 && ((first > 0 && last < n - 1) || gap > 512);
}
// Row k of a checked matrix (0 < k < n) does not meet row k - 1.
__device__ __forceinline__ bool row_apart(const int* rowptr, const int* col, int k) {
    const int s0 = rowptr[k - 1], s = rowptr[k], e = rowptr[k + 1];
    return s0 < s && s < e && (col[s] - 1 > col[s - 1] || col[e - 1] + 1 < col[s0]);
}
// Row r of A takes rows of B that do not meet, or (series) is far from the diagonal.
__device__ __forceinline__ bool row_falls_apart(int n, const int* a_rp, const int* a_col, const int* b_rp,
                                                const int* b_col, int r, bool series) {
    const int s = a_rp[r], e = a_rp[r + 1];
    if (s >= e) return false;
    if (series && far_from_diagonal(n, r, a_col[s], a_col[e - 1], e - s)) return true;
    for (int q = s + 1; q < e; ++q)
        if (row_apart(b_rp, b_col, a_col[q])) return true;
    return false;
}
// How many rows do (a second look, after k_validate or k_validate_batch has
// seen a row apart or far from the diagonal: about 10 us that bands don't pay).
__global__ void k_count_apart(int n, const int* a_rp, const int* a_col, const int* b_rp, const int* b_col, int series,
                              Ctl* ctl) {
    pdl_enter();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = warp_sum(r < n && row_falls_apart(n, a_rp, a_col, b_rp, b_col, r, series != 0) ? 1 : 0);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&ctl->apart_rows, (unsigned)c);
}
__global__ void k_count_apart_batch(int n, const int* inst, const BatchSrc* src, unsigned* count) {
    pdl_enter();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const BatchSrc S = src[inst[r]];
    if (row_falls_apart(S.n, S.rowptr, S.col, S.rowptr, S.col, r - S.off, true)) atomicAdd(count + inst[r], 1u);
}

// Check a canonical CSR input: row pointers non-decreasing from 0 to nnz,
// columns in range and strictly increasing per row, values finite.
__global__ void k_validate(int n, int nnz, const int* rowptr, const int* col, const double* val,
                           Ctl* ctl) {
    pdl_enter();
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false, holes = false, apart = false;
    int bw = 0;
    if (r > n) {
    } else if (r == n) {
        if (rowptr[n] != nnz || (n == 0 && rowptr[0] != 0)) bad = true;
    } else {
        if (r == 0 && rowptr[0] != 0) bad = true;
        int s = rowptr[r], e = rowptr[r + 1];
        if (s > e || s < 0 || e > nnz) {
            bad = true;
        } else {
            int prev = -1;
            for (int q = s; q < e; ++q) {
                int c = col[q];
                double v = val[q];
                bool finite = (mag_bits(v) >> 52) != 0x7ffull;
                if (c <= prev || c >= n || !finite) {
                    bad = true;
                    break;
                }
                prev = c;
            }
            if (e > s && !bad) {
                bw = max(prev - r, r - col[s]);
                holes = prev - col[s] != e - s - 1;
                apart = far_from_diagonal(n, r, col[s], prev, e - s);
                const int s0 = r > 0 ? rowptr[r - 1] : s;  // (the row before may not have passed)
                if (s0 >= 0 && s0 < s) apart = apart || col[s] - 1 > col[s - 1] || prev + 1 < col[s0];
            }
        }
    }
    if (bad) atomicOr(&ctl->status, kDevBadInput);
    // (one store a warp)
    bw = warp_max(bw);
    const unsigned any_holes = __ballot_sync(kFull, holes), any_apart = __ballot_sync(kFull, apart && !holes);
    if ((threadIdx.x & 31) == 0) {
        if (bw > 0) atomicMax(&ctl->bandwidth, (unsigned)bw);
        if (any_holes) ctl->not_band = 1;
        if (any_apart) ctl->apart = 1;
    }
}

// Exclusive scan of row lengths (re - rb, or a pooled matrix's true entries
// when rd is given) into rowptr (n + 1 entries), in two launches over tiles of
// kScanTile rows: the tile sums and their scan, then the scan inside each tile
// plus its tile's offset.
// `sums` holds ceil(n / kScanTile) + 1 values.
constexpr int kScanTile = 1024;

__device__ __forceinline__ long long block_excl_scan(long long v, long long* part, long long* total) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) part[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int nw = (int)(blockDim.x >> 5);
        long long p = lane < nw ? part[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(kFull, p, o);
            if (lane >= o) p += y;
        }
        if (lane < nw) part[lane] = p;  // inclusive warp totals
    }
    __syncthreads();
    const long long before = wid ? part[wid - 1] : 0;
    *total = part[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before + x - v;
}

// The tile sums; the last block to finish scans them.
__global__ void __launch_bounds__(kScanTile) k_scan_tile_sums(int n, const int* rb, const int* re, const RowDesc* rd,
                                                              long long* sums, Ctl* ctl) {
    pdl_enter();
    __shared__ long long part[32];
    __shared__ int last_block;
    const long long r = (long long)blockIdx.x * kScanTile + threadIdx.x;
    const long long len = r < n ? (long long)(rd ? rd_nnz(rd[r]) : re[r] - rb[r]) : 0;
    long long total;
    block_excl_scan(len, part, &total);
    const int ntiles = gridDim.x;
    if (threadIdx.x == 0) {
        sums[blockIdx.x] = total;
        __threadfence();
        last_block = atomicAdd(&ctl->done, 1u) == (unsigned)ntiles - 1u;
    }
    __syncthreads();
    if (!last_block) return;
    // each thread owns a contiguous run of tiles
    const int per = (ntiles + kScanTile - 1) / kScanTile;
    const int t0 = min(ntiles, (int)threadIdx.x * per), t1 = min(ntiles, t0 + per);
    long long s = 0;
    for (int t = t0; t < t1; ++t) s += __ldcg(sums + t);
    long long run = block_excl_scan(s, part, &total);
    for (int t = t0; t < t1; ++t) {
        const long long v = __ldcg(sums + t);
        sums[t] = run;
        run += v;
    }
    if (threadIdx.x == 0) {
        sums[ntiles] = total;
        ctl->nnz_total = (unsigned long long)total;
        ctl->done = 0u;
    }
}

__global__ void __launch_bounds__(kScanTile) k_scan_apply(int n, const int* rb, const int* re, const RowDesc* rd,
                                                           const long long* sums, int* rowptr) {
    pdl_enter();
    __shared__ long long part[32];
    const long long r = (long long)blockIdx.x * kScanTile + threadIdx.x;
    const long long len = r < n ? (long long)(rd ? rd_nnz(rd[r]) : re[r] - rb[r]) : 0;
    long long total;
    const long long ex = block_excl_scan(len, part, &total) + sums[blockIdx.x];
    if (r < n) rowptr[r] = (int)ex;  // the host rejects totals of 2^31 and more
    if (r == n - 1 || (n == 0 && r == 0)) rowptr[n] = (int)sums[gridDim.x];
}

// A row's true entries to col/val at d on, columns less `shift`, by one warp.
__device__ __forceinline__ void gather_row(const RowView& src, int r, long long d, int shift, int* col, double* val,
                                           int lane) {
    const RowDesc rd = src.rd[r];
    const int s = rd.rb, len = rd.re - s;
    if (rd_nnz(rd) == len) {
        for (int q = lane; q < len; q += 32) {
            col[d + q] = src.col[s + q] - shift;
            val[d + q] = src.val[s + q];
        }
        return;
    }
    for (int q0 = 0; q0 < len; q0 += 32) {  // without the holes
        const int q = q0 + lane;
        const double x = q < len ? src.val[s + q] : 0.0;
        const bool nz = mag_bits(x) != 0ull;
        const unsigned m = __ballot_sync(kFull, nz);
        if (nz) {
            const long long at = d + __popc(m & lanemask_lt());
            col[at] = src.col[s + q] - shift;
            val[at] = x;
        }
        d += __popc(m);
    }
}

__global__ void k_gather(int n, RowView src, const int* rowptr, int* col, double* val) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = gw; r < n; r += nwarps) gather_row(src, r, rowptr[r], 0, col, val, lane);
}

// Copy a canonical CSR matrix into the pool: each row gets a 4-entry aligned
// slot of round-up(len, 4) entries (rows start 16-byte aligned, like the
// product kernel's rows).
__global__ void k_copy_rows(int n, const int* rowptr, const int* col, const double* val, int* rb, int* re,
                            RowDesc* rd, int* pool_col, double* pool_val, Ctl* ctl, unsigned long long arena_size,
                            NormSlot* absmax) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    Arena arena;
    unsigned long long mx = 0ull;
    for (int r = gw; r < n; r += nwarps) {
        int s = rowptr[r], e = rowptr[r + 1];
        const long long base = arena_take(arena, (unsigned long long)((e - s + 3) & ~3), arena_size, ctl, pool_val, lane);
        if (base < 0) {
            if (lane == 0) {
                rb[r] = re[r] = 0;
                rd[r] = RowDesc{0, 0, 0, 0};
            }
            continue;
        }
        const int padded = (e - s + 3) & ~3;
        for (int q = lane; q < padded; q += 32) {
            const double v = q < e - s ? val[s + q] : 0.0;
            pool_col[base + q] = q < e - s ? col[s + q] : 0;
            pool_val[base + q] = v;
            const unsigned long long b = mag_bits(v);
            mx = b > mx ? b : mx;
        }
        if (lane == 0) {
            rb[r] = (int)base;
            re[r] = (int)base + (e - s);
            rd[r] = rd_row((int)base, (int)base + (e - s), e > s ? col[s] : 0, e > s ? col[e - 1] : 0);
        }
    }
    arena_close(arena, pool_val, lane);
    if (absmax) {  // max |x| (the fixed point of the norm), one atomic per block
        __shared__ unsigned long long blk;
        if (threadIdx.x == 0) blk = 0ull;
        __syncthreads();
        mx = warp_max_u64(mx);
        if (lane == 0 && mx) atomicMax(&blk, mx);
        __syncthreads();
        if (threadIdx.x == 0 && blk) atomicMax(&absmax->absmax, blk);
    }
    step_done(ctl, 1, nullptr, nullptr, nullptr, 0);
}

// Reset a caller-provided norm workspace for one matrix of n columns and
// nnz entries read in place: clear the control block, the norm slot and the
// column-sum words, and let the matrix's entries [0, nnz) be norm matrix 0.
__global__ void k_norm_scratch_init(Ctl* ctl, NormSlot* slot, unsigned long long* words, unsigned* sticky, int n,
                                    long long nnz) {
    pdl_enter();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nt = (long long)gridDim.x * blockDim.x;
    for (long long i = t; i < (long long)kChunks * n; i += nt) words[i] = 0ull;
    for (long long i = t; i < n; i += nt) sticky[i] = 0u;
    if (t == 0) {
        Ctl c{};
        c.pool_cap = (unsigned long long)nnz;
        c.pool_used = (unsigned long long)nnz;
        c.mark[0] = 0ull;
        c.mark[1] = (unsigned long long)nnz;
        *ctl = c;
        slot->absmax = 0ull;
        slot->result = 0ull;
    }
}

// ---- batches: the instance of every row (binary search over the row
// offsets off[0..ninst], off[ninst] = n)
__global__ void k_inst_table(int n, int ninst, const int* off, int* inst) {
    pdl_enter();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    int lo = 0, hi = ninst - 1;  // largest i with off[i] <= r
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= r) lo = mid;
        else hi = mid - 1;
    }
    inst[r] = lo;
}

// Check every input of a batch like k_validate: thread per global row.
__global__ void k_validate_batch(int n, const int* inst, const BatchSrc* src, const int* nnz, Ctl* ctl,
                                 unsigned char* band) {
    pdl_enter();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int i = inst[r];
    const BatchSrc S = src[i];
    const int l = r - S.off;
    bool bad = false;
    const int s = S.rowptr[l], e = S.rowptr[l + 1];
    if (l == 0 && s != 0) bad = true;
    if (l == S.n - 1 && e != nnz[i]) bad = true;
    if (s > e || s < 0 || e > nnz[i]) {
        bad = true;
    } else {
        int prev = -1;
        for (int q = s; q < e; ++q) {
            const int c = S.col[q];
            const bool finite = (mag_bits(S.val[q]) >> 52) != 0x7ffull;
            if (c <= prev || c >= S.n || !finite) {
                bad = true;
                break;
            }
            prev = c;
        }
        if (e > s && prev - S.col[s] != e - s - 1) band[i] = 0;
        if (e > s && !bad) {
            bool apart = far_from_diagonal(S.n, l, S.col[s], prev, e - s);
            const int s0 = l > 0 ? S.rowptr[l - 1] : s;
            if (s0 >= 0 && s0 < s) apart = apart || S.col[s] - 1 > S.col[s - 1] || prev + 1 < S.col[s0];
            if (apart && prev - S.col[s] == e - s - 1 && __ldcg(&ctl->apart) == 0) ctl->apart = 1;
        }
    }
    if (bad) atomicOr(&ctl->status, kDevBadInput);
}

// Copy the inputs of a batch into the pool as the block-diagonal matrix
// (columns shifted to global), rows padded to 4 entries; records each
// instance's max |x| in absmax[i * stride].
__global__ void k_copy_rows_batch(int n, const int* inst, const BatchSrc* src, int* rb, int* re, RowDesc* rd,
                                  int* pool_col, double* pool_val, Ctl* ctl, unsigned long long arena_size, NormSlot* absmax,
                                  int stride) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    Arena arena;
    for (int r = gw; r < n; r += nwarps) {
        const int i = inst[r];
        const BatchSrc S = src[i];
        const int l = r - S.off;
        const int s = S.rowptr[l], e = S.rowptr[l + 1];
        const long long base = arena_take(arena, (unsigned long long)((e - s + 3) & ~3), arena_size, ctl, pool_val, lane);
        if (base < 0) {
            if (lane == 0) {
                rb[r] = re[r] = 0;
                rd[r] = RowDesc{0, 0, 0, 0};
            }
            continue;
        }
        const int padded = (e - s + 3) & ~3;
        unsigned long long mx = 0ull;
        for (int q = lane; q < padded; q += 32) {
            const bool in = q < e - s;
            const double v = in ? S.val[s + q] : 0.0;
            pool_col[base + q] = in ? S.col[s + q] + S.off : 0;
            pool_val[base + q] = v;
            const unsigned long long b = mag_bits(v);
            mx = b > mx ? b : mx;
        }
        mx = warp_max_u64(mx);
        if (lane == 0) {
            rb[r] = (int)base;
            re[r] = (int)base + (e - s);
            rd[r] = rd_row((int)base, (int)base + (e - s), e > s ? S.col[s] + S.off : 0,
                           e > s ? S.col[e - 1] + S.off : 0);
            if (absmax && mx) atomicMax(&absmax[(size_t)i * stride].absmax, mx);
        }
    }
    arena_close(arena, pool_val, lane);
    step_done(ctl, 1, nullptr, nullptr, nullptr, 0);
}

// out rows <- the rows of matrix sel[inst[r]] of a table of row descriptors.
struct RowTable {
    const RowDesc* rd[kMaxAdd + 2];
};
__global__ void k_compose_rows(int n, const int* inst, const int* sel, RowTable T, int* out_rb, int* out_re,
                               RowDesc* out_rd) {
    pdl_enter();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const RowDesc d = T.rd[sel[inst[r]]][r];
    out_rb[r] = d.rb;
    out_re[r] = d.re;
    out_rd[r] = d;
}

// Split the block-diagonal result (global row pointers rowptr) into the
// instances' CSR: instance i's row pointers start at out_rp + off_i + i
// (n_i + 1 entries, rebased to 0), its entries at rowptr[off_i] with local
// columns.
__global__ void k_gather_batch(int n, int ninst, const int* inst, const int* off, RowView src, const int* rowptr,
                               int* out_rp, int* col, double* val) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int gw = gt >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = gt; i < ninst; i += gridDim.x * blockDim.x)
        out_rp[off[i + 1] + i] = rowptr[off[i + 1]] - rowptr[off[i]];
    for (int r = gw; r < n; r += nwarps) {
        const int i = inst[r];
        const int o = off[i];
        const int d = rowptr[r];
        if (lane == 0) out_rp[r + i] = d - rowptr[o];
        gather_row(src, r, d, o, col, val, lane);
    }
}

// bounds[i] = rowptr[off[i]], i = 0..ninst
__global__ void k_bounds(int ninst, const int* off, const int* rowptr, int* bounds) {
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= ninst) bounds[i] = rowptr[off[i]];
}

__global__ void k_identity(int n, double alpha, int* rowptr, int* col, double* val) {
    pdl_enter();
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) {
        rowptr[r] = r;
        col[r] = r;
        val[r] = alpha;
    }
    if (r == n) rowptr[n] = n;
}

// ---------------------------------------------------------------- launchers
// Launch configuration, per device (set up once by kernels_init, guarded by
// a mutex; a device's entry is published through `ready`).
struct DevCfg {
    int sms = 0, alg1_blocks = 0, alg1_cluster = 0, alg1b_blocks = 0, norm_blocks = 0;
    std::atomic<bool> ready{false};
};
constexpr int kMaxDevices = 64;
static DevCfg g_dev[kMaxDevices];
// wait limit of every grid barrier (PSF_TUNE_BARRIER_BUDGET_NS)
static std::atomic<unsigned long long> g_barrier_budget_ns{kBarrierBudgetDefaultNs};
void set_barrier_budget_ns(unsigned long long ns) { g_barrier_budget_ns.store(ns); }
unsigned long long barrier_budget_ns() { return g_barrier_budget_ns.load(); }
static std::mutex g_init_mu;
static std::atomic<long long> g_launches{0};

long long launch_count() { return g_launches.load(); }
void count_launches(int k) { g_launches += k; }

static const DevCfg& dcfg();
static int sms_now();
static const DevCfg& dcfg() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
    return g_dev[dev];
}

cudaError_t kernels_init() {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    DevCfg& c = g_dev[dev];
    if (c.ready.load(std::memory_order_acquire)) return cudaSuccess;
    std::lock_guard<std::mutex> lock(g_init_mu);
    if (c.ready.load(std::memory_order_acquire)) return cudaSuccess;
    int sms = 0;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    const void* prods[8] = {(const void*)k_product<false, false, true, kListWords>,
                            (const void*)k_product<true, false, false>, (const void*)k_product<false, false, false>,
                            (const void*)k_product<true, true, false>, (const void*)k_product<false, true, false>,
                            (const void*)k_product<false, false, true>,
                            (const void*)k_product<false, false, true, kBmWordsBig>,
                            (const void*)k_product<false, true, false, kBmWordsBig>};
    const int psmem[8] = {(int)prod_smem_bytes<false, kListWords>(),
                          (int)prod_smem_bytes<true>(), (int)prod_smem_bytes<false>(), (int)prod_smem_bytes<true>(),
                          (int)prod_smem_bytes<false>(), (int)prod_smem_bytes<false>(),
                          (int)prod_smem_bytes<false, kBmWordsBig>(), (int)prod_smem_bytes<false, kBmWordsBig>()};
    for (int i = 0; i < 8; ++i) {
        err = cudaFuncSetAttribute(prods[i], cudaFuncAttributeMaxDynamicSharedMemorySize, psmem[i]);
        if (err != cudaSuccess) return err;
    }
    err = cudaFuncSetAttribute((const void*)k_product_cta, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)cta_smem_bytes());
    if (err != cudaSuccess) return err;
    const void* bands[12] = {
        (const void*)k_band<true, false, 1, false>,  (const void*)k_band<true, false, 1, true>,
        (const void*)k_band<false, false, 1, false>, (const void*)k_band<false, false, 4, false>,
        (const void*)k_band<false, true, 1, false>,  (const void*)k_band<false, true, 4, false>,
        (const void*)k_band<true, false, 4, false>,  (const void*)k_band<false, false, 1, true>,
        (const void*)k_band<false, false, 4, true>,  (const void*)k_band<false, true, 1, true>,
        (const void*)k_band<false, true, 4, true>,   (const void*)k_band<true, false, 4, true>};
    for (const void* k : bands) {
        err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)band_smem_bytes());
        if (err != cudaSuccess) return err;
    }
    err = cudaFuncSetAttribute((const void*)k_norms_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)norms_rows_smem_bytes());
    if (err != cudaSuccess) return err;
    int per = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_alg1<false>, kAlg1Threads, 0);
    if (err != cudaSuccess) return err;
    c.alg1_blocks = sms * (per < kAlg1BlocksPerSm ? per : kAlg1BlocksPerSm);
    // one cluster of 16 blocks where the device takes it (8 is what every
    // device does)
    c.alg1_cluster = 8;
    if (cudaFuncSetAttribute((const void*)k_alg1<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t q{};
        q.gridDim = dim3(16);
        q.blockDim = dim3(kAlg1Threads);
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 16;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        q.attrs = &at;
        q.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_alg1<true>, &q) == cudaSuccess && clusters > 0)
            c.alg1_cluster = 16;
    }
    cudaGetLastError();
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_alg1_batch, kAlg1Threads, 0);
    if (err != cudaSuccess) return err;
    c.alg1b_blocks = sms * (per < 4 ? per : 4);
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_norms, kNormThreads, 0);
    if (err != cudaSuccess) return err;
    c.norm_blocks = sms * (per < 2 ? per : 2);
    if (c.alg1_blocks <= 0 || c.alg1b_blocks <= 0 || c.norm_blocks <= 0) return cudaErrorInvalidConfiguration;
    c.sms = sms;
    c.ready.store(true, std::memory_order_release);
    return cudaSuccess;
}

int num_sms() { return dcfg().sms; }
static int sms_now() { return dcfg().sms; }

template <bool TAB, bool BATCH, bool WIDE, int W = kBmWords>
static cudaError_t prod_launch(const ProductArgs& P, cudaStream_t st) {
    constexpr int kWarps = ProdSmem<TAB, W>::kWarps;
    // one wave of resident blocks, rows strided over the warps (each warp
    // keeps one pool arena)
    long long blocks = ((long long)P.n + kWarps - 1) / kWarps;
    const long long cap = (long long)sms_now() * ProdSmem<TAB, W>::kBlocksPerSm;
    if (blocks > cap) blocks = cap;
    // (an ordinary launch: one wave of blocks that fill shared memory must find
    // every SM free.  Brought in while a kernel without shared memory runs,
    // some SMs take fewer of them and the rest make a second wave: cos on a
    // 101 x 97 grid, squared, 2.64 -> 2.87 ms, exp on 128 x 128 3.61 -> 3.72)
    k_product<TAB, BATCH, WIDE, W><<<(unsigned)blocks, kWarps * 32, prod_smem_bytes<TAB, W>(), st>>>(P);
    ++g_launches;
    return cudaGetLastError();
}

static cudaError_t cta_launch(const ProductArgs& P, cudaStream_t st) {
    long long blocks = P.n;
    const long long cap = (long long)sms_now() * 7;
    if (blocks > cap) blocks = cap;
    launch_pdl(k_product_cta, (unsigned)blocks, kCtaWarps * 32, cta_smem_bytes(), st, P);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_product(const ProductArgs& P, bool table, cudaStream_t st, double out_len, bool wide_window,
                           bool cta) {
    if (P.n <= 0) return cudaSuccess;
    if (cta && !table && !P.inst && !P.blists && P.chunk_cols <= 0 && P.chunk_slots <= 0) return cta_launch(P, st);
    if (P.inst) {
        if (table) return prod_launch<true, true, false>(P, st);
        return wide_window ? prod_launch<false, true, false, kBmWordsBig>(P, st) : prod_launch<false, true, false>(P, st);
    }
    if (table) return prod_launch<true, false, false>(P, st);
    if (P.blists) return prod_launch<false, false, true, kListWords>(P, st);
    // rows expected to span more columns than the bitmap covers: the wide
    // window (with every accumulator slot, as WIDE)
    if (wide_window) return prod_launch<false, false, true, kBmWordsBig>(P, st);
    // rows expected near or above the bitmap map's kAccCap - 32 slots: WIDE
    if (out_len > 0.9 * (kAccCap - 32)) return prod_launch<false, false, true>(P, st);
    return prod_launch<false, false, false>(P, st);
}

// In a batch with instances of both kinds the step is two launches, k_product
// and k_band, neither of which reads what the other writes.  k_band is
// launched programmatically, right behind its step's k_product (which itself is
// launched ordinarily: see pdl_enter): its blocks take the SMs that k_product's leave
// (each kernel's warps end at different times, a quarter of them idle on
// average), and it waits for k_product's end before it ends the step itself.
// 128 instances of 64-4096 rows: 17.6 -> 15.8 ms a call, 27: 5.1 -> 4.8 ms.
// (One launch that hands rows of both kinds to the same warps or SMs was
// slower, 19.4-23.3 ms: the two codes together outgrow an SM's instruction
// cache.)
template <bool BATCH, bool TEAM, int R>
static cudaError_t band_launch(const ProductArgs& P, cudaStream_t st) {
    const long long cap = (long long)sms_now() * 7, tiles = ((long long)P.n + R - 1) / R;
    const long long blocks = TEAM ? tiles : (tiles + kBandWarps - 1) / kBandWarps;
    const unsigned grid = (unsigned)(blocks < cap ? blocks : cap);
    ++g_launches;
    // (a batch's rows may be filtered when candidate lists are given)
    return launch_pdl(P.cand_col ? k_band<BATCH, TEAM, R, true> : k_band<BATCH, TEAM, R, false>, grid, kBandWarps * 32,
                      band_smem_bytes(), st, P);
}

cudaError_t launch_band(const ProductArgs& P, double row_len, cudaStream_t st) {
    if (P.n <= 0) return cudaSuccess;
    // The tile, measured over n = 256..100000 and rows of 5-600 columns.  TEAM
    // where a warp per tile leaves the chip idle or a tile is long (us, one
    // warp / team: n = 1000, 41 x 81 entries a row 43.5 / 29.1; n = 5000,
    // 101 x 101 210 / 189, 41 x 81 79 / 89; n = 10000, 201 x 201 1039 / 869,
    // 101 x 101 322 / 362).  Four rows a tile where they make about one round
    // of the chip's warps or several (one row / four: n = 2000, 31 x 61 36 /
    // 57; n = 12000 91 / 83; n = 20000, 1.2 rounds, 140 / 169; n = 65536
    // 408 / 375), and for rows of one 32-column piece, which are mostly
    // set-up (11 x 11: n = 12000 36 / 29, n = 65536 117 / 83).  A batch: four
    // rows from three rounds on where every instance is banded (ms a call, one
    // row / four: 25.6 k rows 5.07 / 5.62, 80 k 7.22 / 7.12, 131 k 13.1 / 12.8,
    // 320 k 26.2 / 24.5), one where k_product shares the step: the tiles then
    // take what SMs its rows leave, and the batch's tile of four rows spills
    // most (one row / four, rows of which banded: 26 k, 13 k 6.26 / 6.95; 26 k,
    // 18 k 4.79 / 4.94; 56 k, 35 k 12.7 / 13.8; 111 k, 83 k 15.8 / 16.3; 268 k,
    // 185 k 42.5 / 43.1).
    const double warps = sms_now() * 7.0 * kBandWarps;
    const double rounds = P.n / (4.0 * warps);  // of tiles of four rows
    const bool team = row_len > 300.0 || (row_len > 128.0 && P.n <= 5.0 * warps / kBandWarps) ||
                      (row_len > 80.0 && P.n <= 2.0 * warps / kBandWarps);
    if (P.inst) return !P.pair && rounds >= 3.0 ? band_launch<true, false, 4>(P, st) : band_launch<true, false, 1>(P, st);
    if (team) return rounds >= 0.9 ? band_launch<false, true, 4>(P, st) : band_launch<false, true, 1>(P, st);
    if (rounds >= (row_len <= 32.0 ? 0.35 : 3.0) || (rounds <= 1.0 && rounds >= 0.45))
        return band_launch<false, false, 4>(P, st);
    return band_launch<false, false, 1>(P, st);
}

cudaError_t launch_copy_result(int n, long long nnz, const int* rowptr, const int* col, const double* val,
                               int* d_rowptr, int* d_col, double* d_val, cudaStream_t st) {
    CopyArgs C{};
    const void* src[3] = {rowptr, col, val};
    void* dst[3] = {d_rowptr, d_col, d_val};
    const long long words[3] = {(long long)n + 1, nnz, 2 * nnz};
    long long most = 0;
    for (int a = 0; a < 3; ++a) {
        C.src[a] = static_cast<const unsigned*>(src[a]);
        C.dst[a] = static_cast<unsigned*>(dst[a]);
        C.words[a] = dst[a] ? words[a] : 0;
        most = most > C.words[a] ? most : C.words[a];
    }
    if (most == 0) return cudaSuccess;
    long long blocks = (most + 1023) / 1024;
    const long long cap = (long long)sms_now() * 8;
    if (blocks > cap) blocks = cap;
    launch_pdl(k_copy_result, (unsigned)blocks, 256, 0, st, C);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_row_lists(int n, const RowView& B, int2* hdr, uint2* lists, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long blocks = ((long long)n + 7) / 8;
    const long long cap = (long long)sms_now() * 8;
    if (blocks > cap) blocks = cap;
    launch_pdl(k_row_lists, (unsigned)blocks, 256, 0, st, n, B, hdr, lists);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_row_bitmaps(int n, const RowView& B, int2* hdr, unsigned* bits, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long blocks = ((long long)n + 7) / 8;
    const long long cap = (long long)sms_now() * 8;
    if (blocks > cap) blocks = cap;
    launch_pdl(k_row_bitmaps, (unsigned)blocks, 256, 0, st, n, B, hdr, bits);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_alg1(const Alg1Args& A, double entries, cudaStream_t st) {
    Alg1Args a = A;  // (cslot is 0: step_done)
    a.budget_ns = barrier_budget_ns();
    ++g_launches;
    if (dcfg().alg1_cluster > 0 && a.budget_ns > 0 && A.n <= kClusterColumns && entries <= kClusterEntries) {
        cudaLaunchConfig_t c{};
        c.gridDim = dim3((unsigned)dcfg().alg1_cluster);
        c.blockDim = dim3(kAlg1Threads);
        c.stream = st;
        cudaLaunchAttribute at[2]{};
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c.gridDim.x;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        c.attrs = at;
        c.numAttrs = 2;
        return cudaLaunchKernelEx(&c, k_alg1<true>, a);
    }
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel((const void*)k_alg1<false>, dim3(dcfg().alg1_blocks), dim3(kAlg1Threads), args,
                                       0, st);
}

cudaError_t launch_norms(const NormArgs& A, cudaStream_t st) {
    NormArgs a = A;
    a.budget_ns = barrier_budget_ns();
    void* args[] = {&a};
    ++g_launches;
    return cudaLaunchCooperativeKernel((const void*)k_norms, dim3(dcfg().norm_blocks), dim3(kNormThreads), args,
                                       0, st);
}

cudaError_t launch_absmax(const double* pool_val, const Ctl* ctl, int i, NormSlot* slot, cudaStream_t st) {
    launch_pdl(k_absmax, sms_now() * 4, 256, 0, st, pool_val, ctl, i, slot);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_validate(int n, int nnz, const int* rowptr, const int* col, const double* val, Ctl* ctl,
                            cudaStream_t st) {
    int blocks = (n + 1 + 255) / 256;
    launch_pdl(k_validate, blocks, 256, 0, st, n, nnz, rowptr, col, val, ctl);
    ++g_launches;
    return cudaGetLastError();
}

size_t scan_scratch_len(int n) { return (size_t)((n + kScanTile - 1) / kScanTile) + 2; }

cudaError_t launch_scan_rows(int n, const int* rb, const int* re, const RowDesc* rd, int* rowptr, Ctl* ctl,
                             long long* sums, cudaStream_t st) {
    const int ntiles = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
    launch_pdl(k_scan_tile_sums, ntiles, kScanTile, 0, st, n, rb, re, rd, sums, ctl);
    ++g_launches;
    launch_pdl(k_scan_apply, ntiles, kScanTile, 0, st, n, rb, re, rd, sums, rowptr);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_gather(int n, const RowView& src, const int* rowptr, int* col, double* val,
                          cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int blocks = (n + 7) / 8;
    if (blocks > sms_now() * 16) blocks = sms_now() * 16;
    launch_pdl(k_gather, blocks, 256, 0, st, n, src, rowptr, col, val);
    ++g_launches;
    return cudaGetLastError();
}

// FP64 rate probe: every thread runs eight independent chains of fused
// multiply-adds (enough in flight to fill the pipe); the result is stored so
// that none of the work can be dropped.
// (Measured on GB300: this form reaches 1.257 TFLOP/s at 2070 MHz, 99.9 %
// of the unit count; a form with __fma_rn and the output pointer last was
// scheduled differently and reached only 1.01-1.06.)
__global__ void k_fp64_probe(double* out, int iters, double a, double b) {
    double x0 = threadIdx.x * 1e-3, x1 = x0 + 1, x2 = x0 + 2, x3 = x0 + 3, x4 = x0 + 4, x5 = x0 + 5, x6 = x0 + 6,
           x7 = x0 + 7;
    for (int i = 0; i < iters; ++i) {
        x0 = fma(x0, a, b);
        x1 = fma(x1, a, b);
        x2 = fma(x2, a, b);
        x3 = fma(x3, a, b);
        x4 = fma(x4, a, b);
        x5 = fma(x5, a, b);
        x6 = fma(x6, a, b);
        x7 = fma(x7, a, b);
    }
    out[blockIdx.x * blockDim.x + threadIdx.x] = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
}

int fp64_probe_blocks() { return sms_now() * 4; }

cudaError_t launch_fp64_probe(int iters, double* out, cudaStream_t st) {
    k_fp64_probe<<<fp64_probe_blocks(), 256, 0, st>>>(out, iters, 0.999999, 1e-7);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_identity(int n, double alpha, int* rowptr, int* col, double* val, cudaStream_t st) {
    launch_pdl(k_identity, (n + 1 + 255) / 256, 256, 0, st, n, alpha, rowptr, col, val);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_copy_rows(int n, const int* rowptr, const int* col, const double* val, int* rb, int* re,
                             RowDesc* rd, int* pool_col, double* pool_val, Ctl* ctl, unsigned long long arena_size,
                             NormSlot* absmax, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    // about four rows per warp: each row is a dependent load pair, so the
    // copy is latency-bound and wants many warps in flight
    long long blocks = ((long long)n + 31) / 32;
    if (blocks > (long long)sms_now() * 8) blocks = (long long)sms_now() * 8;
    launch_pdl(k_copy_rows, (unsigned)blocks, 256, 0, st, n, rowptr, col, val, rb, re, rd, pool_col, pool_val, ctl,
                                                  arena_size, absmax);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_norm_scratch_init(Ctl* ctl, NormSlot* slot, unsigned long long* words, unsigned* sticky, int n,
                                     long long nnz, cudaStream_t st) {
    int blocks = (int)(((long long)kChunks * n + 255) / 256);
    if (blocks < 1) blocks = 1;
    if (blocks > sms_now() * 4) blocks = sms_now() * 4;
    launch_pdl(k_norm_scratch_init, blocks, 256, 0, st, ctl, slot, words, sticky, n, nnz);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_norm_in_place(Ctl* ctl, NormSlot* slot, unsigned long long* words, unsigned* sticky,
                                 const psf_csr_t& M, cudaStream_t st) {
    cudaError_t err = launch_norm_scratch_init(ctl, slot, words, sticky, M.n, M.nnz, st);
    if (err == cudaSuccess) err = launch_validate(M.n, M.nnz, M.rowptr, M.col, M.val, ctl, st);
    if (err == cudaSuccess) err = launch_absmax(M.val, ctl, 0, slot, st);
    if (err != cudaSuccess) return err;
    NormArgs na{};
    na.n = M.n;
    na.count = 1;
    na.pool_col = M.col;
    na.pool_val = M.val;
    na.slots = slot;
    na.words = words;
    na.sticky = sticky;
    na.ctl = ctl;
    return launch_norms(na, st);
}

cudaError_t launch_alg1_batch(const Alg1BatchArgs& A, cudaStream_t st) {
    if (A.ninst > kMaxBatch) return cudaErrorInvalidValue;
    Alg1BatchArgs a = A;  // (cslot is 0: step_done)
    a.budget_ns = barrier_budget_ns();
    void* args[] = {&a};
    ++g_launches;
    return cudaLaunchCooperativeKernel((const void*)k_alg1_batch, dim3(dcfg().alg1b_blocks), dim3(kAlg1Threads), args,
                                       0, st);
}

cudaError_t launch_inst_table(int n, int ninst, const int* off, int* inst, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_inst_table, (n + 255) / 256, 256, 0, st, n, ninst, off, inst);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_count_apart(const psf_csr_t& A, const psf_csr_t& B, bool series, Ctl* ctl, cudaStream_t st) {
    if (A.n <= 0) return cudaSuccess;
    launch_pdl(k_count_apart, (unsigned)((A.n + 255) / 256), 256, 0, st, A.n, A.rowptr, A.col, B.rowptr, B.col,
               series ? 1 : 0, ctl);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_count_apart_batch(int n, const int* inst, const BatchSrc* src, unsigned* count, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_count_apart_batch, (unsigned)((n + 255) / 256), 256, 0, st, n, inst, src, count);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_validate_batch(int n, const int* inst, const BatchSrc* src, const int* nnz, Ctl* ctl,
                                  unsigned char* band, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_validate_batch, (n + 255) / 256, 256, 0, st, n, inst, src, nnz, ctl, band);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_copy_rows_batch(int n, const int* inst, const BatchSrc* src, int* rb, int* re, RowDesc* rd,
                                   int* pool_col, double* pool_val, Ctl* ctl, unsigned long long arena_size, NormSlot* absmax,
                                   int stride, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int blocks = (n + 7) / 8;
    if (blocks > sms_now() * 8) blocks = sms_now() * 8;
    launch_pdl(k_copy_rows_batch, blocks, 256, 0, st, n, inst, src, rb, re, rd, pool_col, pool_val, ctl, arena_size, absmax,
                                              stride);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_compose_rows(int n, const int* inst, const int* sel, const RowDesc* const* rds, int count,
                                int* out_rb, int* out_re, RowDesc* out_rd, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (count > kMaxAdd + 2) return cudaErrorInvalidValue;
    RowTable T{};
    for (int k = 0; k < count; ++k) T.rd[k] = rds[k];
    launch_pdl(k_compose_rows, (n + 255) / 256, 256, 0, st, n, inst, sel, T, out_rb, out_re, out_rd);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_gather_batch(int n, int ninst, const int* inst, const int* off, const RowView& src,
                                const int* rowptr, int* out_rp, int* col, double* val, cudaStream_t st) {
    int blocks = (n + 7) / 8;
    if (blocks < 1) blocks = 1;
    if (blocks > sms_now() * 16) blocks = sms_now() * 16;
    launch_pdl(k_gather_batch, blocks, 256, 0, st, n, ninst, inst, off, src, rowptr, out_rp, col, val);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_bounds(int ninst, const int* off, const int* rowptr, int* bounds, cudaStream_t st) {
    launch_pdl(k_bounds, (ninst + 1 + 255) / 256, 256, 0, st, ninst, off, rowptr, bounds);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_reuse_copy_batch(const ProductArgs& P, cudaStream_t st) {
    if (P.n <= 0) return cudaSuccess;
    long long blocks = ((long long)P.n + 7) / 8;
    const long long cap = (long long)num_sms() * 8;
    if (blocks > cap) blocks = cap;
    launch_pdl(k_reuse_copy_batch, (unsigned)blocks, 256, 0, st, P);
    return cudaGetLastError();
}

cudaError_t launch_reset(Ctl* ctl, unsigned long long cap, unsigned long long cand_cap, unsigned cand_chunk,
                         cudaStream_t st) {
    launch_pdl(k_reset, 1, 32, 0, st, ctl, cap, cand_cap, cand_chunk);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_export(const void* src, void* dst, size_t bytes, cudaStream_t st) {
    launch_pdl(k_export, 1, 256, 0, st, static_cast<const unsigned*>(src), static_cast<unsigned*>(dst), (int)(bytes / 4));
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_reuse_pass1(const ReuseArgs& R, cudaStream_t st) {
    if (R.n <= 0) return cudaSuccess;
    int blocks = (R.n + 7) / 8;
    if (blocks > sms_now() * 8) blocks = sms_now() * 8;
    launch_pdl(k_reuse_pass1, blocks, 256, 0, st, R);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_norms_rows(const NormRowsArgs& A, cudaStream_t st) {
    if (A.n <= 0 || A.count <= 0) return cudaSuccess;
    dim3 grid((unsigned)((A.n + kNormTile - 1) / kNormTile), (unsigned)A.count);
    launch_pdl(k_norms_rows, grid, kNormRowsThreads, norms_rows_smem_bytes(), st, A);
    ++g_launches;
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    const long long total = (long long)A.count * (((long long)A.n + 31) & ~31LL);
    long long blocks = (total + 255) / 256;  // one (matrix, column) per thread
    if (blocks > 65535LL * 64) blocks = 65535LL * 64;
    launch_pdl(k_norms_finish, (unsigned)blocks, 256, 0, st, A.n, A.count, A.slots, A.words, A.sticky, A.ctl, A.inst,
                                                     A.slot_stride);
    ++g_launches;
    return cudaGetLastError();
}


}  // namespace psf
