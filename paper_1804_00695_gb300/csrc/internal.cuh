// Internal definitions shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string>
#include <vector>
#include <algorithm>
#include "../../include/spgemm.h"

namespace sg {

// ---------------------------------------------------------------- errors
void set_error(const char *fmt, ...);
#define SG_CUDA(call)                                                          \
    do {                                                                       \
        cudaError_t e_ = (call);                                               \
        if (e_ != cudaSuccess) {                                               \
            ::sg::set_error("%s failed: %s (%s:%d)", #call,                    \
                            cudaGetErrorString(e_), __FILE__, __LINE__);       \
            return SPGEMM_ERR_CUDA;                                            \
        }                                                                      \
    } while (0)
#define SG_TRY(expr)                                                           \
    do {                                                                       \
        int s_ = (expr);                                                       \
        if (s_ != SPGEMM_OK) return s_;                                        \
    } while (0)

// Device-side error bits (OR-ed into DevState::err by kernels).
enum : int {
    DERR_COL_RANGE = 1,   // a column index of A (>= nrows(B)) or B (>= ncols) out of range
    DERR_PROBE = 2,       // a hash probe sequence exceeded the table
    DERR_COUNT = 4,       // numeric found a different column count than symbolic
    DERR_WINDOW = 8,      // chunked: a column of A outside the rows of B copied for its part
};

constexpr int CLS_SLOTS = 24;   // classes the device state has room for

struct DevState {          // lives in device memory, one per handle
    int err;
    int b_out_of_range;    // B holds values outside the double-word range
    long long sym_hist[SPGEMM_NBINS];   // rows per symbolic bin (by bound)
    long long nnz;         // nnz(C) written by the scan
    long long bin_count[2][SPGEMM_NBINS];   // [0] symbolic, [1] numeric
    long long bin_cursor[SPGEMM_NBINS];
    long long max_row_nnz;   // largest row of C (numeric binning)
    long long flops_total;   // products of the whole product (analysis)
    int b_unsorted;          // some row of B has columns out of ascending order
    int long_rows[2];        // rows the compression left to its second pass: to a warp each, to a block each
    long long max_alen;      // longest row of A (analysis)
    unsigned long long triangles;   // spgemm_triangles: the count
    // numeric rows by class (NumCls): rows, list cursors, largest row of C,
    // largest column span in 32-column blocks
    long long cls_count[CLS_SLOTS];
    long long cls_cursor[CLS_SLOTS];
    int cls_nnz[CLS_SLOTS], cls_words[CLS_SLOTS];
    unsigned long long narrow_flops;   // products of the rows of CLS_NARROW
    unsigned long long next_row;   // rows a kernel has handed out (cleared before it)
    // symbolic phase: whether the 32-slot maps have rows, whether rows are
    // marked; rows of the warps, of the blocks' bitmaps and of the blocks' maps
    int sym_first, sym_marked;
    unsigned long long sym_warp, sym_block, sym_map;   // sym_map: rows of a block's map
    unsigned long long next_map;   // rows of those handed out
};

// ---------------------------------------------------------------- bins
// Rows are binned by the size of the accumulator they need and by their
// product count; each bin has its own kernel shape (Section 3.3: a part of a
// warp, a whole warp or a whole block per row).
constexpr int BIN_EMPTY = 0;
constexpr int BIN_HUGE = 6;     // widest bin: unbounded accumulator
constexpr int NBINS = SPGEMM_NBINS;

// Symbolic phase of a B of at most SYM_BITMAP_WORDS blocks of 32 columns (its
// bitmap fits a block's shared memory), rows that are not narrow, by their
// compressed pairs and the blocks they span (sym_mark; the mark is kept in
// crp[i+1] until the row is counted):
//   at most SYM_FIRST_PAIRS pairs: a 32-slot map, which holds them whatever
//     their blocks (no mark);
//   SYM_MARK_WARP: up to SYM_WARP_PAIRS pairs over at most SYM_WARP_WORDS
//     blocks: a warp and a bitmap of the span; over more, up to SYM_MAP_PAIRS, or
//     SYM_MAP_WIDE_PAIRS over more than SYM_MAP_WIDE_WORDS: a warp and a map;
//   SYM_MARK_MAP: up to SYM_MAP_BLOCK_PAIRS pairs, and one for 28 blocks of the
//     span, over more than SYM_MAP_BLOCK_WORDS: a block and a map;
//   SYM_MARK_BLOCK: the others: a block and a bitmap.
// Why the lines lie there (one GB300, whole symbolic call): a block's bitmap is
// cleared and counted over the whole span, and from 24,576 blocks on one fills
// an SM, so that rows go through it one at a time.  Bitmap -> map, rows over
// 3000 / 12,000 / 50,000 blocks: 200,000 of 40 pairs 784 -> 347, 1613 -> 353,
// 5509 -> 355 us; 78,125 of 256 417 -> 323, 738 -> 336, 2295 -> 340; 66,666 of 300
// 370 (bitmap kept), 650 -> 305, 1979 -> 316; 150,000 of 600 758 (kept), 1364 ->
// 1195, 4409 -> 1267; 20,000 of 1000 214 and 305 (kept), 729 -> 401; 50,000 of 1500
// 409 and 660 (kept), 1679 -> 1094.  (A hundred rows of 400 take 101 by bitmaps, 111
// by maps, of 600 100 and 124; a warp's map of 700 pairs, 0.7 full, takes 1.69 ms for
// 150,000 rows over 10,000 blocks where bitmaps take 1.40.)
// A wider B goes through the optimistic first pass and the lists by bin.
constexpr int64_t SYM_BITMAP_WORDS = 53248;   // 208 KB
constexpr int SYM_WARP_WORDS = 2048;
constexpr long long SYM_FIRST_PAIRS = 32, SYM_WARP_PAIRS = 4096;
constexpr long long SYM_MAP_PAIRS = 256, SYM_MAP_WIDE_PAIRS = 640, SYM_MAP_BLOCK_PAIRS = 2048;
constexpr int SYM_MAP_L = 10, SYM_MAP_BLOCK_L = 12;   // slots of the largest maps (log2): two for every pair
constexpr int SYM_MAP_WIDE_WORDS = 8192, SYM_MAP_BLOCK_WORDS = 12288;
static_assert((2 << SYM_MAP_L) <= SYM_WARP_WORDS, "a warp's map lies where its bitmap does");
constexpr int SYM_MARK_WARP = -1, SYM_MARK_BLOCK = -2, SYM_MARK_MAP = -3;
__host__ __device__ inline int sym_mark(long long cpairs, int words) {
    if (cpairs <= SYM_FIRST_PAIRS) return 0;
    if (words <= SYM_WARP_WORDS) return cpairs <= SYM_WARP_PAIRS ? SYM_MARK_WARP : SYM_MARK_BLOCK;
    if (cpairs <= (words > SYM_MAP_WIDE_WORDS ? SYM_MAP_WIDE_PAIRS : SYM_MAP_PAIRS)) return SYM_MARK_WARP;
    return words > SYM_MAP_BLOCK_WORDS && cpairs <= SYM_MAP_BLOCK_PAIRS && cpairs * 28 <= words ? SYM_MARK_MAP : SYM_MARK_BLOCK;
}

// Numeric bins by exact output count (and product count):
//   1: <= 16 entries, 2: <= 32 (both: lanes of a warp, map in shared memory,
//   rows taken in order), 3: <= 128 (a warp), 4: <= 1024, 5: <= 4096 (a
//   block), 6: larger (a block with a global second-level map).
__host__ __device__ constexpr long long num_cap(int b) {
    return b == 1 ? 16 : b == 2 ? 32 : b == 3 ? 128 : b == 4 ? 1024 : b == 5 ? 4096 : (1LL << 40);
}
__host__ __device__ constexpr long long num_flops(int b) {
    return b <= 2 ? 8192 : b == 3 ? 65536 : b == 4 ? 1048576 : b == 5 ? 16777216 : (1LL << 62);
}
__host__ __device__ inline int num_bin(long long nnz, long long flops) {
    if (nnz <= 0) return BIN_EMPTY;
    int b = 1;
    while (b < BIN_HUGE && (nnz > num_cap(b) || flops > num_flops(b))) b++;
    return b;
}

// Symbolic bins by an upper bound on the row's distinct column blocks:
// every row with bound <= 4096 is first tried with a 32-slot map (most rows
// of sparse products have few blocks); rows that overflow it, and rows with
// a larger bound, go to 2: <= 64 keys, 3: <= 256 (a warp), 4: <= 1024,
// 5: <= 4096 (a block), 6: dense bitmap of all blocks (a block).
constexpr int SYM_FIRST_SLOTS = 32;
__host__ __device__ constexpr long long sym_cap(int b) {
    return b == 1 ? 16 : b == 2 ? 64 : b == 3 ? 256 : b == 4 ? 1024 : b == 5 ? 4096 : (1LL << 40);
}
__host__ __device__ inline int sym_bin(long long keys, long long cpairs) {
    if (keys <= 0) return BIN_EMPTY;
    int b = 1;
    while (b < BIN_HUGE && (keys > sym_cap(b) || cpairs > 64 * sym_cap(b))) b++;
    return b;
}

// Class of a row of numeric bins 2..6: the kernel that takes it, given by
// its outputs, its column span and its products.  The lists of the numeric
// phase are in class order.
//   CLS_B2      bin 2 (a list only when the small-row kernel stops at 16)
//   CLS_WINDOW_W, CLS_WINDOW_B  narrow rows of 33 to WINDOW_NNZ outputs whose
//               word list the symbolic phase left whole: a warp, or from
//               WINDOW_FLOPS products on a block
//   CLS_NARROW  BIN_NARROW (a list only when other rows lie between them)
//   CLS_RANK_W  at most RANK_W_FLOPS products over at most RANK_M_WORDS blocks
//   CLS_RANK_S  at most RANK_S_NNZ outputs over at most RANK_S_WORDS blocks
//   CLS_RANK_V  at most RANK_V_FLOPS products over wider spans up to
//               RANK_M_WORDS blocks
//   CLS_RANK_M4, CLS_RANK_M5  other rows over spans up to RANK_M_WORDS blocks: rows
//               of at most RANK_S_NNZ outputs, and of at most RANK_M_NNZ
//   CLS_WIDE3 .. CLS_WIDE4C   other rows of bins 3 and 4 by outputs
//   CLS_BLOCK, CLS_HUGE       other rows of bins 5 and 6
//   CLS_DENSE   rows of B sorted: rows with many products over their span
//   CLS_DENSE_D, CLS_DENSE, CLS_DENSE_F, CLS_DENSE_S  rows of B sorted: rows with
//               more outputs than the rank accumulators hold, by the types in which
//               dense windows cost less than cursors: FP64 only, both, FP32
//               only (or the row may need folds), neither; see dense_by_window
// Why the lines lie there: 512 products are eight a lane for the two warps of
// a short row (rank.cu has both sides; 8192 blocks keep its first bitmap
// within 1.5 KB), 1024 eight for four warps (13,774 rows of 513 to 1024 FP32
// products over 3125 blocks 228 -> 89 us against CLS_RANK_M4; within 2048
// blocks CLS_RANK_S is the faster, 0.66 against 0.73 ms for 124,998 rows);
// 2048 blocks are the bitmap that 128 threads scan in
// one step of 16 words, 8192 the one that 512 threads do; a row of 8192 FP64
// outputs over 8192 blocks takes 167 KB of shared memory, the next power of
// two would not fit.  Below them the rank accumulators measured 2.6-5x
// faster than the maps and windows (rank.cu has the figures).
enum NumCls {
    CLS_NONE = 0, CLS_B2, CLS_WINDOW_W, CLS_WINDOW_B, CLS_RANK_W, CLS_RANK_S, CLS_RANK_V, CLS_RANK_M4, CLS_RANK_M5, CLS_WIDE3, CLS_WIDE4A, CLS_WIDE4B, CLS_WIDE4C,
    CLS_BLOCK, CLS_DENSE_D, CLS_DENSE, CLS_DENSE_F, CLS_DENSE_S,
    CLS_HUGE, CLS_NARROW, NCLS
};
static_assert(NCLS <= CLS_SLOTS, "DevState keeps the classes' counts");
constexpr int RANK_S_NNZ = 1024, RANK_S_WORDS = 2048, RANK_M_NNZ = 8192, RANK_M_WORDS = 8192;
constexpr int RANK_W_FLOPS = 512, RANK_V_FLOPS = 1024;
constexpr long long RANK_FLOPS = 1LL << 24;   // products (their prefix sums fit 32 bits)
// Dense windows from one product per 8 columns of the span on (their cost per
// row is the span written out plus the products, the rank accumulators' the
// products twice over) and above the 6144 products that a rank block keeps in
// registers: A*A of R-MAT graphs, FP64, scale 16 with 12 edges a vertex 11.9
// ms (one per 4 columns 12.4), scale 15 with 5 2.91 (2.94, one per 2 3.02).
constexpr long long DENSE_FLOPS = 6144;
// Rows with more outputs than the rank accumulators hold choose between the dense
// windows and the windows walked by cursors (k_num_window) by what either costs:
// its columns written out, every entry of the row of A staged (or its cursor
// looked at) in every window, and the products; the cursors' entries more where
// rows of B of over 256 entries go to a warp each.  The weights (0.1 ps of the chip
// for a row, rows enough to fill it) are least-squares fits to 84 measured products
// a kernel and type, spans of 9000 to 4 M columns, rows of B of 2 to 5000, 1 to 64
// columns a product: two of three within 13%, all within 45%; the choice costs 1%
// over the better kernel in the mean, 24% at worst.  Cursors -> dense, 2000 rows
// over rows of B of 64, a product per c columns (ms): 262,144
// columns FP32 c 6 2.00 -> 1.42, 12 1.08 -> 1.02, 16 0.77 -> 0.95, 24 0.60 -> 0.88
// (FP64 2.59 -> 2.30, 1.54 -> 1.36, 1.09 -> 1.25, 0.93 -> 1.15); 1,048,576 columns,
// c 10 4.5 -> 5.3 (6.7 -> 9.5), with rows of B of 1000 4.7 -> 2.0 (9.5 -> 2.7);
// 10,000,000 columns, 10,000 products a row 7.2 -> 22.8 (14.2 -> 30.9).
// Rows that fit the chip at once in dense windows (DENSE_FEW for each SM) take them
// all the same: 40 rows over 524,288 columns, c 16 0.38 -> 0.23 ms, over 4,194,304,
// c 64 3.0 -> 1.9; and so do all where the cursors' workspace has no room.  In FP32
// a row that may hold sums long enough for folds (dense.cu) keeps them.
// Rows of at most RANK_M_NNZ outputs over rows of B of a few entries choose between
// dense windows and the rank accumulators in the same way (2000 rows of 4000
// entries of two products, FP32, over 40,000 columns 574 us by dense windows, 428 by
// rank, over 20,000 331 by dense windows; of 3250 entries over 9000 351 by rank, over
// 60,000 356).
constexpr int DENSE_BYTES = 88 * 1024;   // a window's accumulators
constexpr int DENSE_FEW = 2;
constexpr int DENSE_FOLD_ALEN = 1024;    // entries of a row of A from which on folds begin
constexpr int DENSE_FOLD_TERMS = 2048;   // a sum of so many terms is folded whatever the window
constexpr int WINDOW_NNZ = 256;
constexpr long long WINDOW_FLOPS = 4096;
__host__ __device__ inline long long dense_cost(int vb, long long span, long long alen, long long flops) {
    const long long w = DENSE_BYTES / vb, n = (span + w - 1) / w;
    return vb == 4 ? 13 * span + 281 * alen * n + 38 * flops
                   : 17 * span + (152 + 26 * (n < 32 ? n : 32) / 10) * alen * n + 63 * flops;
}
__host__ __device__ inline long long cursor_cost(int vb, long long span, long long alen, long long flops) {
    const long long w = 32768 / vb, n = (span + w - 1) / w;
    const bool warps = flops > 256 * alen;
    return vb == 4 ? 2 * span + (warps ? 2200 : 63) * alen * n + (warps ? 147 : 184) * flops
                   : 5 * span + (warps ? 2700 : 62) * alen * n + (warps ? 160 : 214) * flops;
}
// listed: the row is narrow and its words are all in its list; alen: entries of
// the row of A (read for bins 5 and 6 only).
__host__ __device__ inline int num_cls(int bin, long long nnz, long long flops, int words, bool listed, bool dense_ok,
                                       long long alen) {
    if (bin < 2) return CLS_NONE;
    if (bin == 7) return CLS_NARROW;
    if (bin == 2) return CLS_B2;
    if (listed && nnz <= WINDOW_NNZ) return flops < WINDOW_FLOPS ? CLS_WINDOW_W : CLS_WINDOW_B;
    if (dense_ok && bin >= 5 && words > 0 && flops < (1LL << 31)) {
        const long long span = (long long)words * 32;
        const bool folds = alen > DENSE_FOLD_ALEN && flops - nnz >= DENSE_FOLD_TERMS;
        if (nnz <= RANK_M_NNZ) {
            bool dense = flops > DENSE_FLOPS && flops * 8 >= span;
            if (flops < 6 * alen && words <= RANK_M_WORDS && !folds)   // short rows of B
                dense = dense_cost(4, span, alen, flops) <= 98 * flops + 370 * alen;
            if (dense) return CLS_DENSE;
        } else {
            const bool d = dense_cost(8, span, alen, flops) <= cursor_cost(8, span, alen, flops);
            const bool f = folds || dense_cost(4, span, alen, flops) <= cursor_cost(4, span, alen, flops);
            return f ? (d ? CLS_DENSE : CLS_DENSE_F) : d ? CLS_DENSE_D : CLS_DENSE_S;
        }
    }
    if (words > 0 && flops <= RANK_FLOPS) {
        if (flops <= RANK_W_FLOPS && words <= RANK_M_WORDS) return CLS_RANK_W;
        if (nnz <= RANK_S_NNZ && bin <= 4 && words <= RANK_S_WORDS) return CLS_RANK_S;
        if (flops <= RANK_V_FLOPS && words <= RANK_M_WORDS) return CLS_RANK_V;
        if (nnz <= RANK_S_NNZ && bin <= 4 && words <= RANK_M_WORDS) return CLS_RANK_M4;
        if (nnz <= RANK_M_NNZ && words <= RANK_M_WORDS) return CLS_RANK_M5;
    }
    if (bin == 3) return CLS_WIDE3;
    if (bin == 4) return nnz <= 256 ? CLS_WIDE4A : nnz <= 512 ? CLS_WIDE4B : CLS_WIDE4C;
    return bin == 5 ? CLS_BLOCK : CLS_HUGE;
}

// Narrow rows (narrow.cu): rows of C whose columns all fall within
// NARROW_W consecutive blocks of 32 columns.  The symbolic phase marks them
// BIN_NARROW (their count done by the window table, nlo[i] = the window's
// first block); the numeric phase gives BIN_NARROW to those of them with at
// most NARROW_NMAX outputs and NARROW_FLOPS products.  Bin 7 is otherwise
// unused in both phases.
constexpr int BIN_NARROW = 7;
constexpr int NARROW_W = 128;
constexpr int NARROW_NMAX = 32;
constexpr long long NARROW_FLOPS = 8192;
constexpr long long NARROW_PAIRS = 4096;
// Row-slot strides of the narrow kernels' shared tables, padded so that the
// row slots of a warp start on different banks (words, bytes, values).
constexpr int NARROW_TAB_STRIDE = NARROW_W + 4;
constexpr int NARROW_BASE_STRIDE = NARROW_W + 4;
constexpr int NARROW_ACC_STRIDE = NARROW_NMAX + 1;

// Blocks of a kernel that fit an SM with `threads` threads and `smem` bytes of
// dynamic shared memory (which the kernel is opted in to).  The driver is asked
// once for each of a kernel's last few shapes on a device; the answers are
// shared by all handles and threads.
int kernel_blocks_per_sm(const void *kern, int threads, size_t smem, int *per_sm);

// Blocks of `kern` that fit on all SMs at once (at least one per SM): the
// kernels that stride over their rows run one resident wave.
template <typename K>
static inline int64_t resident_blocks(K kern, int threads, int nsm) {
    int per_sm = 0;
    if (kernel_blocks_per_sm((const void *)kern, threads, 0, &per_sm) != SPGEMM_OK) per_sm = 1;
    return (int64_t)per_sm * nsm;
}

// Adds this warp's per-bin row counts (bins held by the lanes where `has`)
// to a shared histogram with one ballot per bin.
__device__ __forceinline__ void warp_hist(unsigned long long *hist, bool has, int bin) {
    const unsigned have = __ballot_sync(0xffffffffu, has);
    if (!have) return;
    for (int b = 0; b < NBINS; b++) {
        unsigned m = __ballot_sync(0xffffffffu, has && bin == b);
        if (m && (threadIdx.x & 31) == 0) atomicAdd(&hist[b], (unsigned long long)__popc(m));
    }
}

// Multiplicative hash (Fibonacci) of a non-negative key into [0, 2^log2S).
__device__ __forceinline__ unsigned hash_slot(int key, int log2S) {
    return ((unsigned)key * 0x9E3779B1u) >> (32 - log2S);
}

// Insert block `blk` with mask m into a map of 2^L slots; false if full.
__device__ __forceinline__ bool sym_insert(int *keys, unsigned *masks, int L, int blk, unsigned m) {
    const unsigned msk = (1u << L) - 1;
    unsigned h = hash_slot(blk, L);
#pragma unroll 1
    for (int probe = 0; probe <= (int)msk; probe++) {
        int k = ((volatile int *)keys)[h];
        if (k == blk) {
            atomicOr(&masks[h], m);
            return true;
        }
        if (k == -1) {
            int old = atomicCAS(&keys[h], -1, blk);
            if (old == -1 || old == blk) {
                atomicOr(&masks[h], m);
                return true;
            }
        }
        h = (h + 1) & msk;
    }
    return false;
}

// ---------------------------------------------------------------- launch context
// Every kernel launch goes through a Ctx: it carries the stream and SM count,
// counts launches, and (when timing is on) brackets each launch with CUDA
// events recorded on the launching stream, labelled "<phase>.<kernel>".
struct TimingRec {
    const char *label;
    long long rows;
    cudaEvent_t e0, e1;
};

struct Ctx {
    cudaStream_t s = nullptr;
    int nsm = 0;
    long long *launches = nullptr;
    int timing = 0;                // 0 off, 1 every kernel, 2 numeric-phase kernels only
    bool open = false;             // begin() recorded the current pair's first event
    TimingRec *recs = nullptr;     // handle-owned ring of event pairs
    int *nrec = nullptr;
    int cap = 0;
    const char *phase = "";
    void begin(const char *label, long long rows);
    void end();
};

// ---------------------------------------------------------------- launchers
// analyze.cu
// Compressed column sets (Section 2.1): pairs of row k sit at
// pairs[M.row_ptr[k] .. M.row_ptr[k] + ccnt[k]), each {block, mask};
// minmax[k] = {first block, last block} ({INT_MAX, INT_MIN} for empty rows);
// desc[k] = {row_ptr[k] low, high 32 bits, entries, pairs};
// ana[k] = {entries, pairs}.  Any output may be NULL.
// `unsorted` (may be null) is set to 1 if a row of M is not strictly ascending.
// `long_count` (device, two, cleared by the caller before the call) and
// `long_list` (room for M.nrows): the rows left to the second pass.
int launch_compress(const spgemm_csr &M, int2 *pairs, int32_t *ccnt, int2 *minmax, int4 *desc,
                    int2 *ana, int *err, int *long_count, int32_t *long_list, Ctx &c, int *unsorted = nullptr);
__device__ __forceinline__ int64_t desc_start(int4 d) {
    return (int64_t)(((uint64_t)(unsigned)d.y << 32) | (uint64_t)(unsigned)d.x);
}
size_t scan_tmp_bytes(int64_t n);
size_t scan_binning_tmp_bytes(int64_t n);   // launch_scan_binning
// x[0..n] holds counts in x[1..n]; on return x is the exclusive prefix
// (x[0] = 0); *total (device) = x[n].
int launch_scan_counts(int64_t *x, int64_t n, long long *total, void *tmp, Ctx &c);
// Per row i of A: flops, symbolic bin, column-block span rspan[i] = {first
// block, blocks} of the rows of B it reaches ({INT_MAX, 0} if none; bmm[k] =
// {first block, last block} of B_k); empty rows get crp[i+1] = 0.  bitmaps: B fits
// SYM_BITMAP_WORDS, and rows get their mark (sym_mark) in crp[i+1]; a row with
// a column of A out of range gets 0 then (no kernel may read it).
int launch_analyze(const spgemm_csr &A, const spgemm_csr &B, const int2 *ana, const int2 *bmm, int64_t *flops,
                   uint8_t *bins, int64_t *crp, int2 *rspan, DevState *st, bool bitmaps, Ctx &c);
// launch_scan_counts of the counts of C's rows into st->nnz, and in the same
// pass the numeric bin of every row from its outputs and flops; rows the
// symbolic phase found narrow (nlo[i] >= 0; nlo may be null) that fit the
// narrow numeric kernel get BIN_NARROW.  cls[i]: the row's class (num_cls);
// rows, largest row and span per class in st.
int launch_scan_binning(int64_t *crp, int64_t n, void *tmp, const int64_t *arp, const int64_t *flops, uint8_t *bins,
                        uint8_t *cls, const int2 *rspan, const int32_t *nlo, const uint8_t *nwords, DevState *st, bool dense_ok,
                        Ctx &c);
// Row lists of the symbolic second pass by bin: rows[offset(b) + t], offsets
// from st->bin_count[0].
int launch_scatter_bins(int64_t n, const uint8_t *bins, const int64_t *crp, int32_t *rows, DevState *st, Ctx &c);
// Row lists of the numeric phase by class (classes first_cls and up), offsets
// from st->cls_count.
int launch_scatter_cls(int64_t n, const uint8_t *cls, int32_t *rows, DevState *st, int first_cls, Ctx &c);
int launch_row_flops(const spgemm_csr &A, const spgemm_csr &B, int64_t *flops, int *err, Ctx &c);

// narrow.cu
// Analysis of every row of A (flops, symbolic bin, as launch_analyze) with
// the count of every narrow row done in the same pass (bins[i] =
// BIN_NARROW, nlo[i] = first block of its window; nlo[i] = -1 otherwise).
// bmm[k] = {first block, last block} of B_k; G lanes per row (4..32).
// A narrow row also leaves its non-empty window words, in order, at
// ulist[i*NARROW_NMAX ...] (first NARROW_NMAX of them; {word | rank of its
// first column << 8, mask}) and their number in nwords[i].
int launch_sym_narrow(const spgemm_csr &A, const spgemm_csr &B, const int4 *desc, const int2 *bmm,
                      const int2 *pairs, int64_t *flops, uint8_t *bins, int64_t *crp, int2 *rspan, int32_t *nlo,
                      uint8_t *nwords, uint2 *ulist, DevState *st, bool bitmaps, int G, Ctx &c);
// Numeric phase of the rows of BIN_NARROW (F32 or native F64),
// from the word lists of the symbolic phase; G lanes per row (4, 8 or 16).
// rows: their list (count), or null: every row of A is one.
int launch_num_narrow(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                      const int32_t *nlo, const uint8_t *nwords, const uint2 *ulist, const int32_t *rows,
                      int64_t count, int *err, int G, Ctx &c);

// Numeric phase of the listed rows of CLS_WINDOW_W (block false) or
// CLS_WINDOW_B, FP32 or native FP64; max_nnz: the largest row.  Also the rows
// of BIN_NARROW when they are few (rows null: every row of A).
int launch_num_window(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                      const int32_t *nlo, const uint8_t *nwords, const uint2 *ulist, const int32_t *rows, int64_t count,
                      bool block, int max_nnz, const char *label, int *err, Ctx &c);

// symbolic.cu
// First pass over all rows with a 32-slot map and G lanes per row (rows of
// bins EMPTY, HUGE and NARROW are skipped).  With bitmaps, marked rows are
// skipped too and listed instead (room for all rows in both lists): those for a
// warp from rows[0] on, those for a block from rows[nrows(A) - 1] downwards,
// those for a block's map in maps.
int launch_symbolic_first(const spgemm_csr &A, const uint8_t *bins, const int4 *desc, const int2 *pairs,
                          int64_t *crp, int32_t *rows, int32_t *maps, DevState *st, bool bitmaps, int G, Ctx &c);
// The listed rows (the warps' and blocks' lists in rows, those of SYM_MARK_MAP in
// maps), counted over bitmaps of their span or maps; no list length is needed
// on the host.
int launch_symbolic_bitmaps(const spgemm_csr &A, const spgemm_csr &B, const int4 *desc, const int2 *pairs,
                            const int2 *rspan, const int32_t *rows, const int32_t *maps, const uint8_t *bins,
                            int64_t *crp, DevState *st, Ctx &c);
// Second pass: kernels of bins 2..6; counts[b] = rows in bin b (host),
// rows = concatenated bin lists, rspan[i] = column-block span of row i.
// Writes nnz(C_i) to crp[i+1].
int launch_symbolic(const spgemm_csr &A, const spgemm_csr &B, const int2 *pairs,
                    const int32_t *ccnt, const int32_t *rows, const long long *counts,
                    int64_t *crp, int *err, void *gws, size_t gws_bytes, const int2 *rspan, Ctx &c);
size_t symbolic_global_ws(int64_t ncols_b, int nsm);

// numeric.cu
// Runs the numeric kernels: bins 1-2 over all rows in order (bins[i]), the
// others from the row lists by class (cls rows, largest row and span of each
// class, host).  FP64 uses double-word accumulation unless f64_native;
// bsplit: room for nnz(B) float2.
// Tunables of the numeric phase: lanes per row of the small-row kernel,
// largest output row it takes (16 or 32; bin 2 rows go to the warp kernel
// when 16), and map slots per output entry (2 or 4).
struct NumTune {
    int G = 8;
    int small_cap = 32;
    int slot_factor = 2;
};
struct ClsInfo {
    long long count[NCLS] = {0};
    int nnz[NCLS] = {0}, words[NCLS] = {0};
};
// What the symbolic phase left of the narrow rows (all rows; device).
struct NarrowInfo {
    const int32_t *nlo;
    const uint8_t *nwords;
    const uint2 *ulist;
};
int launch_numeric(int dtype, bool f64_native, const spgemm_csr &A, const spgemm_csr &B,
                   spgemm_csr &C, const uint8_t *bins, const int4 *bdesc, const int2 *rspan,
                   const int32_t *rows,
                   const long long *counts, const ClsInfo &cls, const NarrowInfo &nar, DevState *st, float2 *bsplit, void *gws,
                   size_t gws_bytes, int64_t max_row_nnz, const NumTune &tune, bool b_sorted,
                   int64_t max_alen, Ctx &c);
size_t numeric_global_ws(int64_t max_row_nnz, int64_t ncols_b, int nsm, int dtype);
size_t window_global_ws(int64_t max_alen, int nsm);

// rank.cu: listed rows with a dense rank accumulator (a block each), in FP32
// or native FP64; rows wider than max_words blocks or with more than max_nnz
// outputs are skipped.  RANK_SHORT: rows of CLS_RANK_W; RANK_MID: of CLS_RANK_V; RANK_ROW: of
// CLS_RANK_S (or CLS_B2).
enum RankSize { RANK_SHORT, RANK_MID, RANK_ROW, RANK_LONG };
int launch_num_rank(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                    const int2 *rspan, const int32_t *rows, int64_t count, RankSize size, int64_t max_nnz,
                    int64_t max_words, int *err, Ctx &c);

// Whether so many rows that cost less by cursors go to them, which need
// window_global_ws(max_alen) bytes of ws_bytes.
inline bool dense_by_window(long long count, int nsm, int64_t max_alen, size_t ws_bytes) {
    return count > (long long)DENSE_FEW * nsm && window_global_ws(max_alen, nsm) <= ws_bytes;
}

// dense.cu: listed rows over windows of a dense accumulator (rows of B
// sorted); ws holds the split table (dense_ws, either type) and behind it, when a row of
// A is long enough for folds, the folded windows (dense_fold_ws); next: device counter.
size_t dense_ws(int64_t nrows_b, int64_t ncols_b);
size_t dense_fold_ws(int64_t max_alen, int nsm);
int launch_num_dense(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                     const int2 *rspan, const int32_t *rows, int64_t count, int64_t max_alen, void *ws,
                     size_t ws_bytes, unsigned long long *next, int *err, Ctx &c);

// batched.cu: one instance of a batch, with its place in the stacked arrays.
struct BatchInst {
    const int64_t *arp, *brp;
    const int32_t *acol, *bcol;
    const void *aval, *bval;
    int64_t a_rows, a_nnz, b_rows, b_nnz;
    int64_t a_p0, b_p0;                  // row_ptr[0] of each operand
    int64_t a_row_off, a_nnz_off, b_row_off, b_nnz_off;
};
// Stack operand `which` (0 = A, 1 = B) of all instances: offsets and
// (shifted) columns when `pattern`, values when val is not null.
int launch_stack(const BatchInst *dinst, int nb, int64_t max_rows, int64_t max_nnz, int which, bool pattern,
                 int vb, int64_t total_rows, int64_t total_nnz, int64_t *rp, int32_t *col, void *val,
                 Ctx &c);

// triangles.cu: triangles of the undirected graph with the symmetric
// pattern A by the masked product L*L .* L (degree-ordered lower triangle
// L, compressed right-hand operand); the count lands in *total (device);
// perm_out / vcount (device, optional): labels, per-vertex counts.
size_t triangles_ws(int64_t n, int64_t nnz, int nsm);
int launch_triangles(const spgemm_csr &A, void *ws, int64_t *perm_out, int64_t *vcount, unsigned long long *total,
                     int *err, Ctx &c);

// backward.cu: dA on pattern(A), dB on pattern(B) from dC on pattern(C).
int launch_backward(int dtype, const spgemm_csr &A, const spgemm_csr &B, const spgemm_csr &C, void *da,
                    void *db, int *err, Ctx &c);

// plan.cu: Algorithm 4.  Cuts are part boundaries (first 0, last nrows).
struct ChunkPlan {
    int algorithm = 0, branch = 0;
    std::vector<int64_t> ac_cuts, b_cuts;
    int64_t size_a = 0, size_b = 0, size_c = 0, cost1 = 0, cost2 = 0;
};
int plan_chunks(const int64_t *a_rp, int64_t n_ac, const int64_t *c_rp, const int64_t *b_rp,
                int64_t n_b, int vb_ac, int vb_b, int64_t fast, ChunkPlan &p);
// BinarySearch cuts of one matrix (rp2 null) or a row-aligned pair.
bool cut_rows(const int64_t *rp1, const int64_t *rp2, int64_t n, int vb, double psize,
              std::vector<int64_t> &cuts);

// chunked.cu: Algorithms 2 and 3 with host operands.
// What a chunked symbolic call learns about its operands and hands on to the
// chunked numeric call of the same product: the column range of every block
// of CHUNK_RB rows of A (the rows of B each part of A reaches, known before
// the part is copied) and the longest row of C.  Valid only for the same
// host arrays and sizes.
constexpr int CHUNK_RB_L = 10, CHUNK_RB = 1 << CHUNK_RB_L;
struct ChunkCache {
    bool valid = false;
    const void *a_rp = nullptr, *a_col = nullptr, *b_rp = nullptr, *b_col = nullptr, *c_rp = nullptr;
    int64_t a_nrows = 0, a_ncols = 0, a_nnz = 0, b_nrows = 0, b_ncols = 0, b_nnz = 0;
    std::vector<int2> brange;   // per block of CHUNK_RB rows of A: {min, max} column ({INT_MAX, INT_MIN} if none)
    int64_t max_row = 0;        // largest row of C
};
// Events of a chunked call: the numeric call uses five groups of up to
// CHUNK_MAX_BUF (one per buffer of a group), the symbolic call the first 8.
constexpr int CHUNK_MAX_BUF = 3;
constexpr int CHUNK_EVENTS = 5 * CHUNK_MAX_BUF;
// Host waits of the library (for a count, a copied-back state or a part's
// column range): wait_ms <= 0 waits as long as it takes; otherwise the wait
// polls and gives up after wait_ms milliseconds with SPGEMM_ERR_TIMEOUT (the
// queued device work keeps running).
int host_wait_stream(cudaStream_t s, int64_t wait_ms, const char *what);
int host_wait_event(cudaEvent_t e, int64_t wait_ms, const char *what);

struct ChunkEnv {
    Ctx *ctx = nullptr;
    ChunkCache *cache = nullptr;
    void *arena = nullptr;        // exactly the budget, device
    cudaStream_t s_in = nullptr, s_out = nullptr;
    cudaEvent_t ev[CHUNK_EVENTS] = {};
    int nbuf = 2;                 // buffers per streamed operand: 2 (double) or 3 (triple)
    int64_t wait_ms = 0;          // limit of the host's waits (0: none)
    int *err = nullptr;
    std::vector<int64_t> *zeros = nullptr;   // host scratch: offsets of an empty C
    int *host_mm = nullptr;                  // pinned: column ranges of the A parts in the buffers
};
struct ChunkStats {
    int algorithm = 0, branch = 0;
    int64_t n_ac = 0, n_b = 0, cost1 = 0, cost2 = 0, h2d = 0, d2h = 0, skipped_b = 0,
            device_bytes = 0, b_windows = 0;
};
int chunked_numeric(ChunkEnv &env, int dtype, const spgemm_csr &A, const spgemm_csr &B,
                    spgemm_csr &C, size_t budget, ChunkStats &stats);
int chunked_symbolic(ChunkEnv &env, const spgemm_csr &A, const spgemm_csr &B, int64_t *C_row_ptr,
                     int64_t *nnz_C, size_t budget, ChunkStats &stats);

}  // namespace sg
