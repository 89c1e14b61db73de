// Row analysis: column compression of B (Section 2.1), per-row product
// counts and binning (Section 3.1, Section 3.3), exclusive scan of counts.
#include <algorithm>
#include <climits>
#include "internal.cuh"

namespace sg {

// ---------------------------------------------------------------- compression
// One thread per row of M: consecutive stored columns that fall in the same
// 32-column block are merged into one (block, mask) pair, so that a set of
// columns is held in fewer integers and unions become bitwise ORs (the
// compression of Section 2.1).  Rows need not be sorted; a sorted row yields
// one pair per block, ascending.  The row's descriptors are written
// alongside: desc = {first entry (int64), entries, pairs} for the product
// kernels, ana = {entries, pairs} for the analysis, and the row's first and
// last block (minmax) for the span tests.
//
// A warp takes 32 consecutive rows.  When their entries together number at
// most COMPRESS_STAGE, the warp first copies them into shared memory with
// coalesced asynchronous copies (a lane's row alone is a short run of
// addresses 32 rows apart from its neighbours' in one load instruction), and
// every lane then reads its row from there; otherwise every lane loads its
// own row.
constexpr int64_t COMPRESS_LONG = 128;   // rows longer than this take a warp each
constexpr int64_t COMPRESS_MID = 256;    // and longer than this a block
constexpr int COMPRESS_STAGE = 1024;     // staged entries per warp
constexpr int COMPRESS_WPB = 8;

__global__ void __launch_bounds__(COMPRESS_WPB * 32) k_compress(
    int64_t nrows, int64_t ncols, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
    int2 *__restrict__ pairs, int32_t *__restrict__ ccnt, int2 *__restrict__ minmax, int4 *__restrict__ desc,
    int2 *__restrict__ ana, int *err, int *unsorted_flag, int *long_count, int32_t *__restrict__ long_list) {
    __shared__ int stage_all[COMPRESS_WPB * COMPRESS_STAGE];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int *stage = stage_all + w * COMPRESS_STAGE;
    const int64_t r0 = ((int64_t)blockIdx.x * COMPRESS_WPB + w) * 32;
    if (r0 >= nrows) return;
    const int64_t r = r0 + lane;
    const bool live = r < nrows;
    const int64_t beg = live ? rp[r] : 0, end = live ? rp[r + 1] : 0;
    const int64_t rlast = min(r0 + 32, nrows);
    const int64_t wbeg = __shfl_sync(0xffffffffu, beg, 0);
    const int64_t wend = rp[rlast];
    const bool staged = wend - wbeg <= COMPRESS_STAGE;
    if (staged) {
        // asynchronous copies global -> shared (cp.async, 4 bytes a lane and
        // step: coalesced, no registers held while they are in flight); each
        // lane waits for its own, the warp barrier then publishes them all
        const int span = (int)(wend - wbeg);
        for (int x = lane; x < span; x += 32) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(stage + x);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(col + wbeg + x) : "memory");
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    __syncwarp();
    const bool lng = end - beg > COMPRESS_LONG;   // k_compress_long
    if (__any_sync(0xffffffffu, lng)) {   // the warps' rows from the front, the blocks' from the back
        const bool blk = end - beg > COMPRESS_MID;
        const unsigned mw = __ballot_sync(0xffffffffu, lng && !blk), mb = __ballot_sync(0xffffffffu, blk);
        const unsigned below = (1u << lane) - 1u;
        int at = 0;
        if (lane == 0 && mw) at = atomicAdd(&long_count[0], __popc(mw));
        if (lane == 1 && mb) at = atomicAdd(&long_count[1], __popc(mb));
        const int aw = __shfl_sync(0xffffffffu, at, 0), ab = __shfl_sync(0xffffffffu, at, 1);
        if (blk) long_list[nrows - 1 - (ab + __popc(mb & below))] = (int32_t)r;
        else if (lng) long_list[aw + __popc(mw & below)] = (int32_t)r;
    }
    if (!live || lng) return;
    const int *src = staged ? stage + (beg - wbeg) : col + beg;
    const int len = (int)(end - beg);
    int cur = -1;
    unsigned m = 0;
    int n = 0, bmin = INT_MAX, bmax = INT_MIN, prev = -1;
    bool bad = false, unsorted = false;
    // four columns at a time, their loads issued together
    for (int p0 = 0; p0 < len; p0 += 4) {
        int cc[4];
#pragma unroll
        for (int u = 0; u < 4; u++) cc[u] = p0 + u < len ? src[p0 + u] : 0;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (p0 + u >= len) break;
            const int c = cc[u];
            if (c < 0 || (int64_t)c >= ncols) { bad = true; continue; }
            unsorted |= c <= prev;
            prev = c;
            const int b = c >> 5;
            if (b != cur) {
                if (cur >= 0 && pairs) pairs[beg + n] = make_int2(cur, (int)m);
                if (cur >= 0) n++;
                cur = b;
                m = 0;
            }
            m |= 1u << (c & 31);
            bmin = min(bmin, b);
            bmax = max(bmax, b);
        }
    }
    if (cur >= 0) {
        if (pairs) pairs[beg + n] = make_int2(cur, (int)m);
        n++;
    }
    if (ccnt) ccnt[r] = n;
    if (minmax) minmax[r] = make_int2(bmin, bmax);
    if (desc) desc[r] = make_int4((int)(unsigned)(uint64_t)beg, (int)((uint64_t)beg >> 32), len, n);
    if (ana) ana[r] = make_int2(len, n);
    if (bad) atomicOr(err, DERR_COL_RANGE);
    if (unsorted && unsorted_flag) atomicOr(unsorted_flag, 1);
}

// The same for the listed rows, longer than COMPRESS_LONG.  Beyond COMPRESS_MID a
// block per row, COMPRESS_CHUNK entries at a time staged in shared memory: a pair
// starts where an entry's block differs from the previous entry's (its place is
// the number of starts before it, a block scan), and the thread at a start ORs
// the bits of the run that follows.  A warp per row of any length, 32 entries at a
// time with a segmented scan of the masks and a carried run, was a serial chain
// of 488 steps for the longest row of an R-MAT graph of scale 17, 1.5 ms for its
// 3.7 M entries (0.07 now; scale 13 0.25 -> 0.016 ms).  Up to COMPRESS_MID a warp
// per row, the whole row at once, the starts counted by ballots (296,296 rows of
// 135 entries 194 us, 200,000 of 200 172; by a block each 971 and 670, since
// most of a block's threads then only wait at its barriers).  Rows of 400
// entries, 100,000 of them, take 385 us by blocks; a hundred of them alone 8.
constexpr int COMPRESS_BS = 256, COMPRESS_PT = 4, COMPRESS_CHUNK = COMPRESS_BS * COMPRESS_PT;
static_assert(COMPRESS_BS / 32 * COMPRESS_MID <= 2 * COMPRESS_CHUNK, "a warp's rows are staged where a block's are");

__global__ void __launch_bounds__(COMPRESS_BS) k_compress_long(
    int64_t nrows, int64_t ncols, const int64_t *__restrict__ rp, const int32_t *__restrict__ col, int2 *__restrict__ pairs,
    int32_t *__restrict__ ccnt, int2 *__restrict__ minmax, int4 *__restrict__ desc, int2 *__restrict__ ana, int *err,
    int *unsorted_flag, const int *long_count, const int32_t *__restrict__ long_list) {
    constexpr int NW = COMPRESS_BS / 32;
    __shared__ __align__(16) int st[2 * COMPRESS_CHUNK];
    __shared__ int wsum[NW], wmin[NW], wmax[NW];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    // (plain loads: k_compress is through, and the warps of an SM share the line; past the L1 every
    // warp of the grid asks the L2 for it, 2.5 us a load when no row is long)
    const int nmid = long_count[0], nlong = long_count[1];
    bool bad = false, unsorted = false;
    for (int t = blockIdx.x; t < nlong; t += gridDim.x) {
        const int64_t r = long_list[nrows - 1 - t];
        const int64_t beg = rp[r], end = rp[r + 1];
        int npairs = 0, bmin = INT_MAX, bmax = INT_MIN;
        for (int64_t base = beg; base < end; base += COMPRESS_CHUNK) {
            const int n = (int)min((int64_t)COMPRESS_CHUNK, end - base);
            __syncthreads();
#pragma unroll
            for (int u = 0; u < COMPRESS_PT; u++) {
                const int x = tid + u * COMPRESS_BS;
                int c = x < n ? col[base + x] : -1;
                if (x < n && (c < 0 || (int64_t)c >= ncols)) { bad = true; c = -1; }   // breaks its run
                st[x] = c;
            }
            int prev = -1;
            if (tid == 0 && base > beg) {
                prev = col[base - 1];
                if (prev < 0 || (int64_t)prev >= ncols) prev = -1;
            }
            __syncthreads();
            const int e0 = tid * COMPRESS_PT;
            if (tid > 0) prev = st[e0 - 1];
            unsigned starts = 0;
#pragma unroll
            for (int u = 0; u < COMPRESS_PT; u++) {
                const int c = st[e0 + u];
                if (c >= 0) {
                    if (prev < 0 || (c >> 5) != (prev >> 5)) starts |= 1u << u;
                    unsorted |= c <= prev;
                    bmin = min(bmin, c >> 5);
                    bmax = max(bmax, c >> 5);
                }
                prev = c;
            }
            const int mine = __popc(starts);
            int incl = mine;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            if (lane == 31) wsum[w] = incl;
            __syncthreads();
            int idx = npairs + incl - mine;
#pragma unroll
            for (int j = 0; j < NW; j++) {
                if (j < w) idx += wsum[j];
                npairs += wsum[j];
            }
            while (starts) {
                const int e = e0 + __ffs(starts) - 1;
                starts &= starts - 1u;
                const int b = st[e] >> 5;
                unsigned m = 0;
                int p = e;
                for (; p < n && st[p] >> 5 == b; p++) m |= 1u << (st[p] & 31);   // -1 >> 5 is no block
                for (int64_t q = base + n; p == n && q < end; q++) {             // a run past the chunk
                    const int c = col[q];
                    if (c >> 5 != b) break;
                    m |= 1u << (c & 31);
                }
                if (pairs) pairs[beg + idx] = make_int2(b, (int)m);
                idx++;
            }
        }
        bmin = __reduce_min_sync(0xffffffffu, bmin);
        bmax = __reduce_max_sync(0xffffffffu, bmax);
        if (lane == 0) {
            wmin[w] = bmin;
            wmax[w] = bmax;
        }
        __syncthreads();
        if (tid == 0) {
            for (int j = 1; j < NW; j++) {
                bmin = min(bmin, wmin[j]);
                bmax = max(bmax, wmax[j]);
            }
            const int len = (int)(end - beg);
            if (ccnt) ccnt[r] = npairs;
            if (minmax) minmax[r] = make_int2(bmin, bmax);
            if (desc) desc[r] = make_int4((int)(unsigned)(uint64_t)beg, (int)((uint64_t)beg >> 32), len, npairs);
            if (ana) ana[r] = make_int2(len, npairs);
        }
    }
    if (nmid > 0) {
        __syncthreads();
        int *ws = st + w * COMPRESS_MID;
        // from the last block on, a warp of each in turn: the first ones have the blocks' rows
        for (int t = w * gridDim.x + gridDim.x - 1 - blockIdx.x; t < nmid; t += gridDim.x * NW) {
            const int64_t r = long_list[t];
            const int64_t beg = rp[r];
            const int len = (int)(rp[r + 1] - beg);
            int npairs = 0, bmin = INT_MAX, bmax = INT_MIN;
            __syncwarp();
#pragma unroll
            for (int u = 0; u < COMPRESS_MID / 32; u++) {
                const int x = lane + 32 * u;
                int c = x < len ? col[beg + x] : -1;
                if (x < len && (c < 0 || (int64_t)c >= ncols)) { bad = true; c = -1; }
                ws[x] = c;
            }
            __syncwarp();
            for (int x = lane; x - lane < len; x += 32) {
                const int c = ws[x], prev = x > 0 ? ws[x - 1] : -1;
                const bool start = c >= 0 && (prev < 0 || (c >> 5) != (prev >> 5));
                const unsigned m = __ballot_sync(0xffffffffu, start);
                if (c >= 0) {
                    unsorted |= c <= prev;
                    bmin = min(bmin, c >> 5);
                    bmax = max(bmax, c >> 5);
                }
                if (start && pairs) {
                    unsigned bits = 0;
                    for (int p = x; p < len && ws[p] >> 5 == c >> 5; p++) bits |= 1u << (ws[p] & 31);
                    pairs[beg + npairs + __popc(m & ((1u << lane) - 1u))] = make_int2(c >> 5, (int)bits);
                }
                npairs += __popc(m);
            }
            bmin = __reduce_min_sync(0xffffffffu, bmin);
            bmax = __reduce_max_sync(0xffffffffu, bmax);
            if (lane == 0) {
                if (ccnt) ccnt[r] = npairs;
                if (minmax) minmax[r] = make_int2(bmin, bmax);
                if (desc) desc[r] = make_int4((int)(unsigned)(uint64_t)beg, (int)((uint64_t)beg >> 32), len, npairs);
                if (ana) ana[r] = make_int2(len, npairs);
            }
        }
    }
    if (bad) atomicOr(err, DERR_COL_RANGE);
    if (unsorted && unsorted_flag) *unsorted_flag = 1;
}

int launch_compress(const spgemm_csr &M, int2 *pairs, int32_t *ccnt, int2 *minmax, int4 *desc,
                    int2 *ana, int *err, int *long_count, int32_t *long_list, Ctx &c, int *unsorted) {
    if (M.nrows == 0) return SPGEMM_OK;
    int64_t blocks = (M.nrows + COMPRESS_WPB * 32 - 1) / (COMPRESS_WPB * 32);
    c.begin("compress", M.nrows);
    k_compress<<<(unsigned)blocks, COMPRESS_WPB * 32, 0, c.s>>>(M.nrows, M.ncols, M.row_ptr, M.col_idx, pairs,
                                                    ccnt, minmax, desc, ana, err, unsorted, long_count, long_list);
    c.end();
    if (M.nnz > COMPRESS_LONG) {
        // one resident wave (it returns at once when no row is long)
        const int64_t wblocks = std::min<int64_t>(M.nnz / (COMPRESS_LONG + 1), resident_blocks(k_compress_long, COMPRESS_BS, c.nsm));
        c.begin("compress_long", M.nrows);
        k_compress_long<<<(unsigned)wblocks, COMPRESS_BS, 0, c.s>>>(M.nrows, M.ncols, M.row_ptr, M.col_idx, pairs,
                                                                    ccnt, minmax, desc, ana, err, unsorted, long_count,
                                                                    long_list);
        c.end();
    }
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

// ---------------------------------------------------------------- analysis
// Eight lanes per row of A.  For row i: flops_i = sum_k nnz(B_k) (the number
// of accumulator insertions, Section 3.1) and cpairs_i = sum_k pairs(B_k).
// The symbolic accumulator needs at most min(cpairs_i, ceil(ncols/32)) keys
// (the second pass narrows rows down by their column span itself).
// Empty rows get their count (0) here; rows for the dense bitmap (bin 6)
// are marked -1 for the second pass.
constexpr int AN_G = 8;
__global__ void k_analyze(int64_t nrows, int64_t nrows_b, int64_t nwords,
                          const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
                          const int2 *__restrict__ ana, const int2 *__restrict__ bmm, int64_t *__restrict__ flops,
                          uint8_t *__restrict__ bins, int64_t *__restrict__ crp, int2 *__restrict__ rspan,
                          DevState *st, bool bitmaps) {
    __shared__ unsigned long long hist[NBINS];
    __shared__ unsigned long long fsum;
    __shared__ unsigned long long alen_max;
    __shared__ int marks[2];   // rows without a mark, with one
    if (threadIdx.x < 2) marks[threadIdx.x] = 0;
    if (threadIdx.x < NBINS) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) { fsum = 0; alen_max = 0; }
    __syncthreads();
    const int lane = threadIdx.x % AN_G;
    const unsigned gmask = ((1u << AN_G) - 1) << ((threadIdx.x & 31) & ~(AN_G - 1));
    // a fixed grid strides over the rows, so the block's totals reach the
    // global counters once per block, not once per 32 rows
    const int64_t rstride = (int64_t)gridDim.x * (blockDim.x / AN_G);
    long long wf = 0, wl = 0;   // this lane's share of the products and the longest row
    bool bad = false;
    for (int64_t i0 = (int64_t)blockIdx.x * (blockDim.x / AN_G); i0 < nrows; i0 += rstride) {
        const int64_t i = i0 + threadIdx.x / AN_G;
        const bool live = i < nrows;
        long long f = 0, cp = 0;
        int lo = INT_MAX, hi = -1;
        bool rowbad = false;
        if (live) {
            for (int64_t p = arp[i] + lane; p < arp[i + 1]; p += AN_G) {
                int k = acol[p];
                if (k < 0 || (int64_t)k >= nrows_b) { bad = rowbad = true; continue; }
                const int2 d = ana[k], m = bmm[k];
                f += d.x;
                cp += d.y;
                lo = min(lo, m.x);
                hi = max(hi, m.y);
            }
        }
        for (int d = AN_G / 2; d > 0; d >>= 1) {
            f += __shfl_xor_sync(gmask, f, d, AN_G);
            cp += __shfl_xor_sync(gmask, cp, d, AN_G);
            lo = min(lo, __shfl_xor_sync(gmask, lo, d, AN_G));
            hi = max(hi, __shfl_xor_sync(gmask, hi, d, AN_G));
        }
        rowbad = (__ballot_sync(0xffffffffu, rowbad) & gmask) != 0;
        int b = BIN_EMPTY;
        const bool lead = live && lane == 0;
        if (lead) {
            const long long keys = min(cp, (long long)nwords);
            b = sym_bin(keys, cp);
            flops[i] = f;
            bins[i] = (uint8_t)b;
            rspan[i] = make_int2(lo, hi >= lo ? hi - lo + 1 : 0);
            if (bitmaps) {
                if (rowbad) b = BIN_EMPTY;
                bins[i] = (uint8_t)b;
                const int mark = b == BIN_EMPTY ? 0 : sym_mark(cp, hi - lo + 1);
                crp[i + 1] = mark;
                if (b != BIN_EMPTY) marks[mark != 0] = 1;
            } else {
                if (b == BIN_EMPTY) crp[i + 1] = 0;
                if (b == BIN_HUGE) crp[i + 1] = -1;
            }
            wf += f;
            wl = max(wl, (long long)(arp[i + 1] - arp[i]));
        }
        warp_hist(hist, lead, b);
    }
    if (bad) atomicOr(&st->err, DERR_COL_RANGE);
    // products of the warp's rows and its longest row of A
    for (int d = 16; d > 0; d >>= 1) {
        wf += __shfl_xor_sync(0xffffffffu, wf, d);
        wl = max(wl, __shfl_xor_sync(0xffffffffu, wl, d));
    }
    if ((threadIdx.x & 31) == 0 && wf) atomicAdd(&fsum, (unsigned long long)wf);
    if ((threadIdx.x & 31) == 0 && wl) atomicMax(&alen_max, (unsigned long long)wl);
    __syncthreads();
    if (threadIdx.x == 0 && fsum) atomicAdd((unsigned long long *)&st->flops_total, fsum);
    if (threadIdx.x == 0 && marks[0]) *(volatile int *)&st->sym_first = 1;
    if (threadIdx.x == 0 && marks[1]) *(volatile int *)&st->sym_marked = 1;
    if (threadIdx.x == 0 && alen_max && alen_max > (unsigned long long)*(volatile long long *)&st->max_alen)
        atomicMax((unsigned long long *)&st->max_alen, alen_max);
    if (threadIdx.x < NBINS && hist[threadIdx.x]) {
        atomicAdd((unsigned long long *)&st->sym_hist[threadIdx.x], hist[threadIdx.x]);
        if (threadIdx.x == BIN_HUGE)
            atomicAdd((unsigned long long *)&st->bin_count[0][BIN_HUGE], hist[threadIdx.x]);
    }
}

int launch_analyze(const spgemm_csr &A, const spgemm_csr &B, const int2 *ana, const int2 *bmm, int64_t *flops,
                   uint8_t *bins, int64_t *crp, int2 *rspan, DevState *st, bool bitmaps, Ctx &c) {
    if (A.nrows == 0) return SPGEMM_OK;
    int64_t threads = A.nrows * AN_G;
    int64_t blocks = (threads + 255) / 256;
    blocks = std::min<int64_t>(blocks, (int64_t)c.nsm * 16);
    int64_t nwords = (B.ncols + 31) / 32;
    c.begin("analyze", A.nrows);
    k_analyze<<<(unsigned)blocks, 256, 0, c.s>>>(A.nrows, B.nrows, nwords, A.row_ptr, A.col_idx,
                                                   ana, bmm, flops, bins, crp, rspan, st, bitmaps);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

// Products per row only (inspection entry point).
__global__ void k_row_flops(int64_t nrows, int64_t nrows_b, const int64_t *__restrict__ arp,
                            const int32_t *__restrict__ acol, const int64_t *__restrict__ brp,
                            int64_t *__restrict__ flops, int *err) {
    const int lane = threadIdx.x % AN_G;
    const unsigned gmask = ((1u << AN_G) - 1) << ((threadIdx.x & 31) & ~(AN_G - 1));
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / AN_G;
    long long f = 0;
    bool bad = false;
    if (i < nrows) {
        for (int64_t p = arp[i] + lane; p < arp[i + 1]; p += AN_G) {
            int k = acol[p];
            if (k < 0 || (int64_t)k >= nrows_b) { bad = true; continue; }
            f += brp[k + 1] - brp[k];
        }
    }
    for (int d = AN_G / 2; d > 0; d >>= 1) f += __shfl_xor_sync(gmask, f, d, AN_G);
    if (bad) atomicOr(err, DERR_COL_RANGE);
    if (i < nrows && lane == 0) flops[i] = f;
}

int launch_row_flops(const spgemm_csr &A, const spgemm_csr &B, int64_t *flops, int *err,
                     Ctx &c) {
    if (A.nrows == 0) return SPGEMM_OK;
    int64_t blocks = (A.nrows * AN_G + 255) / 256;
    c.begin("row_flops", A.nrows);
    k_row_flops<<<(unsigned)blocks, 256, 0, c.s>>>(A.nrows, B.nrows, A.row_ptr, A.col_idx,
                                                     B.row_ptr, flops, err);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

// ---------------------------------------------------------------- row lists
// Row lists for the list-driven kernels.  CLS false (symbolic second pass):
// rows marked -1 in crp[i+1] (overflowed the first pass, or bin 6), listed by
// max(key[i], 2), key the bins.  CLS true (numeric): rows of the classes
// `first` and up, key the classes.  Within a warp the lanes with the same
// list reserve their slots with one atomic (__match_any_sync), so rows stay
// in ascending order inside each warp.
template <bool CLS>
__global__ void k_scatter_rows(int64_t n, const uint8_t *__restrict__ key, const int64_t *__restrict__ crp,
                               int32_t *__restrict__ rows, DevState *st, int first) {
    constexpr int NL = CLS ? (int)NCLS : (int)NBINS;
    __shared__ long long off[NL];
    long long *cursor = CLS ? st->cls_cursor : st->bin_cursor;
    if (threadIdx.x == 0) {
        long long o = 0;
        for (int b = 0; b < NL; b++) {
            off[b] = o;
            if (b >= first && (CLS || b <= BIN_HUGE)) o += CLS ? st->cls_count[b] : st->bin_count[0][b];
        }
    }
    __syncthreads();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int b = 0;   // none
    if (i < n) {
        if (CLS) b = key[i] >= first ? key[i] : 0;
        else if (crp[i + 1] < 0) b = max((int)key[i], first);
    }
    unsigned act = __ballot_sync(0xffffffffu, b != 0);
    if (b == 0) return;
    unsigned peers = __match_any_sync(act, b);
    int lane = threadIdx.x & 31;
    int leader = __ffs(peers) - 1;
    long long base = 0;
    if (lane == leader) base = atomicAdd((unsigned long long *)&cursor[b], (unsigned long long)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    int rank = __popc(peers & ((1u << lane) - 1));
    rows[off[b] + base + rank] = (int32_t)i;
}

int launch_scatter_bins(int64_t n, const uint8_t *bins, const int64_t *crp, int32_t *rows, DevState *st, Ctx &c) {
    if (n == 0) return SPGEMM_OK;
    SG_CUDA(cudaMemsetAsync(st->bin_cursor, 0, sizeof(st->bin_cursor), c.s));
    c.begin("scatter_bins", n);
    k_scatter_rows<false><<<(unsigned)((n + 255) / 256), 256, 0, c.s>>>(n, bins, crp, rows, st, 2);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_scatter_cls(int64_t n, const uint8_t *cls, int32_t *rows, DevState *st, int first_cls, Ctx &c) {
    if (n == 0) return SPGEMM_OK;
    SG_CUDA(cudaMemsetAsync(st->cls_cursor, 0, sizeof(st->cls_cursor), c.s));
    c.begin("scatter_cls", n);
    k_scatter_rows<true><<<(unsigned)((n + 255) / 256), 256, 0, c.s>>>(n, cls, nullptr, rows, st, first_cls);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

// ---------------------------------------------------------------- scan
// Reduce-then-scan over tiles of counts: tile sums, then every tile
// is rescanned with the sum of the tiles before it (with more than SCAN_DIRECT
// tiles, one block scans the sums first, looping with a carry).  x[0] is set to 0 and x[1..n] becomes the inclusive prefix.
// A thread takes SCAN_PT counts of a tile; where the rows are also binned,
// SCAN_BIN_PT, or one while the rows are at most SCAN_FEW (binning a row is a
// chain of loads, and with eight rows a thread a handful of blocks walked eight
// such chains one after another).  Measured, k_scan_apply<true> with 8 -> these:
// 4096 rows 12.3 -> 8.2 us, 8192 20.4 -> 10.2, 20,001 16.4 -> 8.9, 2.1 M and
// 79,507 together 49 -> 37 (one a thread there 41; 39 since classing a row takes
// divisions, at six blocks an SM: 43 with the 60 registers it takes unasked).
constexpr int SCAN_BS = 256, SCAN_PT = 8, SCAN_BIN_PT = 4;
constexpr int64_t SCAN_FEW = 131072;

// Enough for any number of rows up to n.
size_t scan_binning_tmp_bytes(int64_t n) {
    const int64_t few = (std::min(n, SCAN_FEW) + SCAN_BS - 1) / SCAN_BS;
    return (size_t)(std::max(few, (n + SCAN_BS * SCAN_BIN_PT - 1) / (SCAN_BS * SCAN_BIN_PT)) + 1) * sizeof(long long);
}

size_t scan_tmp_bytes(int64_t n) {
    const int64_t tiles = (n + SCAN_BS * SCAN_PT - 1) / (SCAN_BS * SCAN_PT);
    return (size_t)(tiles + 1) * sizeof(long long);
}

__device__ __forceinline__ long long block_excl_scan(long long v, long long *sh, long long *total) {
    // sh: SCAN_BS/32 entries
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = v;
    for (int d = 1; d < 32; d <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) sh[w] = incl;
    __syncthreads();
    if (w == 0) {
        long long s = lane < SCAN_BS / 32 ? sh[lane] : 0;
        long long si = s;
        for (int d = 1; d < 32; d <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, si, d);
            if (lane >= d) si += t;
        }
        if (lane < SCAN_BS / 32) sh[lane] = si - s;
        if (lane == SCAN_BS / 32 - 1) *total = si;
    }
    __syncthreads();
    long long r = sh[w] + incl - v;
    __syncthreads();
    return r;
}

template <int PT>
__global__ void k_scan_tiles(const int64_t *__restrict__ x1, int64_t n, long long *tile_sums) {
    __shared__ long long sh[SCAN_BS / 32];
    __shared__ long long tot;
    int64_t base = ((int64_t)blockIdx.x * SCAN_BS + threadIdx.x) * PT;
    long long s = 0;
#pragma unroll
    for (int j = 0; j < PT; j++)
        if (base + j < n) s += x1[base + j];
    block_excl_scan(s, sh, &tot);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(long long *tile_sums, int64_t tiles, long long *total) {
    __shared__ long long sh[SCAN_BS / 32];
    __shared__ long long tot;
    long long carry = 0;
    for (int64_t b0 = 0; b0 < tiles; b0 += SCAN_BS) {
        int64_t t = b0 + threadIdx.x;
        long long v = t < tiles ? tile_sums[t] : 0;
        long long e = block_excl_scan(v, sh, &tot);
        if (t < tiles) tile_sums[t] = carry + e;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// Numeric bin and class of the rows whose counts the scan walks over, in the
// same pass (k_scan_apply<true>): the counts are in registers there, and a
// pass of its own read the offsets again and cost a launch.
struct ScanBins {
    const int64_t *arp, *flops;
    uint8_t *bins, *cls;
    const int2 *rspan;
    const int32_t *nlo;   // may be null
    const uint8_t *nwords;
    DevState *st;
    bool dense_ok;
};

// SUMMED: tile_sums holds the tiles' exclusive prefix (k_scan_sums); else
// every block adds up the sums of the tiles before its own, which costs less
// than the launch of k_scan_sums while there are at most SCAN_DIRECT tiles,
// and the last block writes the total.
constexpr int64_t SCAN_DIRECT = 4096;

template <bool BINS, bool SUMMED, int PT>
__global__ void __launch_bounds__(SCAN_BS, PT == SCAN_BIN_PT ? 6 : 0) k_scan_apply(int64_t *__restrict__ x, int64_t n,
                                                        const long long *__restrict__ tile_sums, long long *total,
                                                        ScanBins b) {
    __shared__ long long sh[SCAN_BS / 32];
    __shared__ long long tot;
    __shared__ unsigned long long hist[NBINS];
    __shared__ int ccnt[NCLS], cnnz[NCLS], cwords[NCLS], narrow_flops;   // at most NARROW_FLOPS a row
    if (BINS) {
        if (threadIdx.x == 0) narrow_flops = 0;
        if (threadIdx.x < NBINS) hist[threadIdx.x] = 0;
        if (threadIdx.x < NCLS) ccnt[threadIdx.x] = cnnz[threadIdx.x] = cwords[threadIdx.x] = 0;
    }
    long long before = 0;
    if (SUMMED) {
        before = tile_sums[blockIdx.x];
    } else if (blockIdx.x > 0) {
        long long s = 0;
        for (unsigned t = threadIdx.x; t < blockIdx.x; t += SCAN_BS) s += tile_sums[t];
        block_excl_scan(s, sh, &tot);
        before = tot;
    }
    int64_t *x1 = x + 1;
    const int64_t base = ((int64_t)blockIdx.x * SCAN_BS + threadIdx.x) * PT;
    long long v[PT];
    long long s = 0;
#pragma unroll
    for (int j = 0; j < PT; j++) {
        v[j] = base + j < n ? x1[base + j] : 0;
        s += v[j];
    }
    long long e = before + block_excl_scan(s, sh, &tot);
    if (!SUMMED && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = before + tot;
#pragma unroll
    for (int j = 0; j < PT; j++) {
        e += v[j];
        if (base + j < n) x1[base + j] = e;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) x[0] = 0;
    if (!BINS) return;
#pragma unroll
    for (int j = 0; j < PT; j++) {
        const int64_t i = base + j;
        int bin = BIN_EMPTY, nf = 0;
        if (i < n) {
            const long long c = v[j], f = b.flops[i];
            bin = c > 0 ? num_bin(c, f) : BIN_EMPTY;
            if (bin != BIN_EMPTY && b.nlo && b.nlo[i] >= 0 && c <= NARROW_NMAX && f <= NARROW_FLOPS) bin = BIN_NARROW;
            b.bins[i] = (uint8_t)bin;
            if (bin == BIN_HUGE) atomicMax((unsigned long long *)&b.st->max_row_nnz, (unsigned long long)c);
            int k = bin == BIN_NARROW ? CLS_NARROW : CLS_NONE;
            if (bin == BIN_NARROW) nf = (int)f;
            if (bin >= 2 && bin <= BIN_HUGE) {
                const int words = b.rspan[i].y;
                const bool listed = b.nlo && b.nlo[i] >= 0 && b.nwords[i] <= NARROW_NMAX;
                k = num_cls(bin, c, f, words, listed, b.dense_ok && b.st->b_unsorted == 0,
                            bin >= 5 ? b.arp[i + 1] - b.arp[i] : 0);
                atomicAdd(&ccnt[k], 1);
                if (c > cnnz[k]) atomicMax(&cnnz[k], (int)min(c, (long long)INT_MAX));
                if (words > cwords[k]) atomicMax(&cwords[k], words);
            }
            b.cls[i] = (uint8_t)k;
        }
        warp_hist(hist, i < n, bin);
        nf = __reduce_add_sync(0xffffffffu, nf);
        if ((threadIdx.x & 31) == 0 && nf) atomicAdd(&narrow_flops, nf);
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t == 0 && narrow_flops) atomicAdd(&b.st->narrow_flops, (unsigned long long)narrow_flops);
    if (t < NBINS && hist[t]) atomicAdd((unsigned long long *)&b.st->bin_count[1][t], hist[t]);
    if (t == BIN_NARROW && hist[t]) atomicAdd((unsigned long long *)&b.st->cls_count[CLS_NARROW], hist[t]);
    if (t < NCLS && ccnt[t]) {
        atomicAdd((unsigned long long *)&b.st->cls_count[t], (unsigned long long)ccnt[t]);
        if (cnnz[t] > *(volatile int *)&b.st->cls_nnz[t]) atomicMax(&b.st->cls_nnz[t], cnnz[t]);
        if (cwords[t] > *(volatile int *)&b.st->cls_words[t]) atomicMax(&b.st->cls_words[t], cwords[t]);
    }
}

template <bool BINS, int PT>
static int run_scan(int64_t *x, int64_t n, long long *total, void *tmp, const ScanBins &b, Ctx &c) {
    const int64_t tiles = (n + SCAN_BS * PT - 1) / (SCAN_BS * PT);
    long long *sums = (long long *)tmp;
    if (tiles > 1) {
        c.begin("scan_tiles", n);
        k_scan_tiles<PT><<<(unsigned)tiles, SCAN_BS, 0, c.s>>>(x + 1, n, sums);
        c.end();
    }
    if (tiles > SCAN_DIRECT) {
        c.begin("scan_sums", tiles);
        k_scan_sums<<<1, SCAN_BS, 0, c.s>>>(sums, tiles, total);
        c.end();
    }
    c.begin("scan_apply", n);
    if (tiles > SCAN_DIRECT)
        k_scan_apply<BINS, true, PT><<<(unsigned)tiles, SCAN_BS, 0, c.s>>>(x, n, sums, total, b);
    else
        k_scan_apply<BINS, false, PT><<<(unsigned)tiles, SCAN_BS, 0, c.s>>>(x, n, sums, total, b);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_scan_counts(int64_t *x, int64_t n, long long *total, void *tmp, Ctx &c) {
    if (n == 0) {
        SG_CUDA(cudaMemsetAsync(x, 0, sizeof(int64_t), c.s));
        SG_CUDA(cudaMemsetAsync(total, 0, sizeof(long long), c.s));
        return SPGEMM_OK;
    }
    return run_scan<false, SCAN_PT>(x, n, total, tmp, ScanBins{}, c);
}

int launch_scan_binning(int64_t *crp, int64_t n, void *tmp, const int64_t *arp, const int64_t *flops, uint8_t *bins,
                        uint8_t *cls, const int2 *rspan, const int32_t *nlo, const uint8_t *nwords, DevState *st, bool dense_ok,
                        Ctx &c) {
    if (n == 0) return launch_scan_counts(crp, n, &st->nnz, tmp, c);
    const ScanBins b{arp, flops, bins, cls, rspan, nlo, nwords, st, dense_ok};
    return n <= SCAN_FEW ? run_scan<true, 1>(crp, n, &st->nnz, tmp, b, c) : run_scan<true, SCAN_BIN_PT>(crp, n, &st->nnz, tmp, b, c);
}

}  // namespace sg
