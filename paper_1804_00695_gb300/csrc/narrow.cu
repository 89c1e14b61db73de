// Narrow rows: rows of C whose columns all fall within a window of
// NARROW_W consecutive blocks of 32 columns (4096 columns), the common case
// of banded and stencil-like products such as the multigrid Galerkin
// operators of Section 3.2.
//
// Section 2.1 compresses each row of B into (block, 32-bit mask) pairs so
// that the union of column sets becomes bitwise ORs.  Over a narrow window
// the union needs no hash at all: a dense table of NARROW_W masks, indexed
// by block minus the window's first block, holds it exactly.
//
// * Symbolic (k_sym_narrow): one pass over every row of A computes the
//   row's products (Section 3.1: accumulator insertions = multiplications),
//   its compressed pairs and its column window from the first/last block of
//   each B_k; rows that fit the window OR their pairs into the table and
//   count popcounts (nnz(C_i)); every other row gets the analysis the hash
//   kernels need (symbolic bin, -1 marks for the second pass).
//   A narrow row with at most NARROW_NMAX outputs also leaves its union for
//   the numeric phase, as the list of its non-empty words in order, each
//   with its mask and the rank of its first column (prefix counts of the
//   masks).
// * Numeric (k_num_narrow): the row's list is scattered back into the window
//   table, which then gives every column its rank in the sorted output:
//   rank(c) = base[w] + popc(mask[w] & bits below c), w = c/32 - first
//   block.  The dense accumulator of Section 3.1 is indexed by rank, so the
//   row is written in column order with no hash probe and no sort.
//   Products are taken one chunk of G consecutive entries of B_k at a time
//   by the G lanes of a row: entries of one row of B have distinct columns,
//   so within a chunk no two lanes of a row add to the same rank and the
//   update is a plain read-modify-write of shared memory.
#include <climits>
#include <type_traits>
#include "internal.cuh"

namespace sg {

// Quad (four words) of a row's window that lane gl of its G lanes takes in
// its j-th turn: rounds of G*P consecutive quads, P consecutive ones per
// lane (with G = 4, P = 2 puts the lanes 32 bytes apart, so that the two row
// slots served by one quarter of a warp, 4 words apart, use different banks).
template <int G, int P>
__device__ __forceinline__ int quad_of(int j, int gl) {
    return ((j / P) * G + gl) * P + (j % P);
}

// ---------------------------------------------------------------- symbolic
constexpr int NARROW_SYM_WPB = 8;
constexpr int SYM_EU = 4;   // entries of A per lane whose loads are in flight together

// G lanes per row, 32/G rows per warp.  For row i: flops, pairs and window
// from desc[k] = {start, entries, pairs} and bmm[k] = {first block, last
// block} of every stored a_ik (lanes strided over the entries).  A row is narrow when it has products, no
// column of A out of range, a window of at most NARROW_W blocks and at most
// NARROW_PAIRS pairs; its count goes to crp[i+1], its first block to
// nlo[i] and BIN_NARROW to bins[i]; its non-empty words, in order, to
// ulist[i*NARROW_NMAX ...] as {word | rank of its first column << 8, mask}
// (the first NARROW_NMAX of them) and their number to nwords[i].  Other
// rows get nlo[i] = -1 and the symbolic bin of their bound (crp[i+1] = 0
// for empty rows, -1 for the dense-bitmap bin), exactly as the analysis
// kernel gives them.
// With four lanes a row, four blocks an SM (64 registers): with three (80)
// the same products take 0.98 ms, with five (48 registers, and 34 KB less for
// the L1, which the gathers of B live in) 0.76 ms.
template <int G>
__global__ void __launch_bounds__(NARROW_SYM_WPB * 32, G == 4 ? 4 : 0) k_sym_narrow(
    int64_t n, int64_t nrows_b, int64_t nwords_b, const int64_t *__restrict__ arp,
    const int32_t *__restrict__ acol, const int4 *__restrict__ desc, const int2 *__restrict__ bmm,
    const int2 *__restrict__ pairs, int64_t *__restrict__ flops, uint8_t *__restrict__ bins,
    int64_t *__restrict__ crp, int2 *__restrict__ rspan, int32_t *__restrict__ nlo, uint8_t *__restrict__ nwords,
    uint2 *__restrict__ ulist, DevState *st, bool bitmaps) {
    constexpr int WPB = NARROW_SYM_WPB;
    constexpr int RPW = 32 / G, NR = WPB * RPW, QPL = NARROW_W / 4 / G;
    constexpr int P = G >= 8 ? 1 : 8 / G;
    __shared__ __align__(16) unsigned tab_all[NR * NARROW_TAB_STRIDE];
    __shared__ unsigned long long hist[NBINS];
    __shared__ unsigned long long fsum, alen_max;
    __shared__ int marks[2];   // rows without a mark (sym_mark), with one
    if (threadIdx.x < 2) marks[threadIdx.x] = 0;
    if (threadIdx.x < NBINS) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) { fsum = 0; alen_max = 0; }
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / G, gl = lane % G, gbase = g * G;
    const unsigned gm = (G == 32) ? 0xffffffffu : (((1u << G) - 1) << gbase);
    const int slot = w * RPW + g;
    unsigned *t = tab_all + slot * NARROW_TAB_STRIDE;
    long long wf = 0, wl = 0;
    bool bad = false;
    int flag = 0;
    const int64_t stride = (int64_t)gridDim.x * NR;
    for (int64_t base = (int64_t)blockIdx.x * NR + w * RPW; base < n; base += stride) {
        const int64_t i = base + g;
        const bool live = i < n;
        const int64_t p0 = live ? arp[i] : 0;
        const int plen = live ? (int)(arp[i + 1] - p0) : 0;
        const int maxlen = __reduce_max_sync(0xffffffffu, plen);
        long long f = 0, cp = 0;
        int lo = INT_MAX, hi = INT_MIN;
        bool rowbad = false;
        // SYM_EU entries per lane at a time: their loads of A, then of the
        // rows' descriptors, issued together
        for (int e0 = 0; e0 < plen; e0 += G * SYM_EU) {
            int k[SYM_EU];
#pragma unroll
            for (int u = 0; u < SYM_EU; u++) {
                const int e = e0 + gl + G * u;
                k[u] = e < plen ? acol[p0 + e] : -1;
            }
            int4 d[SYM_EU];
            int2 m[SYM_EU];
#pragma unroll
            for (int u = 0; u < SYM_EU; u++) {
                const bool ok = (unsigned)k[u] < (unsigned)nrows_b;
                rowbad |= !ok && e0 + gl + G * u < plen;
                d[u] = ok ? desc[k[u]] : make_int4(0, 0, 0, 0);
                m[u] = ok ? bmm[k[u]] : make_int2(INT_MAX, INT_MIN);
            }
#pragma unroll
            for (int u = 0; u < SYM_EU; u++) {
                f += d[u].z;
                cp += d[u].w;
                lo = min(lo, m[u].x);
                hi = max(hi, m[u].y);
            }
        }
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) {
            f += __shfl_xor_sync(0xffffffffu, f, d, G);
            cp += __shfl_xor_sync(0xffffffffu, cp, d, G);
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d, G));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d, G));
        }
        rowbad = (__ballot_sync(0xffffffffu, rowbad) & gm) != 0;
        bad |= rowbad;
        const bool nar = live && f > 0 && !rowbad && hi >= lo && hi - lo < NARROW_W && cp <= NARROW_PAIRS;
        int cnt = 0, nz = 0;
        // words of the widest window of the warp's rows: the table is cleared
        // and read over so many, a round of 4 * G * P at a time (128^3
        // Galerkin products: 0.68 -> 0.66 ms; windows of 3 to 61 words)
        const int wide = __reduce_max_sync(0xffffffffu, nar ? hi - lo + 1 : 0);
        if (wide > 0) {
            if (nar) {
#pragma unroll
                for (int j = 0; j < QPL; j++)
                    if (4 * G * (j - j % P) < wide)
                        *(uint4 *)&t[4 * quad_of<G, P>(j, gl)] = make_uint4(0u, 0u, 0u, 0u);
            }
            __syncwarp();
            // the union: every lane ORs the pairs of its own entries (lanes of
            // a row may hit the same word: atomic OR), SYM_EU entries at a
            // time, the loads of one pair of each issued together
            if (nar) {
                for (int e0 = 0; e0 < plen; e0 += G * SYM_EU) {
                    int k[SYM_EU];
#pragma unroll
                    for (int u = 0; u < SYM_EU; u++) {
                        const int e = e0 + gl + G * u;
                        k[u] = e < plen ? acol[p0 + e] : -1;
                    }
                    const int2 *pp[SYM_EU];
                    int np[SYM_EU];
                    int npmax = 0;
#pragma unroll
                    for (int u = 0; u < SYM_EU; u++) {
                        const int4 d = k[u] >= 0 ? desc[k[u]] : make_int4(0, 0, 0, 0);
                        pp[u] = pairs + desc_start(d);
                        np[u] = d.w;   // at most NARROW_PAIRS in a narrow row
                        npmax = max(npmax, np[u]);
                    }
                    for (int tt = 0; tt < npmax; tt++) {
                        int2 x[SYM_EU];
#pragma unroll
                        for (int u = 0; u < SYM_EU; u++) x[u] = tt < np[u] ? pp[u][tt] : make_int2(lo, 0);
#pragma unroll
                        for (int u = 0; u < SYM_EU; u++) {
                            const unsigned wx = (unsigned)(x[u].x - lo);
                            if (wx < (unsigned)NARROW_W) {
                                if (x[u].y) atomicOr(&t[wx], (unsigned)x[u].y);
                            } else {
                                flag |= DERR_COUNT;
                            }
                        }
                    }
                }
            }
            __syncwarp();
            // count, and the list of non-empty words in order with the rank
            // of each word's first column (quads in order, group scans)
            uint2 *ul = ulist + (live ? i : 0) * NARROW_NMAX;
#pragma unroll
            for (int j = 0; j < QPL / P; j++) {
                if (4 * G * P * j >= wide) break;
                uint4 v[P];
                int cl = 0, zl = 0;
#pragma unroll
                for (int pq = 0; pq < P; pq++) {
                    v[pq] = make_uint4(0u, 0u, 0u, 0u);
                    if (nar) v[pq] = *(const uint4 *)&t[4 * quad_of<G, P>(j * P + pq, gl)];
                    cl += __popc(v[pq].x) + __popc(v[pq].y) + __popc(v[pq].z) + __popc(v[pq].w);
                    zl += (v[pq].x != 0) + (v[pq].y != 0) + (v[pq].z != 0) + (v[pq].w != 0);
                }
                int ci = cl, zi = zl;
#pragma unroll
                for (int d = 1; d < G; d <<= 1) {
                    const int y1 = __shfl_up_sync(0xffffffffu, ci, d, G);
                    const int y2 = __shfl_up_sync(0xffffffffu, zi, d, G);
                    if (gl >= d) { ci += y1; zi += y2; }
                }
                int run = cnt + ci - cl, idx = nz + zi - zl;
#pragma unroll
                for (int pq = 0; pq < P; pq++) {
                    const unsigned mw[4] = {v[pq].x, v[pq].y, v[pq].z, v[pq].w};
                    const int w0 = 4 * quad_of<G, P>(j * P + pq, gl);
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        if (nar && mw[u] && idx < NARROW_NMAX)
                            ul[idx] = make_uint2((unsigned)(w0 + u) | ((unsigned)run << 8), mw[u]);
                        idx += mw[u] != 0u;
                        run += __popc(mw[u]);
                    }
                }
                cnt += __shfl_sync(0xffffffffu, ci, G - 1, G);
                nz += __shfl_sync(0xffffffffu, zi, G - 1, G);
            }
            __syncwarp();
        }
        int b = BIN_EMPTY;
        const bool lead = live && gl == 0;
        if (lead) {
            flops[i] = f;
            rspan[i] = make_int2(lo, hi >= lo ? hi - lo + 1 : 0);
            wf += f;
            wl = max(wl, (long long)plen);
            if (nar) {
                b = BIN_NARROW;
                bins[i] = (uint8_t)BIN_NARROW;
                crp[i + 1] = cnt;
                nlo[i] = lo;
                nwords[i] = (uint8_t)min(nz, 255);
            } else {
                const long long keys = cp < (long long)nwords_b ? cp : (long long)nwords_b;
                b = sym_bin(keys, cp);
                if (bitmaps) {
                    if (rowbad) b = BIN_EMPTY;
                    const int mark = b == BIN_EMPTY ? 0 : sym_mark(cp, hi - lo + 1);
                    crp[i + 1] = mark;
                    if (b != BIN_EMPTY) marks[mark != 0] = 1;
                } else {
                    if (b == BIN_EMPTY) crp[i + 1] = 0;
                    if (b == BIN_HUGE) crp[i + 1] = -1;
                }
                bins[i] = (uint8_t)b;
                nlo[i] = -1;
            }
        }
        warp_hist(hist, lead, b);
    }
    if (bad) atomicOr(&st->err, DERR_COL_RANGE);
    if (flag) atomicOr(&st->err, flag);
    for (int d = 16; d > 0; d >>= 1) {
        wf += __shfl_xor_sync(0xffffffffu, wf, d);
        wl = max(wl, __shfl_xor_sync(0xffffffffu, wl, d));
    }
    if (lane == 0 && wf) atomicAdd(&fsum, (unsigned long long)wf);
    if (lane == 0 && wl) atomicMax(&alen_max, (unsigned long long)wl);
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

template <int G>
static int run_sym_narrow(const spgemm_csr &A, const spgemm_csr &B, const int4 *desc, const int2 *bmm,
                          const int2 *pairs, int64_t *flops, uint8_t *bins, int64_t *crp, int2 *rspan, int32_t *nlo,
                          uint8_t *nwords, uint2 *ulist, DevState *st, bool bitmaps, Ctx &c) {
    constexpr int NT = NARROW_SYM_WPB * 32, NR = NARROW_SYM_WPB * (32 / G);
    int64_t blocks = (A.nrows + NR - 1) / NR;
    const int64_t cap = resident_blocks(k_sym_narrow<G>, NT, c.nsm);
    blocks = blocks < cap ? blocks : cap;
    const int64_t nwb = (B.ncols + 31) / 32;
    c.begin("symbolic.narrow", A.nrows);
    k_sym_narrow<G><<<(unsigned)blocks, NT, 0, c.s>>>(A.nrows, B.nrows, nwb, A.row_ptr, A.col_idx, desc, bmm,
                                                      pairs, flops, bins, crp, rspan, nlo, nwords, ulist, st, bitmaps);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_sym_narrow(const spgemm_csr &A, const spgemm_csr &B, const int4 *desc, const int2 *bmm,
                      const int2 *pairs, int64_t *flops, uint8_t *bins, int64_t *crp, int2 *rspan, int32_t *nlo,
                      uint8_t *nwords, uint2 *ulist, DevState *st, bool bitmaps, int G, Ctx &c) {
    if (A.nrows == 0) return SPGEMM_OK;
    switch (G) {
        case 4: return run_sym_narrow<4>(A, B, desc, bmm, pairs, flops, bins, crp, rspan, nlo, nwords, ulist, st, bitmaps, c);
        case 8: return run_sym_narrow<8>(A, B, desc, bmm, pairs, flops, bins, crp, rspan, nlo, nwords, ulist, st, bitmaps, c);
        case 16: return run_sym_narrow<16>(A, B, desc, bmm, pairs, flops, bins, crp, rspan, nlo, nwords, ulist, st, bitmaps, c);
        default: return run_sym_narrow<32>(A, B, desc, bmm, pairs, flops, bins, crp, rspan, nlo, nwords, ulist, st, bitmaps, c);
    }
}

// ---------------------------------------------------------------- numeric
struct NarrowP {
    const int64_t *arp; const int32_t *acol; const void *aval;
    const int32_t *bcol; const void *bval;
    const int64_t *crp; int32_t *ccol; void *cval;
    const int4 *bdesc; const int32_t *nlo; const uint8_t *nwords; const uint2 *ulist; const int32_t *rows;
    int64_t n, nrows_b;   // n: rows of the list, or of A
};

// A staged entry of the product pass: the start of B_k in B (as 32-bit
// halves: with fewer than 2^31 entries in B the high half is free and holds
// the length of B_k), and a_ik.
template <typename V>
struct __align__(16) NarrowEnt {
    int q, hl;
    V a;
};

// popc of the bits of m below bit s (0 <= s < 32): m shifted up by 32 - s,
// a shift of 32 giving 0 (the PTX shift clamps its amount).
__device__ __forceinline__ int popc_below(unsigned m, unsigned s) {
    unsigned r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(m), "r"(32u - s));
    return __popc(r);
}

// Shared memory of k_num_narrow.  Per warp, for its 32/G row slots: the
// window's masks and the rank of each word's first column (a byte: rows
// hold at most NARROW_NMAX < 256 entries), word major and row slot minor,
// so that in one instruction the lanes of different row slots never meet on
// a bank whatever words their rows look up; and the accumulator by rank,
// rank major and row slot minor among the RH rows that one pass over the
// banks serves (half a warp's with 8-byte values): only the lanes of a row
// can meet, on ranks RH apart in the count of banks.  What bounds the kernel
// is these passes over the banks (86% of the peak on the 96^3 Galerkin A*P,
// DRAM 15%): with every slot's ranks adjacent and the slots 34 words apart
// the numeric phase of the 128^3 triple product took 1.45 ms, so 1.43 ms.
// Per row slot: the batch of stored entries ({start, value}, length; the
// lengths apart only when B has 2^31 entries or more), padded so that the
// slots of a warp start on different banks.
template <int G, int WPB, int E, typename V, bool IDX32>
struct NarrowSmem {
    static constexpr int RPW = 32 / G, NR = WPB * RPW, ES = E + 1;
    // rows whose lanes access shared memory in one pass: half a warp's with 8-byte values
    static constexpr int RH = RPW / (sizeof(V) == 8 ? 2 : 1);
    static constexpr int ACC_RS = RH, ACC_SZ = NARROW_NMAX * RPW;
    NarrowEnt<V> ent[NR * ES];
    unsigned tab[WPB * NARROW_W * RPW];
    V acc[WPB * ACC_SZ];
    int elen[IDX32 ? 1 : NR * ES];
    unsigned char base[WPB * NARROW_W * RPW];
};

// Chunks per lane and step in the product pass: their loads of B are issued
// before any of their updates (three: with four, the registers of the
// four-lane kernel leave room for five blocks an SM instead of six).
constexpr int NARROW_U = 3;

// Blocks an SM of the four-lane kernel: six (24 warps; 80 registers a
// thread, 37.4 KB of shared memory a block).  The other lane counts leave
// the register count to the compiler (a minimum of 0 blocks): with eight
// lanes it takes 64 registers, eight blocks an SM.
constexpr int NARROW_MINB4 = 6;

// G lanes per row, 32/G rows per warp, WPB warps per block, batches of E
// stored entries; LIST: the rows of a list, else all rows.  (In elasticity's
// A*P 41% of the rows have more than 32 outputs; taken in row order they left
// two of five row slots idle.)  The row's
// word list (left by the symbolic phase) is scattered into the window table
// and kept in registers for the output (and to clear the table again after
// the row: the table is cleared once at the start and holds only the
// current rows' words).  The product pass walks a staged batch one chunk of
// G entries of B_k at a time, every lane of a row holding the same cursor
// (the current entry's start, value and length); an idle lane loads the
// first entry of B and skips its update (predicated), and so does a column
// missing from the row's window (flagged).  IDX32: B has fewer than 2^31
// entries (32-bit offsets).
template <int G, int WPB, int E, typename V, bool IDX32, bool LIST>
__global__ void __launch_bounds__(WPB * 32, G == 4 ? NARROW_MINB4 : 0) k_num_narrow(NarrowP a, int *err) {
    using S = NarrowSmem<G, WPB, E, V, IDX32>;
    constexpr int RPW = 32 / G, NR = WPB * RPW, U = NARROW_U, EL = E / G;
    constexpr int LPL = NARROW_NMAX / G;
    __shared__ __align__(16) S sm;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / G, gl = lane % G;
    const int slot = w * RPW + g;
    // this row slot's column of the warp's tables: word wd at tab[wd * RPW]
    unsigned *tab = sm.tab + w * NARROW_W * RPW + g;
    unsigned char *base = sm.base + w * NARROW_W * RPW + g;
    V *acc = sm.acc + w * S::ACC_SZ + g / S::RH * (NARROW_NMAX * S::RH) + g % S::RH;
    NarrowEnt<V> *ent = sm.ent + slot * S::ES;
    int *elen = sm.elen + slot * S::ES;
    const V *__restrict__ aval = (const V *)a.aval;
    const V *__restrict__ bval = (const V *)a.bval;
    const int32_t *__restrict__ bcol = a.bcol;
    {
        uint4 *t4 = (uint4 *)(sm.tab + w * NARROW_W * RPW);
#pragma unroll
        for (int q = lane; q < NARROW_W * RPW / 4; q += 32) t4[q] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
    int flag = 0;
    const int64_t stride = (int64_t)gridDim.x * NR;
    for (int64_t rb = (int64_t)blockIdx.x * NR + w * RPW; rb < a.n; rb += stride) {
        bool act = rb + g < a.n;
        const int64_t i = LIST ? (act ? a.rows[rb + g] : 0) : rb + g;
        const int lo = act ? a.nlo[i] : 0;
        const int64_t p0 = act ? a.arp[i] : 0;
        int plen = act ? (int)(a.arp[i + 1] - p0) : 0;
        const int64_t out = act ? a.crp[i] : 0;
        const int nn = act ? (int)(a.crp[i + 1] - out) : 0;
        const int nw = act ? (int)a.nwords[i] : 0;
        if (act && (nn > NARROW_NMAX || nw > nn || lo < 0)) { flag |= DERR_COUNT; act = false; }
        // the row's words: from its list into the window table
        uint2 lw[LPL];
        const uint2 *ul = a.ulist + (act ? i : 0) * NARROW_NMAX;
#pragma unroll
        for (int u = 0; u < LPL; u++) {
            const int x = gl + G * u;
            lw[u] = act && x < nw ? ul[x] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int r = gl; r < NARROW_NMAX; r += G) acc[r * S::ACC_RS] = (V)0;
        int cl = 0;
#pragma unroll
        for (int u = 0; u < LPL; u++) {
            if (lw[u].y == 0u) continue;
            const int wd = (int)(lw[u].x & 0xffu) & (NARROW_W - 1);
            tab[wd * RPW] = lw[u].y;
            base[wd * RPW] = (unsigned char)(lw[u].x >> 8);
            cl += __popc(lw[u].y);
        }
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) cl += __shfl_xor_sync(0xffffffffu, cl, d, G);
        if (act && cl != nn) { flag |= DERR_COUNT; act = false; }
        if (!act) plen = 0;
        const int maxlen = __reduce_max_sync(0xffffffffu, plen);
        __syncwarp();
        // products, a batch of stored entries at a time
        bool bad = false;
        unsigned miss = 0;   // set by a column absent from the row's window union
        for (int pb = 0; pb < maxlen; pb += E) {
            // E lanes to a row, so that a load covers a row's consecutive
            // entries and a store a run of shared memory (with a row's G
            // lanes on its own entries, a load met a line per row: 128^3
            // Galerkin product, both numeric phases, 1.43 -> 1.34 ms)
            const int be = pb + lane % E;
            int k[EL];
            V x[EL];
#pragma unroll
            for (int u = 0; u < EL; u++) {
                const int from = (u * (32 / E) + lane / E) * G;
                const int64_t q = __shfl_sync(0xffffffffu, p0, from) + be;
                const bool ok = be < __shfl_sync(0xffffffffu, plen, from);
                k[u] = ok ? a.acol[q] : -1;
                x[u] = ok ? aval[q] : (V)0;
                if (ok && (unsigned)k[u] >= (unsigned)a.nrows_b) { k[u] = -1; bad = true; }
            }
#pragma unroll
            for (int u = 0; u < EL; u++) {
                int4 d = k[u] >= 0 ? a.bdesc[k[u]] : make_int4(0, 0, 0, 0);
                if (d.z > NARROW_W * 32) { bad = true; d.x = d.y = d.z = 0; }
                const long long q0 = desc_start(d);
                const int at = (w * RPW + u * (32 / E) + lane / E) * S::ES + lane % E;
                NarrowEnt<V> t;
                t.q = (int)(unsigned long long)q0;
                t.hl = IDX32 ? d.z : (int)((unsigned long long)q0 >> 32);
                t.a = x[u];
                sm.ent[at] = t;
                if (!IDX32) sm.elen[at] = d.z;
            }
            __syncwarp();
            const int nb = min(E, plen - pb);
            int e = 0, j = gl, clen = 0;
            long long cq = 0;
            V ca = 0;
            if (nb > 0) {
                const NarrowEnt<V> x = ent[0];
                cq = IDX32 ? (long long)x.q : (long long)(((unsigned long long)(unsigned)x.hl << 32) | (unsigned)x.q);
                ca = x.a;
                clen = IDX32 ? x.hl : elen[0];
            }
            while (__any_sync(0xffffffffu, e < nb)) {
                int c[U], r[U];
                V v[U], av[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const bool ok = j < clen;
                    r[u] = ok ? 0 : NARROW_NMAX;
                    if (IDX32) {
                        const int q = ok ? (int)cq + j : 0;
                        c[u] = bcol[q];
                        v[u] = bval[q];
                    } else {
                        const long long q = ok ? cq + j : 0;
                        c[u] = bcol[q];
                        v[u] = bval[q];
                    }
                    av[u] = ca;
                    j += G;
                    if (j - gl >= clen && e < nb) {
                        e++;
                        j = gl;
                        clen = 0;
                        if (e < nb) {
                            const NarrowEnt<V> x = ent[e];
                            cq = IDX32 ? (long long)x.q
                                       : (long long)(((unsigned long long)(unsigned)x.hl << 32) | (unsigned)x.q);
                            ca = x.a;
                            clen = IDX32 ? x.hl : elen[e];
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int wd = ((c[u] >> 5) - lo) & (NARROW_W - 1);
                    const unsigned m = tab[wd * RPW];
                    const unsigned sh = (unsigned)c[u] & 31u;
                    const int rk = base[wd * RPW] + popc_below(m, sh);
                    const bool hit = (m >> sh) & 1u;
                    const bool live = r[u] == 0;
                    miss |= live && !hit ? 1u : 0u;
                    r[u] = live && hit ? min(rk, NARROW_NMAX) : NARROW_NMAX;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (r[u] < NARROW_NMAX) acc[r[u] * S::ACC_RS] = fma(av[u], v[u], acc[r[u] * S::ACC_RS]);
                    __syncwarp();
                }
            }
            __syncwarp();
        }
        if (miss) flag |= DERR_COUNT;
        if (bad) flag |= DERR_COL_RANGE;
        // write the row in column order (every lane its listed words) and
        // clear the row's words from the table
#pragma unroll
        for (int u = 0; u < LPL; u++) {
            unsigned m = lw[u].y;
            if (m == 0u) continue;
            int rr = (int)(lw[u].x >> 8);
            const int wd = (int)(lw[u].x & 0xffu);
            const int col0 = (lo + wd) * 32;
            tab[(wd & (NARROW_W - 1)) * RPW] = 0u;
            if (act) {
                while (m && rr < nn) {
                    const int bpos = __ffs(m) - 1;
                    m &= m - 1u;
                    a.ccol[out + rr] = col0 + bpos;
                    ((V *)a.cval)[out + rr] = acc[rr * S::ACC_RS];
                    rr++;
                }
            }
        }
        __syncwarp();
    }
    if (flag) atomicOr(err, flag);
}

template <int G, int E, typename V, bool IDX32, bool LIST>
static int run_num_narrow(const NarrowP &p, int *err, Ctx &c) {
    constexpr int WPB = 4, NR = WPB * (32 / G);
    int64_t blocks = (p.n + NR - 1) / NR;
    const int64_t cap = resident_blocks(k_num_narrow<G, WPB, E, V, IDX32, LIST>, WPB * 32, c.nsm);
    blocks = blocks < cap ? blocks : cap;
    c.begin("numeric.narrow", p.n);
    k_num_narrow<G, WPB, E, V, IDX32, LIST><<<(unsigned)blocks, WPB * 32, 0, c.s>>>(p, err);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

template <typename V, bool IDX32, bool LIST>
static int run_num_narrow_g(const NarrowP &p, int *err, int G, Ctx &c) {
    switch (G) {
        case 4: return run_num_narrow<4, 16, V, IDX32, LIST>(p, err, c);
        case 8: return run_num_narrow<8, 32, V, IDX32, LIST>(p, err, c);
        default: return run_num_narrow<16, 32, V, IDX32, LIST>(p, err, c);
    }
}

template <typename V>
static int run_num_narrow_v(const NarrowP &p, bool i32, int *err, int G, Ctx &c) {
    if (p.rows) return i32 ? run_num_narrow_g<V, true, true>(p, err, G, c) : run_num_narrow_g<V, false, true>(p, err, G, c);
    return i32 ? run_num_narrow_g<V, true, false>(p, err, G, c) : run_num_narrow_g<V, false, false>(p, err, G, c);
}

int launch_num_narrow(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                      const int32_t *nlo, const uint8_t *nwords, const uint2 *ulist, const int32_t *rows,
                      int64_t count, int *err, int G, Ctx &c) {
    if (count == 0) return SPGEMM_OK;
    NarrowP p{A.row_ptr, A.col_idx, A.values, B.col_idx, B.values, C.row_ptr, C.col_idx, C.values,
              bdesc, nlo, nwords, ulist, rows, count, B.nrows};
    const bool i32 = B.nnz < ((int64_t)1 << 31);
    return dtype == SPGEMM_F32 ? run_num_narrow_v<float>(p, i32, err, G, c) : run_num_narrow_v<double>(p, i32, err, G, c);
}

// ---------------------------------------------------------------- wider narrow rows
// Narrow rows of 33 to WINDOW_NNZ outputs (block operators: elasticity's
// triple products): the same window table and ranks, WR warps per row.  A
// row's entries are dealt out over subgroups of 16 lanes, each with an
// accumulator of its own: within a subgroup the lanes hold entries of one row
// of B, whose columns are distinct, so an update is a plain read-fma-write (one
// FP64 operation, no atomic, no retry where thousands of products meet in a
// few dozen slots).  The subgroups' sums are added when the row is written.
//
// What bounds it: the chain of loads and the shared-memory lookups of a step
// (20-odd instructions for 32 products); the FP64 floor of the products is a
// third of it.  Measured (one GB300, elasticity on 32^3, FP64): A*P and
// R*(AP), 61,398 such rows, 1.61 -> 0.45 ms against the rank accumulators,
// whose atomics retried on the few slots of a row and of which a row of
// R*(AP) (12,000 products) had one block's share of a chip that 3,969 rows do
// not fill.  The block variant from 4096 products on.  Rows of at most 32
// outputs come here too when they fill less than a wave of warps at eight
// lanes a row: R*(AP) of 45^3 (3375 rows) 0.09 -> 0.03 ms, and the 24 such
// rows of elasticity's R*(AP) 0.15 -> 0.02 ms.
constexpr int WIN_G = 16, WIN_U = 4;

template <typename V, typename Q>
struct WinEnt {
    Q q;
    int len;
    V a;
};

struct WindowP {
    const int64_t *arp; const int32_t *acol; const void *aval;
    const int32_t *bcol; const void *bval;
    const int64_t *crp; int32_t *ccol; void *cval;
    const int4 *bdesc; const int32_t *nlo; const uint8_t *nwords; const uint2 *ulist;
    const int32_t *rows;
    int64_t count, nrows_b;
    int stride;   // slots of an accumulator (odd: the subgroups' start on different banks)
};

template <typename V, typename Q, int WR>
struct WindowSmem {   // per row in flight
    static constexpr int E = WR == 1 ? 64 : WR * 32, NSG = WR * (32 / WIN_G);
    static size_t bytes(int stride) {
        return ((size_t)NSG * stride * sizeof(V) + 15) / 16 * 16 + (sizeof(WinEnt<V, Q>) * E + 15) / 16 * 16 + NARROW_W * 5;
    }
};

template <typename V, typename Q, int WR>
__global__ void __launch_bounds__(256) k_num_window_rows(WindowP a, size_t per_row, int *err) {
    using S = WindowSmem<V, Q, WR>;
    constexpr int NT = WR * 32, RPB = 8 / WR, NSG = S::NSG, E = S::E, U = WIN_U;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int ok_s;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = WR == 1 ? wid : 0, tid = WR == 1 ? lane : (int)threadIdx.x;
    const int sg = tid / WIN_G, gl = tid % WIN_G;
    unsigned char *mine = smem_raw + (size_t)slot * per_row;
    V *acc_all = (V *)mine;
    V *acc = acc_all + sg * a.stride;
    WinEnt<V, Q> *ent = (WinEnt<V, Q> *)(mine + ((size_t)NSG * a.stride * sizeof(V) + 15) / 16 * 16);
    unsigned *tab = (unsigned *)((unsigned char *)ent + (sizeof(WinEnt<V, Q>) * E + 15) / 16 * 16);
    unsigned char *base = (unsigned char *)(tab + NARROW_W);
    const V *__restrict__ aval = (const V *)a.aval;
    const V *__restrict__ bval = (const V *)a.bval;
    const int32_t *__restrict__ bcol = a.bcol;
    auto sync = [] {
        if (WR == 1) __syncwarp();
        else __syncthreads();
    };
    for (int x = tid; x < NARROW_W; x += NT) tab[x] = 0u;
    sync();
    int flag = 0;
    for (int64_t t = (int64_t)blockIdx.x * RPB + slot; t < a.count; t += (int64_t)gridDim.x * RPB) {
        const int i = a.rows ? a.rows[t] : (int)t;
        const int lo = a.nlo[i], nw = a.nwords[i];
        const int64_t p0 = a.arp[i], out = a.crp[i];
        const int plen = (int)(a.arp[i + 1] - p0);
        const int64_t nn64 = a.crp[i + 1] - out;
        const int nn = (int)nn64;
        uint2 lw = make_uint2(0u, 0u);
        bool ok = lo >= 0 && nn64 <= a.stride && nw <= NARROW_NMAX;
        if (WR == 1 || wid == 0) {
            if (ok && lane < nw) lw = a.ulist[(int64_t)i * NARROW_NMAX + lane];
            const int total = __reduce_add_sync(0xffffffffu, __popc(lw.y));
            ok = ok && total == nn;
            if (!ok) lw = make_uint2(0u, 0u);
            if (lw.y) {
                tab[lw.x & (NARROW_W - 1)] = lw.y;
                base[lw.x & (NARROW_W - 1)] = (unsigned char)(lw.x >> 8);
            }
            if (WR > 1 && lane == 0) ok_s = ok;
        }
        for (int x = tid; x < NSG * a.stride; x += NT) acc_all[x] = V(0);
        sync();
        if (WR > 1) ok = ok_s;
        if (!ok) flag |= DERR_COUNT;   // not the pattern of the symbolic phase
        for (int pb = 0; ok && pb < plen; pb += E) {
            const int nb = min(E, plen - pb);
            for (int x = tid; x < nb; x += NT) {
                const int k = a.acol[p0 + pb + x];
                WinEnt<V, Q> en;
                en.q = 0;
                en.len = 0;
                en.a = aval[p0 + pb + x];
                if ((unsigned)k < (unsigned)a.nrows_b) {
                    const int4 d = a.bdesc[k];
                    en.q = (Q)desc_start(d);
                    en.len = d.z;
                } else {
                    flag |= DERR_COL_RANGE;
                }
                ent[x] = en;
            }
            sync();
            int e = sg, j = gl, clen = 0;
            Q cq = 0;
            V ca = V(0);
            if (e < nb) {
                cq = ent[e].q;
                clen = ent[e].len;
                ca = ent[e].a;
            }
            while (__any_sync(0xffffffffu, e < nb)) {
                int c[U], rk[U];
                V v[U], av[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const bool live = j < clen;
                    rk[u] = live ? 0 : -1;
                    c[u] = 0;
                    v[u] = V(0);
                    if (live) {
                        c[u] = bcol[cq + j];
                        v[u] = bval[cq + j];
                    }
                    av[u] = ca;
                    j += WIN_G;
                    if (j - gl >= clen && e < nb) {
                        e += NSG;
                        j = gl;
                        clen = 0;
                        if (e < nb) {
                            cq = ent[e].q;
                            clen = ent[e].len;
                            ca = ent[e].a;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const unsigned wd = (unsigned)((c[u] >> 5) - lo) & (NARROW_W - 1);
                    const unsigned m = tab[wd], sh = (unsigned)c[u] & 31u;
                    const bool hit = (m >> sh) & 1u;
                    if (rk[u] == 0 && !hit) flag |= DERR_COUNT;
                    rk[u] = rk[u] == 0 && hit ? min((int)base[wd] + popc_below(m, sh), a.stride - 1) : -1;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (rk[u] >= 0) acc[rk[u]] = fma(av[u], v[u], acc[rk[u]]);
                    __syncwarp();
                }
            }
            sync();
        }
        if (ok)
            for (int x = tid; x < nn; x += NT) {
                V s = acc_all[x];
#pragma unroll
                for (int y = 1; y < NSG; y++) s += acc_all[y * a.stride + x];
                ((V *)a.cval)[out + x] = s;
            }
        if (lw.y) {
            unsigned m = lw.y;
            int64_t at = out + (int)(lw.x >> 8);
            const int wd = (int)(lw.x & (NARROW_W - 1));
            for (; m; m &= m - 1u) a.ccol[at++] = (lo + wd) * 32 + __ffs(m) - 1;
            tab[wd] = 0u;
        }
        sync();
    }
    if (flag) atomicOr(err, flag);
}

template <typename V, typename Q, int WR>
static int run_window_rows(WindowP &p, int *err, const char *label, Ctx &c) {
    const size_t per_row = (WindowSmem<V, Q, WR>::bytes(p.stride) + 15) / 16 * 16, smem = per_row * (8 / WR);
    int per_sm = 0;
    SG_TRY(kernel_blocks_per_sm((const void *)k_num_window_rows<V, Q, WR>, 256, smem, &per_sm));
    const int64_t blocks = std::min<int64_t>((p.count * WR + 7) / 8, (int64_t)per_sm * c.nsm);
    c.begin(label, p.count);
    k_num_window_rows<V, Q, WR><<<(unsigned)blocks, 256, smem, c.s>>>(p, per_row, err);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_num_window(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                      const int32_t *nlo, const uint8_t *nwords, const uint2 *ulist, const int32_t *rows, int64_t count,
                      bool block, int max_nnz, const char *label, int *err, Ctx &c) {
    if (count <= 0) return SPGEMM_OK;
    WindowP p{A.row_ptr, A.col_idx, A.values, B.col_idx, B.values, C.row_ptr, C.col_idx, C.values,
              bdesc, nlo, nwords, ulist, rows, count, B.nrows, max_nnz | 1};
    auto go = [&](auto v, auto q) -> int {
        using V = decltype(v);
        using Q = decltype(q);
        return block ? run_window_rows<V, Q, 8>(p, err, label, c) : run_window_rows<V, Q, 1>(p, err, label, c);
    };
    const bool i32 = B.nnz < ((int64_t)1 << 31);
    if (dtype == SPGEMM_F32) return i32 ? go(0.f, 0) : go(0.f, 0LL);
    return i32 ? go(0.0, 0) : go(0.0, 0LL);
}

}  // namespace sg
