// Rows of C with more than 32 outputs whose columns span a bitmap that fits
// shared memory: a block per row with a dense rank accumulator (the dense
// accumulator of Section 3.1, restricted to the row's column span).
//
//   1. The row's products a_ik * b_kj are dealt out flat over the block's
//      warps, 32 consecutive products a step.  The stored a_ik are staged in
//      shared memory with the prefix sums of nnz(B_k); a step finds the
//      entries its 32 products belong to from one load of the prefix sums:
//      the entries that start within the step set a bit each (a warp-wide
//      OR), and a product's entry is the number of bits up to its lane.
//   2. Every column is marked in a bitmap of the span; prefix counts of the
//      bitmap's words turn a column into its rank in the sorted row.
//   3. Values are summed by rank and leave together with the columns as two
//      contiguous copies: no hash probe, no sort, coalesced stores.
//
// A row of at most T*U products keeps each product and its column in
// registers between the steps, so B is read once; the lane that marks a
// column first stores its product instead of adding it (no atomic, and no
// second FP64 operation, for the entries that only one product reaches), and
// the others add atomically after a barrier.  Longer rows walk B twice.
//
// What bounds it: instruction issue (2.6 of 4 slots a cycle on rows of about
// 320 products; DRAM 9%, L1 48%), about 2,400 warp instructions a row of
// which some 60% do not depend on the products.  Measured (one GB300):
// 294 M products of 921,066 rows of 4-32 by 4-32 uniform entries (FP32) 9.65
// -> 3.47 ms (3.00 since two warps take the shorter ones, see below) against a
// warp per row with two passes over B, 13 warps an SM
// and stores scattered by word; 41,472 rows of about 4,500 outputs over
// 41,472 columns (FP64) 9.56 -> 1.79 ms (1.87 while a product that is added
// looked its rank up a second time) against a block's hash map with its
// ordering (bin 5) and the window kernel (bin 6).  Blocks of 64 and 32
// threads took 4.1 and 8.7 ms on the first (shared memory then holds too few
// warps), 256 took 5.9; on the second 1024 x 8 took 2.9, 512 x 8 (a second
// walk of B for the longer rows) 2.2 and 256 x 24 2.3 ms.
#include <climits>
#include "internal.cuh"

namespace sg {

// A bitmap word's place in shared memory: 16 words and 4 words of padding in
// turn, so that the 16-word runs that the threads scan start on different
// banks for 16-byte loads (and 8-byte stores of the 16-bit prefix counts).
__device__ __forceinline__ int rank_phys(int w) { return w + ((w >> 4) << 2); }

// Shared memory of a block for bitmaps of bw words (a multiple of 16) and
// rows of nmax outputs.
template <typename V, int T>
struct RankSmem {
    size_t acc, eq, ea, pre, cols, bits, pref, bytes;
    __host__ __device__ RankSmem(int bw, int nmax) {
        size_t o = 0;
        auto take = [&](size_t b) { const size_t p = o; o += (b + 15) & ~(size_t)15; return p; };
        const size_t pw = (size_t)bw + (size_t)bw / 4;
        bits = take(pw * 4);
        pref = take(pw * 2);
        acc = take((size_t)nmax * sizeof(V));
        cols = take((size_t)nmax * 4);
        eq = take((size_t)T * 8);
        ea = take((size_t)T * sizeof(V));
        pre = take((size_t)(T + 40) * 4);
        bytes = o;
    }
};

template <typename V>
struct RankP {
    const int64_t *arp; const int32_t *acol; const V *aval;
    const int32_t *bcol; const V *bval;
    const int64_t *crp; int32_t *ccol; V *cval;
    const int4 *bdesc; const int2 *rspan; const int32_t *rows;
    int64_t count;
    int bw, nmax;
};

// Q: offsets into B (int when it has fewer than 2^31 entries).
template <typename V, typename Q, int T, int U, int MINB>
__global__ void __launch_bounds__(T, MINB) k_num_rank_block(RankP<V> a, int *err) {
    constexpr int NW = T / 32, UB = 4;
    static_assert(U % UB == 0, "products are loaded UB at a time");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int wsum[NW], wcnt[NW];
    const RankSmem<V, T> L(a.bw, a.nmax);
    V *acc = (V *)(smem_raw + L.acc);
    Q *eq = (Q *)(smem_raw + L.eq);                    // start of B_k minus the entry's first product
    V *ea = (V *)(smem_raw + L.ea);
    int *pre = (int *)(smem_raw + L.pre);              // first product of every entry
    int *cols = (int *)(smem_raw + L.cols);
    unsigned *bits = (unsigned *)(smem_raw + L.bits);
    unsigned short *pref = (unsigned short *)(smem_raw + L.pref);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const unsigned below = (1u << lane) - 1u;
    const int32_t *__restrict__ bcol = a.bcol;
    const V *__restrict__ bval = a.bval;
    int flag = 0;
    for (int x = tid; x < (a.bw + a.bw / 4) / 4; x += T) ((uint4 *)bits)[x] = make_uint4(0u, 0u, 0u, 0u);

    // Stage the entries [pb, pb + T) of the row at p0 (those with an empty
    // row of B left out): ne entries of `total` products.  All threads.
    int ne = 0, total = 0;
    auto stage = [&](int64_t p0, int plen, int pb) {
        const int idx = pb + tid;
        int len = 0;
        Q q0 = 0;
        V av = V(0);
        if (idx < plen) {
            const int4 d = a.bdesc[a.acol[p0 + idx]];
            av = a.aval[p0 + idx];
            len = d.z;
            q0 = (Q)desc_start(d);
        }
        int incl = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        const unsigned some = __ballot_sync(0xffffffffu, len > 0);
        if (lane == 31) wsum[w] = incl;
        if (lane == 0) wcnt[w] = __popc(some);
        __syncthreads();
        int base = 0, cb = 0, tot = 0, n = 0;
        const int nwu = min(NW, (plen - pb + 31) >> 5);   // warps that hold entries
        for (int j = 0; j < nwu; j++) {
            const int s = wsum[j], c = wcnt[j];
            if (j < w) { base += s; cb += c; }
            tot += s;
            n += c;
        }
        if (len > 0) {
            const int pos = cb + __popc(some & below), first = base + incl - len;
            pre[pos] = first;
            eq[pos] = q0 - first;
            ea[pos] = av;
        }
        if (tid < 33) pre[n + tid] = INT_MAX;   // a step looks 32 entries ahead
        ne = n;
        total = tot;
        __syncthreads();
    };
    // Last staged entry whose first product is at most t (uniform in a warp).
    auto entry_of = [&](int t) {
        int e = -1;
        for (int j = 0; j < ne; j += 32) {
            const unsigned m = __ballot_sync(0xffffffffu, j + lane < ne && pre[j + lane] <= t);
            e += __popc(m);
            if (m != 0xffffffffu) break;
        }
        return e;
    };
    // Entry of product tc + lane, e0 being the entry of product tc; e0 moves
    // on to the entry of product tc + 32.
    auto step_entry = [&](int tc, int &e0) {
        const int b = pre[e0 + 1 + lane] - tc;
        const unsigned m = __reduce_or_sync(0xffffffffu, b < 32 ? 1u << b : 0u);
        const int e = e0 + __popc(m & (2u * below + 1u));
        e0 += __popc(__ballot_sync(0xffffffffu, b <= 32));
        return e;
    };

    for (int64_t t = blockIdx.x; t < a.count; t += gridDim.x) {
        const int i = a.rows[t];
        const int2 sp = a.rspan[i];
        const int64_t out = a.crp[i];
        const int64_t nn64 = a.crp[i + 1] - out;
        const int bmin = sp.x, nw = sp.y;
        if (nw > a.bw || nw <= 0 || nn64 > a.nmax) continue;   // another kernel's row
        const int nn = (int)nn64;
        const int64_t p0 = a.arp[i];
        const int plen = (int)(a.arp[i + 1] - p0);
        if (plen <= 0) { flag |= DERR_COUNT; continue; }   // A changed since the symbolic phase
        stage(p0, plen, 0);
        const bool once = plen <= T && total <= T * U;
        // products per warp: whole steps of 32, the same number for all warps
        const int per = once ? (((total + 31) >> 5) + NW - 1) / NW : 0;
        int c[U];
        V p[U];
        unsigned mine = 0, first = 0;
        if (once) {
            int tc = w * per * 32;
            int e0 = tc < total ? entry_of(tc) : 0;
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += UB) {
                if (u0 >= per) break;
                int ee[UB];
#pragma unroll
                for (int u = 0; u < UB; u++) {
                    ee[u] = -1;
                    c[u0 + u] = 0;
                    p[u0 + u] = V(0);
                    if (u0 + u < per && tc < total) {   // uniform in the warp
                        const int e = step_entry(tc, e0);
                        if (tc + lane < total) {
                            const Q q = eq[e] + (Q)(tc + lane);
                            ee[u] = e;
                            c[u0 + u] = bcol[q];
                            p[u0 + u] = bval[q];
                        }
                        tc += 32;
                    }
                }
#pragma unroll
                for (int u = 0; u < UB; u++) {
                    if (ee[u] < 0) continue;
                    p[u0 + u] *= ea[ee[u]];
                    const int wd = (c[u0 + u] >> 5) - bmin;
                    if ((unsigned)wd >= (unsigned)nw) { flag |= DERR_COUNT; continue; }
                    const unsigned bit = 1u << (c[u0 + u] & 31);
                    mine |= 1u << (u0 + u);
                    if (!(atomicOr(&bits[rank_phys(wd)], bit) & bit)) first |= 1u << (u0 + u);
                }
            }
        } else {
            for (int x = tid; x < nn; x += T) acc[x] = V(0);
            for (int pb = 0; pb < plen; pb += T) {
                if (pb > 0) stage(p0, plen, pb);
                const int nch = (total + 31) >> 5, pw = (nch + NW - 1) / NW;
                int tc = w * pw * 32;
                const int tend = min(total, tc + pw * 32);
                int e0 = tc < tend ? entry_of(tc) : 0;
                for (; tc < tend; tc += 32) {
                    const int e = step_entry(tc, e0);
                    if (tc + lane < total) {
                        const int col = bcol[eq[e] + (Q)(tc + lane)];
                        const int wd = (col >> 5) - bmin;
                        if ((unsigned)wd >= (unsigned)nw) flag |= DERR_COUNT;
                        else atomicOr(&bits[rank_phys(wd)], 1u << (col & 31));
                    }
                }
                __syncthreads();
            }
        }
        __syncthreads();
        // prefix counts of the bitmap's words: a thread takes 16 words
        int tot = 0;
        {
            uint4 b4[4];
            int s = 0;
            const bool has = tid * 16 < nw;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                b4[j] = has ? *(const uint4 *)&bits[tid * 20 + 4 * j] : make_uint4(0u, 0u, 0u, 0u);
                s += __popc(b4[j].x) + __popc(b4[j].y) + __popc(b4[j].z) + __popc(b4[j].w);
            }
            int incl = s;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            if (lane == 31) wsum[w] = incl;
            __syncthreads();
            int base = 0;
#pragma unroll
            for (int j = 0; j < NW; j++) {
                const int x = wsum[j];
                if (j < w) base += x;
                tot += x;
            }
            if (has) {
                unsigned r = (unsigned)(base + incl - s);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const unsigned r1 = r + __popc(b4[j].x), r2 = r1 + __popc(b4[j].y), r3 = r2 + __popc(b4[j].z);
                    *(uint2 *)&pref[tid * 20 + 4 * j] = make_uint2(r | (r1 << 16), r2 | (r3 << 16));
                    r = r3 + __popc(b4[j].w);
                }
            }
        }
        __syncthreads();
        if (tot == nn) {
            auto rank_of = [&](int col) {
                const int ph = rank_phys((col >> 5) - bmin);
                return (int)pref[ph] + __popc(bits[ph] & ((1u << (col & 31)) - 1u));
            };
            if (once) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (u >= per) break;
                    if (!((mine >> u) & 1u)) continue;
                    const int r = rank_of(c[u]);
                    if ((first >> u) & 1u) {
                        acc[r] = p[u];
                        cols[r] = c[u];
                    } else {
                        c[u] = r;   // only the place is needed from here on
                    }
                }
                mine &= ~first;
                if (__syncthreads_or(mine != 0)) {
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        if (u >= per) break;
                        if ((mine >> u) & 1u) atomicAdd(&acc[c[u]], p[u]);
                    }
                    __syncthreads();
                }
            } else {
                for (int pb = 0; pb < plen; pb += T) {
                    if (plen > T) stage(p0, plen, pb);
                    const int nch = (total + 31) >> 5, pw = (nch + NW - 1) / NW;
                    int tc = w * pw * 32;
                    const int tend = min(total, tc + pw * 32);
                    int e0 = tc < tend ? entry_of(tc) : 0;
                    for (; tc < tend; tc += 32) {
                        const int e = step_entry(tc, e0);
                        if (tc + lane < total) {
                            const Q q = eq[e] + (Q)(tc + lane);
                            const int col = bcol[q];
                            const V v = ea[e] * bval[q];
                            if ((unsigned)((col >> 5) - bmin) < (unsigned)nw) {
                                const int r = rank_of(col);
                                atomicAdd(&acc[r], v);
                                cols[r] = col;
                            }
                        }
                    }
                    __syncthreads();
                }
            }
            for (int x = tid; x < nn; x += T) {
                a.ccol[out + x] = cols[x];
                a.cval[out + x] = acc[x];
            }
        } else {
            flag |= DERR_COUNT;   // not the pattern of the symbolic phase: nothing is written
        }
        if (tid * 16 < nw) {
#pragma unroll
            for (int j = 0; j < 4; j++) *(uint4 *)&bits[tid * 20 + 4 * j] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
    }
    if (flag) atomicOr(err, flag);
}

template <typename V, typename Q, int T, int U, int MINB>
static int run_rank_block(const RankP<V> &p, int *err, const char *label, Ctx &c) {
    auto kern = k_num_rank_block<V, Q, T, U, MINB>;
    const size_t smem = RankSmem<V, T>(p.bw, p.nmax).bytes;
    int per_sm = 0;
    SG_TRY(kernel_blocks_per_sm((const void *)kern, T, smem, &per_sm));
    const int64_t blocks = std::min<int64_t>(p.count, (int64_t)per_sm * c.nsm);
    c.begin(label, p.count);
    kern<<<(unsigned)blocks, T, smem, c.s>>>(p, err);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

// ---------------------------------------------------------------- short rows
// Rows of at most F products: T threads per row (RANK_W_FLOPS with two warps,
// RANK_V_FLOPS with four), the products in their registers, and the bitmap of the span in two levels.  A first bitmap
// holds a bit per 32-column block of the span; its prefix counts number the
// row's non-empty blocks, and only these get a word of the second bitmap.  So
// what is cleared and scanned is a word per 1024 columns and a word per
// non-empty block (at most one per output) instead of a word per 32 columns,
// and shared memory follows the outputs, not the span.
//
//   1. The stored a_ik are staged 32 at a time, one a lane; the row's
//      products 32s .. 32s+31 are slot s / NW of warp s % NW.  Every
//      product's block is marked in the first bitmap.
//   2. Its prefix counts give a product's word of the second bitmap; the lane
//      that sets a bit there first keeps the product as the entry's value.
//   3. The prefix counts of the second bitmap turn a bit into its rank; first
//      products are stored, the others added; values and columns leave as
//      contiguous copies.
// What bounds it: instruction issue (2.3 of 4 slots a cycle; about 2,100 warp
// instructions a row of 290 products, of which loading the products takes
// 360, the two bitmaps 480, the ranks 260, the output 290) and the chain of
// loads and barriers behind it.  Measured (one GB300, FP32): 795,129 rows of
// 64 products of up to 65,536 columns, with the block kernel's 124,998 longer
// ones, 3.47 -> 3.00 ms; 86,197 such rows over 100,000 columns (spans that the
// 128-thread block's bitmap does not hold) 1.36 -> 0.36 ms with the 13,774 of
// 513 to 1024 products beside them; FP64, 299,537
// rows with 48,168 longer ones, 1.45 -> 1.22 ms.  Two warps a row: a warp
// with 16 products a lane takes 3.04 ms for the first (its code no longer
// fits the instruction cache), 128 threads with four a lane 2.83; 96 threads
// for up to 768 products take all its rows at 3.20.
//
// The lanes past a row's last product carry a column of their own beyond the
// span, whose place in every table is one that nothing reads: no branch keeps
// them apart.
template <typename V>
struct RankWSmem {
    int np;   // outputs in whole 16-byte words: the place of what nothing reads
    size_t eq, ea, pre, coarse, cpre, masks, info, cols, acc, bytes;
    __host__ __device__ RankWSmem(int cw, int nmax) {
        size_t o = 0;
        auto take = [&](size_t b) { const size_t p = o; o += (b + 15) & ~(size_t)15; return p; };
        np = (nmax + 3) & ~3;
        eq = take(32 * 8);
        ea = take(32 * sizeof(V));
        pre = take(32 * 4);
        coarse = take((size_t)(cw + 1) * 4);
        cpre = take((size_t)(cw + 1) * 2);
        masks = take((size_t)(np + 1) * 4);
        info = take((size_t)(np + 1) * 4);     // per word: block << 16, then + rank of its first column
        cols = take((size_t)(np + 1) * 4);
        acc = take((size_t)(np + 1) * sizeof(V));
        bytes = o;
    }
};

// bw, nmax of the parameters: words of the first bitmap, outputs.
template <typename V, typename Q, int T, int F, int MINB>
__global__ void __launch_bounds__(T, MINB) k_num_rank_short(RankP<V> a, int *err) {
    constexpr int NW = T / 32, U = F / T, UB = 8;
    static_assert(U * T == F && U % UB == 0, "whole slots");
    extern __shared__ __align__(16) unsigned char mem[];
    __shared__ int s_nz, s_done;
    const RankWSmem<V> L(a.bw, a.nmax);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    Q *eq = (Q *)(mem + L.eq);
    V *ea = (V *)(mem + L.ea), *acc = (V *)(mem + L.acc);
    int *pre = (int *)(mem + L.pre), *cols = (int *)(mem + L.cols);
    unsigned *coarse = (unsigned *)(mem + L.coarse), *masks = (unsigned *)(mem + L.masks), *info = (unsigned *)(mem + L.info);
    unsigned short *cpre = (unsigned short *)(mem + L.cpre);
    const unsigned below = (1u << lane) - 1u, upto = 2u * below + 1u;
    const int none = a.bw * 1024;   // column (less the span's first) of no product
    const int32_t *__restrict__ bcol = a.bcol;
    const V *__restrict__ bval = a.bval;
    int flag = 0;
    for (int x = tid; x < a.bw; x += T) coarse[x] = 0u;
    for (int x = tid; x < L.np; x += T) masks[x] = 0u;
    if (tid == 0) {
        coarse[a.bw] = 0u;
        cpre[a.bw] = (unsigned short)L.np;
        masks[L.np] = 0xffffffffu;   // never the first
    }
    auto scan = [&](int v) {   // inclusive sum over the lanes
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += y;
        }
        return v;
    };

    for (int64_t t = blockIdx.x; t < a.count; t += gridDim.x) {
        const int i = a.rows[t];
        const int2 sp = a.rspan[i];
        const int64_t out = a.crp[i];
        const int nn = (int)(a.crp[i + 1] - out);
        const int col0 = sp.x * 32, ncol = sp.y * 32, cwn = (sp.y + 31) >> 5;
        const int64_t p0 = a.arp[i];
        const int plen = (int)(a.arp[i + 1] - p0);
        if (sp.y <= 0 || cwn > a.bw || nn > a.nmax) { flag |= DERR_COUNT; continue; }
        int c[U];
        V p[U];
#pragma unroll
        for (int u = 0; u < U; u++) c[u] = none;
        int total = 0;
        bool fits = true;
        for (int pb = 0; pb < plen; pb += 32) {   // every warp the same, warp 0 writes
            int len = 0;
            Q q0 = 0;
            if (pb + lane < plen) {
                const int4 d = a.bdesc[a.acol[p0 + pb + lane]];
                len = d.z;
                q0 = (Q)desc_start(d);
            }
            const int incl = scan(len), tot = __shfl_sync(0xffffffffu, incl, 31);
            const unsigned some = __ballot_sync(0xffffffffu, len > 0);
            fits = tot <= F - total && __all_sync(0xffffffffu, len <= F);
            if (!fits) break;   // A or B changed since the symbolic phase
            if (pb > 0) __syncthreads();
            if (w == 0 && len > 0) {
                const int pos = __popc(some & below), at = total + incl - len;
                pre[pos] = at;
                eq[pos] = q0 - at;
                ea[pos] = a.aval[p0 + pb + lane];
            }
            __syncthreads();
            const int at = lane < __popc(some) ? pre[lane] : INT_MAX;   // first product of entry `lane`
            const int tend = total + tot;
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += UB) {
                if (32 * (NW * u0 + w) >= tend) break;
                V av[UB];
#pragma unroll
                for (int u = 0; u < UB; u++) {
                    const int tc = 32 * (NW * (u0 + u) + w), g = tc + lane;
                    av[u] = V(1);
                    if (tc < tend && tc + 32 > total) {
                        // entries that start before the step, and those up to the lane's product
                        const int b = at - tc;
                        const unsigned m = __reduce_or_sync(0xffffffffu, (unsigned)b < 32u ? 1u << b : 0u);
                        const int e = __popc(__ballot_sync(0xffffffffu, b < 0)) + __popc(m & upto) - 1;
                        if (g >= total && g < tend) {
                            const Q q = eq[e] + (Q)g;
                            c[u0 + u] = bcol[q];
                            p[u0 + u] = bval[q];
                            av[u] = ea[e];
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < UB; u++) {
                    const int tc = 32 * (NW * (u0 + u) + w), g = tc + lane;
                    if (tc >= tend) break;
                    p[u0 + u] *= av[u];
                    int &cc = c[u0 + u];
                    if (g >= total && g < tend) {
                        cc -= col0;
                        if ((unsigned)cc >= (unsigned)ncol) {
                            flag |= DERR_COUNT;
                            cc = none;
                        }
                    }
                    atomicOr(&coarse[cc >> 10], 1u << (cc >> 5 & 31));
                }
            }
            total = tend;
        }
        __syncthreads();
        if (w == 0) {
            // prefix counts of the first bitmap's words
            int n = 0;
            for (int x0 = 0; x0 < cwn; x0 += 32) {
                const int x = x0 + lane, s = x < cwn ? __popc(coarse[x]) : 0, incl = scan(s);
                if (x < cwn) cpre[x] = (unsigned short)(n + incl - s);
                n += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) s_nz = n;
        }
        __syncthreads();
        const int nz = s_nz;
        const bool listed = fits && nz <= nn;
        unsigned first = 0, more = 0;
        if (listed) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (32 * (NW * u + w) >= total) break;
                const int x = c[u] >> 10;
                const int k = (int)cpre[x] + __popc(coarse[x] & ((1u << (c[u] >> 5 & 31)) - 1u));
                const unsigned bit = 1u << (c[u] & 31);
                const bool is = !(atomicOr(&masks[k], bit) & bit);
                info[k] = (unsigned)(c[u] >> 5) << 16;
                first |= is ? 1u << u : 0u;
                more |= !is && c[u] != none ? 1u << u : 0u;
                c[u] = (k << 5) | (c[u] & 31);
            }
            __syncthreads();
            if (w == 0) {
                // prefix counts of the second bitmap's words, four a lane
                int n = 0;
                for (int x0 = 0; x0 < nz; x0 += 128) {
                    const int x = x0 + 4 * lane;
                    uint4 v = x < nz ? *(const uint4 *)&masks[x] : make_uint4(0u, 0u, 0u, 0u);
                    v.x = __popc(v.x);
                    v.y = v.x + __popc(v.y);
                    v.z = v.y + __popc(v.z);
                    v.w = v.z + __popc(v.w);
                    const int incl = scan((int)v.w);
                    if (x < nz) {
                        const unsigned r = (unsigned)(n + incl) - v.w;
                        uint4 f = *(const uint4 *)&info[x];
                        f.x += r;
                        f.y += r + v.x;
                        f.z += r + v.y;
                        f.w += r + v.z;
                        *(uint4 *)&info[x] = f;
                    }
                    n += __shfl_sync(0xffffffffu, incl, 31);
                }
                if (lane == 0) s_done = n;
            }
        }
        __syncthreads();
        if (listed && s_done == nn) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (32 * (NW * u + w) >= total) break;
                const int k = c[u] >> 5, b = c[u] & 31;
                const unsigned in = info[k];
                const int r = (int)(in & 0xffffu) + __popc(masks[k] & ((1u << b) - 1u));
                if ((first >> u) & 1u) {
                    acc[r] = p[u];
                    cols[r] = col0 + (int)(in >> 16) * 32 + b;
                }
                c[u] = r;
            }
            if (__syncthreads_or(more != 0)) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (32 * (NW * u + w) >= total) break;
                    if ((more >> u) & 1u) atomicAdd(&acc[c[u]], p[u]);
                }
                __syncthreads();
            }
            for (int x = tid; x < nn; x += T) {
                a.ccol[out + x] = cols[x];
                a.cval[out + x] = acc[x];
            }
        } else {
            flag |= DERR_COUNT;   // not the pattern of the symbolic phase: nothing is written
        }
        if (listed)
            for (int x = 4 * tid; x < nz; x += 4 * T) *(uint4 *)&masks[x] = make_uint4(0u, 0u, 0u, 0u);
        for (int x = tid; x < cwn; x += T) coarse[x] = 0u;
        __syncthreads();
    }
    if (flag) atomicOr(err, flag);
}

template <typename V, typename Q, int T, int F, int MINB>
static int run_rank_short(const RankP<V> &p, int *err, const char *label, Ctx &c) {
    auto kern = k_num_rank_short<V, Q, T, F, MINB>;
    const size_t smem = RankWSmem<V>(p.bw, p.nmax).bytes;
    int per_sm = 0;
    SG_TRY(kernel_blocks_per_sm((const void *)kern, T, smem, &per_sm));
    const int64_t blocks = std::min<int64_t>(p.count, (int64_t)per_sm * c.nsm);
    c.begin(label, p.count);
    kern<<<(unsigned)blocks, T, smem, c.s>>>(p, err);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

template <typename V, typename Q>
static int num_rank(const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc, const int2 *rspan,
                    const int32_t *rows, int64_t count, RankSize size, int64_t max_nnz, int64_t max_words, int *err,
                    Ctx &c) {
    if (size == RANK_SHORT || size == RANK_MID) {
        RankP<V> p{A.row_ptr, A.col_idx, (const V *)A.values, B.col_idx, (const V *)B.values,
                   C.row_ptr, C.col_idx, (V *)C.values, bdesc, rspan, rows, count,
                   (int)((max_words + 31) / 32), (int)max_nnz};
        if (size == RANK_SHORT) return run_rank_short<V, Q, 64, RANK_W_FLOPS, 16>(p, err, "numeric.rank_short", c);
        return run_rank_short<V, Q, 128, RANK_V_FLOPS, 8>(p, err, "numeric.rank_mid", c);
    }
    const int bw = (int)((max_words + 15) & ~(int64_t)15);
    RankP<V> p{A.row_ptr, A.col_idx, (const V *)A.values, B.col_idx, (const V *)B.values,
               C.row_ptr, C.col_idx, (V *)C.values, bdesc, rspan, rows, count, bw, (int)max_nnz};
    if (size == RANK_ROW) return run_rank_block<V, Q, 128, 8, 8>(p, err, "numeric.rank_row", c);
    return run_rank_block<V, Q, 512, 12, 2>(p, err, "numeric.rank_long", c);
}

int launch_num_rank(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                    const int2 *rspan, const int32_t *rows, int64_t count, RankSize size, int64_t max_nnz,
                    int64_t max_words, int *err, Ctx &c) {
    if (count <= 0) return SPGEMM_OK;
    auto go = [&](auto run) { return run(A, B, C, bdesc, rspan, rows, count, size, max_nnz, max_words, err, c); };
    if (B.nnz < ((int64_t)1 << 31) - RANK_FLOPS)   // offsets less a row's first products stay in an int
        return dtype == SPGEMM_F32 ? go(num_rank<float, int>) : go(num_rank<double, int>);
    return dtype == SPGEMM_F32 ? go(num_rank<float, long long>) : go(num_rank<double, long long>);
}

}  // namespace sg
