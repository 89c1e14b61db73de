// Symbolic phase (Section 2.1): nnz(C_i) = | union over stored a_ik of the
// column set of B_k |, computed on compressed column sets: every set is a
// list of (block = col/32, 32-bit mask) pairs, a union is a hash map from
// block to the OR of its masks, and the count is the sum of popcounts
// (Section 2.1: compression turns union into bitwise operations).
//
// When a bitmap of all column blocks of B fits shared memory (up to 1.7 M
// columns), rows with at most 32 pairs take a 32-slot map, G lanes sharing the
// row's stored a_ik, and the others a bitmap of their span, by a warp or a
// block, or, with few pairs over a wide span, a map of their blocks (k_sym_rows).
//
// With a wider B, rows are sized by an upper bound on their distinct blocks.
// A first pass takes every row with bound <= 4096 in row order with the
// 32-slot map; rows that do not fit are marked and, with the rows whose bound
// exceeds 4096, handled by a second pass from row lists.  In bins 2-5 a row whose column blocks span at most
// 2048 blocks takes a warp with a bitmap over its span (k_sym_span); wider
// rows take a warp with a 128- or 512-slot map (bins 2, 3) or a block with
// a 2048- or 8192-slot map (bins 4, 5).  Bin 6 takes a block with a dense
// bitmap over all column blocks (shared memory when it fits, global memory
// otherwise).  Maps live in shared memory (Section 3.3).
#include <climits>
#include "internal.cuh"

namespace sg {


// Per-row-slot layout of k_sym_first in 32-bit words: keys[32], masks[32],
// eq0[E] (int64), pre[E+1]; the stride is padded to G (mod 32) words so that
// the row slots of a warp start on different banks.
template <int G>
struct SymFirstLayout {
    static constexpr int S = SYM_FIRST_SLOTS, E = 32;
    static constexpr int raw = 2 * S + 2 * E + E + 1;
    static constexpr int stride = G == 32 ? ((raw + 1) & ~1) : raw + ((G - raw % 32) + 32) % 32;
    static_assert(stride % 2 == 0, "8-byte arrays need an even stride");
    static constexpr int o_keys = 0, o_masks = S, o_eq0 = 2 * S, o_pre = 2 * S + 2 * E;
};

// First pass: a warp takes 32/G consecutive rows, G lanes per row, 32-slot
// map per row.  The stored a_ik are staged E at a time in shared memory with
// the prefix sums of pairs(B_k); each lane takes a contiguous run of the
// batch's compressed pairs (ceil(total/G) of them), finds its first a_ik
// once by bisection of the prefix sums and walks on in registers, so a pair
// costs one load and one insertion.  Insertions are atomic (CAS on the key,
// OR on the mask).  A row whose map fills up is marked crp[i+1] = -1 and
// counted in its second-pass bin.
// True when the analysis left no row for the first pass (every row empty,
// of the widest bin or narrow: the histogram of the analysis, complete
// before this kernel starts on the same stream); the kernel then returns
// at once instead of reading every row's bin.
// With bitmaps: the rows it left unmarked.
__device__ __forceinline__ bool first_pass_empty(const DevState *st, bool bitmaps) {
    if (bitmaps) return *(volatile const int *)&st->sym_first == 0;
    long long m = 0;
#pragma unroll
    for (int b = 1; b < BIN_HUGE; b++) m += *(volatile const long long *)&st->sym_hist[b];
    return m == 0;
}

// The marked rows' lists: a warp takes 32 rows at a time and reserves their
// places with one atomic per list.
__device__ __forceinline__ void list_marked(int64_t n, const int64_t *__restrict__ crp, int32_t *__restrict__ rows,
                                            int32_t *__restrict__ maps, DevState *st) {
    if (*(volatile int *)&st->sym_marked == 0) return;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n;
         i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + lane;
        const int64_t m = i < n ? crp[i + 1] : 0;
        const unsigned mw = __ballot_sync(0xffffffffu, m == SYM_MARK_WARP), mb = __ballot_sync(0xffffffffu, m == SYM_MARK_BLOCK),
                       mm = __ballot_sync(0xffffffffu, m == SYM_MARK_MAP);
        long long at = 0;
        if (lane == 0 && mw) at = (long long)atomicAdd(&st->sym_warp, (unsigned long long)__popc(mw));
        if (lane == 1 && mb) at = (long long)atomicAdd(&st->sym_block, (unsigned long long)__popc(mb));
        if (lane == 2 && mm) at = (long long)atomicAdd(&st->sym_map, (unsigned long long)__popc(mm));
        const long long aw = __shfl_sync(0xffffffffu, at, 0), ab = __shfl_sync(0xffffffffu, at, 1),
                        am = __shfl_sync(0xffffffffu, at, 2);
        if (m == SYM_MARK_WARP) rows[aw + __popc(mw & below)] = (int32_t)i;
        if (m == SYM_MARK_BLOCK) rows[n - 1 - (ab + __popc(mb & below))] = (int32_t)i;
        if (m == SYM_MARK_MAP) maps[am + __popc(mm & below)] = (int32_t)i;
    }
}

template <int G>
__global__ void __launch_bounds__(256) k_sym_first(
    int64_t n, const uint8_t *__restrict__ bins, const int64_t *__restrict__ arp,
    const int32_t *__restrict__ acol, const int4 *__restrict__ desc,
    const int2 *__restrict__ pairs, int64_t *__restrict__ crp, int32_t *__restrict__ rows, int32_t *__restrict__ maps, DevState *st,
    bool bitmaps) {
    using Lay = SymFirstLayout<G>;
    constexpr int S = Lay::S, L = 5, RPW = 32 / G, WPB = 8, PER = S / G;
    constexpr int E = Lay::E, EL = E / G, NR = WPB * RPW;
    __shared__ __align__(16) int sm[NR * Lay::stride];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / G, gl = lane % G, gbase = g * G;
    const int rs = w * RPW + g;
    int *reg = sm + rs * Lay::stride;
    int *keys = reg + Lay::o_keys;
    unsigned *masks = (unsigned *)(reg + Lay::o_masks);
    long long *eq0 = (long long *)(reg + Lay::o_eq0);
    int *pre = reg + Lay::o_pre;
    const unsigned lmask = (G == 32) ? 0xffffffffu : ((1u << G) - 1);
    const int64_t stride = (int64_t)gridDim.x * WPB * RPW;
    if (bitmaps) list_marked(n, crp, rows, maps, st);
    if (first_pass_empty(st, bitmaps)) return;
    for (int64_t base = ((int64_t)blockIdx.x * WPB + w) * RPW; base < n; base += stride) {
        const int64_t i = base + g;
        const int b = i < n ? bins[i] : 0;
        const bool active = b != BIN_EMPTY && b != BIN_NARROW && (bitmaps ? crp[i + 1] >= 0 : b != BIN_HUGE);
        if (!__any_sync(0xffffffffu, active)) continue;   // rows done elsewhere
        const int64_t p0 = active ? arp[i] : 0;
        const int plen = active ? (int)(arp[i + 1] - p0) : 0;
#pragma unroll
        for (int t = 0; t < PER; t++) {
            keys[gl + t * G] = -1;
            masks[gl + t * G] = 0;
        }
        const int maxlen = __reduce_max_sync(0xffffffffu, plen);
        bool fail = false;
        __syncwarp();
        for (int pb = 0; pb < maxlen; pb += E) {
            int cnt[EL];
            int lsum = 0;
#pragma unroll
            for (int u = 0; u < EL; u++) {
                const int e = gl * EL + u;
                int c = 0;
                if (pb + e < plen) {
                    const int4 d = desc[acol[p0 + pb + e]];
                    c = d.w;
                    eq0[e] = desc_start(d);
                }
                cnt[u] = c;
                lsum += c;
            }
            int incl = lsum;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d, G);
                if (gl >= d) incl += y;
            }
            int run = incl - lsum;
#pragma unroll
            for (int u = 0; u < EL; u++) {
                pre[gl * EL + u] = run;
                run += cnt[u];
            }
            if (gl == G - 1) pre[E] = incl;
            int total = __shfl_sync(0xffffffffu, incl, gbase + G - 1);
            if (fail) total = 0;
            __syncwarp();
            const int chunk = (total + G - 1) / G;
            const int t0 = min(total, gl * chunk), t1 = min(total, t0 + chunk);
            if (t0 < t1) {
                int lo_e = 0, hi_e = E - 1;   // last e with pre[e] <= t0
                while (lo_e < hi_e) {
                    const int mid = (lo_e + hi_e + 1) >> 1;
                    if (pre[mid] <= t0) lo_e = mid; else hi_e = mid - 1;
                }
                int e = lo_e;
                int pe1 = pre[e + 1];
                int64_t q = eq0[e] + (t0 - pre[e]);
                int64_t qend = q + (pe1 - t0);
                for (int t = t0; t < t1 && !fail; t++) {
                    while (q == qend) {
                        e++;
                        const int pa = pre[e];
                        pe1 = pre[e + 1];
                        q = eq0[e];
                        qend = q + (pe1 - pa);
                    }
                    const int2 pr = pairs[q];
                    fail = !sym_insert(keys, masks, L, pr.x, (unsigned)pr.y);
                    q++;
                }
            }
            const unsigned fl = __ballot_sync(0xffffffffu, fail);
            fail = ((fl >> gbase) & lmask) != 0;
            __syncwarp();
        }
        int c = 0;
#pragma unroll
        for (int t = 0; t < PER; t++) c += __popc(masks[gl + t * G]);
        for (int d = G / 2; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (active && gl == 0) {
            if (fail) {
                crp[i + 1] = -1;
                atomicAdd((unsigned long long *)&st->bin_count[0][max(b, 2)], 1ull);
            } else {
                crp[i + 1] = c;
            }
        }
        __syncwarp();
    }
}

// The same first pass with the pairs dealt out in stride (lane l takes the
// t-th pair for t = l, l + G, ...): loads of pairs coalesce within each B_k
// at the cost of a forward-moving cursor in shared memory; faster than the
// contiguous runs when few lanes share a row (G <= 8).
template <int G>
__global__ void __launch_bounds__(256) k_sym_first_strided(
    int64_t n, const uint8_t *__restrict__ bins, const int64_t *__restrict__ arp,
    const int32_t *__restrict__ acol, const int4 *__restrict__ desc,
    const int2 *__restrict__ pairs, int64_t *__restrict__ crp, int32_t *__restrict__ rows, int32_t *__restrict__ maps, DevState *st,
    bool bitmaps) {
    using Lay = SymFirstLayout<G>;
    constexpr int S = Lay::S, L = 5, RPW = 32 / G, WPB = 8, PER = S / G;
    constexpr int E = Lay::E, EL = E / G, NR = WPB * RPW;
    __shared__ __align__(16) int sm[NR * Lay::stride];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / G, gl = lane % G, gbase = g * G;
    const int rs = w * RPW + g;
    int *reg = sm + rs * Lay::stride;
    int *keys = reg + Lay::o_keys;
    unsigned *masks = (unsigned *)(reg + Lay::o_masks);
    long long *eq0 = (long long *)(reg + Lay::o_eq0);
    int *pre = reg + Lay::o_pre;
    const unsigned lmask = (G == 32) ? 0xffffffffu : ((1u << G) - 1);
    const int64_t stride = (int64_t)gridDim.x * WPB * RPW;
    if (bitmaps) list_marked(n, crp, rows, maps, st);
    if (first_pass_empty(st, bitmaps)) return;
    for (int64_t base = ((int64_t)blockIdx.x * WPB + w) * RPW; base < n; base += stride) {
        const int64_t i = base + g;
        const int b = i < n ? bins[i] : 0;
        const bool active = b != BIN_EMPTY && b != BIN_NARROW && (bitmaps ? crp[i + 1] >= 0 : b != BIN_HUGE);
        if (!__any_sync(0xffffffffu, active)) continue;   // rows done elsewhere
        const int64_t p0 = active ? arp[i] : 0;
        const int plen = active ? (int)(arp[i + 1] - p0) : 0;
#pragma unroll
        for (int t = 0; t < PER; t++) {
            keys[gl + t * G] = -1;
            masks[gl + t * G] = 0;
        }
        const int maxlen = __reduce_max_sync(0xffffffffu, plen);
        bool fail = false;
        __syncwarp();
        for (int pb = 0; pb < maxlen; pb += E) {
            int cnt[EL];
            int lsum = 0;
#pragma unroll
            for (int u = 0; u < EL; u++) {
                const int e = gl * EL + u;
                int c = 0;
                if (pb + e < plen) {
                    const int4 d = desc[acol[p0 + pb + e]];
                    c = d.w;
                    eq0[e] = desc_start(d);
                }
                cnt[u] = c;
                lsum += c;
            }
            int incl = lsum;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d, G);
                if (gl >= d) incl += y;
            }
            int run = incl - lsum;
#pragma unroll
            for (int u = 0; u < EL; u++) {
                pre[gl * EL + u] = run;
                run += cnt[u];
            }
            if (gl == G - 1) pre[E] = incl;
            int total = __shfl_sync(0xffffffffu, incl, gbase + G - 1);
            if (fail) total = 0;
            __syncwarp();
            int e = 0;
            const int maxtot = __reduce_max_sync(0xffffffffu, total);
            for (int t0 = 0; t0 < maxtot; t0 += G) {
                const int t = t0 + gl;
                if (t < total && !fail) {
                    while (pre[e + 1] <= t) e++;
                    const int2 pr = pairs[eq0[e] + (t - pre[e])];
                    fail = !sym_insert(keys, masks, L, pr.x, (unsigned)pr.y);
                }
            }
            const unsigned fl = __ballot_sync(0xffffffffu, fail);
            fail = ((fl >> gbase) & lmask) != 0;
            __syncwarp();
        }
        int c = 0;
#pragma unroll
        for (int t = 0; t < PER; t++) c += __popc(masks[gl + t * G]);
        for (int d = G / 2; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (active && gl == 0) {
            if (fail) {
                crp[i + 1] = -1;
                atomicAdd((unsigned long long *)&st->bin_count[0][max(b, 2)], 1ull);
            } else {
                crp[i + 1] = c;
            }
        }
        __syncwarp();
    }
}

// Second pass for rows whose column blocks span at most BW blocks: a warp
// per row ORs the compressed pairs into a bitmap over the span (one word
// per block) and counts its bits; a summary bitmap (one bit per word) lists
// the touched words so that the count and the clean-up visit only those.
// The pairs of the row are dealt out over the lanes through prefix sums of
// pairs(B_k), as in the first pass.  A union of compressed sets by bitwise
// OR, with no hash map (Section 2.1).
constexpr int SPAN_U = 4;   // pairs per lane per step in k_sym_span

template <int BW, int WPB>
struct SpanLayout {
    static constexpr int NS = BW / 32, E = 32;
    static constexpr int words = BW + NS + 2 * E + E + 2;   // bits, summ, eq0 (int64), pre
};

template <int BW, int WPB>
__global__ void __launch_bounds__(WPB * 32) k_sym_span(
    const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const int64_t *__restrict__ brp, const int32_t *__restrict__ ccnt,
    const int2 *__restrict__ pairs, const int2 *__restrict__ rspan, const int32_t *__restrict__ rows,
    int64_t count, int64_t *__restrict__ crp) {
    using Lay = SpanLayout<BW, WPB>;
    constexpr int NS = Lay::NS, E = Lay::E;
    extern __shared__ __align__(16) unsigned span_smem[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned *bits = span_smem + (size_t)w * Lay::words;
    unsigned *summ = bits + BW;
    long long *eq0 = (long long *)(summ + NS);
    int *pre = (int *)(eq0 + E);
    for (int x = lane; x < BW; x += 32) bits[x] = 0;
    for (int x = lane; x < NS; x += 32) summ[x] = 0;
    __syncwarp();
    for (int64_t t = (int64_t)blockIdx.x * WPB + w; t < count; t += (int64_t)gridDim.x * WPB) {
        const int i = rows[t];
        const int2 sp = rspan[i];
        const int bmin = sp.x, nw = sp.y;
        if (nw > BW) continue;
        const int64_t p0 = arp[i];
        const int plen = (int)(arp[i + 1] - p0);
        for (int pb = 0; pb < plen; pb += E) {
            int len = 0;
            if (pb + lane < plen) {
                const int k = acol[p0 + pb + lane];
                len = ccnt[k];
                eq0[lane] = brp[k];
            }
            int incl = len;
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            pre[lane] = incl - len;
            if (lane == 31) pre[E] = incl;
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
            // SPAN_U pairs per lane per step, their loads issued together
            int e = 0;
            for (int t0 = 0; t0 < total; t0 += 32 * SPAN_U) {
                int64_t qq[SPAN_U];
                int2 pr[SPAN_U];
#pragma unroll
                for (int u = 0; u < SPAN_U; u++) {
                    const int tt = t0 + u * 32 + lane;
                    qq[u] = -1;
                    if (tt < total) {
                        while (pre[e + 1] <= tt) e++;
                        qq[u] = eq0[e] + (tt - pre[e]);
                    }
                }
#pragma unroll
                for (int u = 0; u < SPAN_U; u++) pr[u] = qq[u] >= 0 ? pairs[qq[u]] : make_int2(0, 0);
#pragma unroll
                for (int u = 0; u < SPAN_U; u++) {
                    if (qq[u] < 0) continue;
                    const int wd = pr[u].x - bmin;
                    if (atomicOr(&bits[wd], (unsigned)pr[u].y) == 0) atomicOr(&summ[wd >> 5], 1u << (wd & 31));
                }
            }
            __syncwarp();
        }
        const int ns = (nw + 31) / 32;
        int c = 0;
        for (int y = lane; y < ns; y += 32) {
            unsigned sw = summ[y];
            while (sw) {
                const int x = y * 32 + __ffs(sw) - 1;
                sw &= sw - 1;
                c += __popc(bits[x]);
                bits[x] = 0;
            }
            summ[y] = 0;
        }
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0) crp[i + 1] = c;
        __syncwarp();
    }
}

// A warp per row from a row list, S-slot map, lanes walk the pairs of B_k.
template <int S>
__global__ void __launch_bounds__(256) k_sym_warp(
    const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const int64_t *__restrict__ brp, const int32_t *__restrict__ ccnt,
    const int2 *__restrict__ pairs, const int32_t *__restrict__ rows, int64_t count,
    int64_t *__restrict__ crp, int *err, const int2 *__restrict__ rspan, int skip_span) {
    constexpr int L = __builtin_ctz(S), WPB = 8;
    extern __shared__ int smem[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *keys = smem + w * S;
    unsigned *masks = (unsigned *)(smem + WPB * S) + w * S;
    bool fail = false;
    for (int64_t t = (int64_t)blockIdx.x * WPB + w; t < count; t += (int64_t)gridDim.x * WPB) {
        const int i = rows[t];
        if (skip_span > 0 && rspan[i].y <= skip_span) continue;
        for (int s = lane; s < S; s += 32) {
            keys[s] = -1;
            masks[s] = 0;
        }
        __syncwarp();
        const int64_t pe = arp[i + 1];
        for (int64_t p = arp[i]; p < pe; p++) {
            const int k = acol[p];
            const int64_t q0 = brp[k];
            const int cnt = ccnt[k];
            for (int u = lane; u < cnt; u += 32) {
                const int2 pr = pairs[q0 + u];
                fail |= !sym_insert(keys, masks, L, pr.x, (unsigned)pr.y);
            }
        }
        __syncwarp();
        int c = 0;
        for (int s = lane; s < S; s += 32) c += __popc(masks[s]);
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0) crp[i + 1] = c;
        __syncwarp();
    }
    if (fail) atomicOr(err, DERR_PROBE);
}

// A whole block per row; each warp takes stored a_ik in turn and its lanes
// stride over the pairs of B_k.
template <int BS, int S>
__global__ void __launch_bounds__(BS) k_sym_block(
    const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const int64_t *__restrict__ brp, const int32_t *__restrict__ ccnt,
    const int2 *__restrict__ pairs, const int32_t *__restrict__ rows, int64_t count,
    int64_t *__restrict__ crp, int *err, const int2 *__restrict__ rspan, int skip_span) {
    constexpr int L = __builtin_ctz(S);
    extern __shared__ int smem[];
    __shared__ int red[BS / 32];
    int *keys = smem;
    unsigned *masks = (unsigned *)(smem + S);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool fail = false;
    for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
        const int i = rows[t];
        if (skip_span > 0 && rspan[i].y <= skip_span) continue;   // uniform over the block
        for (int s = threadIdx.x; s < S; s += BS) {
            keys[s] = -1;
            masks[s] = 0;
        }
        __syncthreads();
        const int64_t pe = arp[i + 1];
        for (int64_t p = arp[i] + w; p < pe; p += BS / 32) {
            const int k = acol[p];
            const int64_t q0 = brp[k];
            const int n = ccnt[k];
            for (int q = lane; q < n; q += 32) {
                int2 pr = pairs[q0 + q];
                fail |= !sym_insert(keys, masks, L, pr.x, (unsigned)pr.y);
            }
        }
        __syncthreads();
        int c = 0;
        for (int s = threadIdx.x; s < S; s += BS) c += __popc(masks[s]);
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0) red[w] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int j = 0; j < BS / 32; j++) tot += red[j];
            crp[i + 1] = tot;
        }
        __syncthreads();
    }
    if (fail) atomicOr(err, DERR_PROBE);
}

// Dense bitmap of all column blocks (one word per block of 32 columns).
template <int BS>
__global__ void __launch_bounds__(BS) k_sym_bitmap(
    const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const int64_t *__restrict__ brp, const int32_t *__restrict__ ccnt,
    const int2 *__restrict__ pairs, const int32_t *__restrict__ rows, int64_t count,
    int64_t *__restrict__ crp, int64_t nwords, unsigned *gbits) {
    extern __shared__ unsigned sbits[];
    __shared__ long long red[BS / 32];
    unsigned *bits = gbits ? gbits + (size_t)blockIdx.x * (size_t)nwords : sbits;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
        const int i = rows[t];
        for (int64_t s = threadIdx.x; s < nwords; s += BS) bits[s] = 0;
        __syncthreads();
        const int64_t pe = arp[i + 1];
        for (int64_t p = arp[i] + w; p < pe; p += BS / 32) {
            const int k = acol[p];
            const int64_t q0 = brp[k];
            const int n = ccnt[k];
            for (int q = lane; q < n; q += 32) {
                int2 pr = pairs[q0 + q];
                atomicOr(&bits[pr.x], (unsigned)pr.y);
            }
        }
        __syncthreads();
        long long c = 0;
        for (int64_t s = threadIdx.x; s < nwords; s += BS) c += __popc(bits[s]);
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0) red[w] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long tot = 0;
            for (int j = 0; j < BS / 32; j++) tot += red[j];
            crp[i + 1] = tot;
        }
        __syncthreads();
    }
}

constexpr int BITMAP_BS = 512;
constexpr int64_t SMEM_BITMAP_WORDS = SYM_BITMAP_WORDS;

size_t symbolic_global_ws(int64_t ncols_b, int nsm) {
    int64_t nwords = (ncols_b + 31) / 32;
    if (nwords <= SMEM_BITMAP_WORDS) return 0;
    return (size_t)nwords * 4 * (size_t)nsm;
}

// Opt in to the dynamic shared memory a launch needs (static shared memory
// comes on top, so the attribute is set for every non-trivial size).
template <typename K>
static int prep(K kern, size_t smem) {
    if (smem > 16 * 1024)
        SG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return SPGEMM_OK;
}

template <int G>
static int run_first(const spgemm_csr &A, const uint8_t *bins, const int4 *desc, const int2 *pairs,
                     int64_t *crp, int32_t *rows, int32_t *maps, DevState *st, bool bitmaps, Ctx &c) {
    constexpr int GPB = 256 / G;   // rows per block: 8 warps x 32/G rows
    int64_t blocks = (A.nrows + GPB - 1) / GPB;
    // one resident wave striding over the rows: when the analysis left this
    // pass no row, every block returns at once, and a wave costs one round
    // of block launches where 32 blocks an SM cost several
    const int64_t cap = G <= 8 ? resident_blocks(k_sym_first_strided<G>, 256, c.nsm)
                               : resident_blocks(k_sym_first<G>, 256, c.nsm);
    blocks = blocks < cap ? blocks : cap;
    c.begin("symbolic.first", A.nrows);
    if (G <= 8)
        k_sym_first_strided<G><<<(unsigned)blocks, 256, 0, c.s>>>(A.nrows, bins, A.row_ptr, A.col_idx, desc,
                                                                  pairs, crp, rows, maps, st, bitmaps);
    else
        k_sym_first<G><<<(unsigned)blocks, 256, 0, c.s>>>(A.nrows, bins, A.row_ptr, A.col_idx, desc,
                                                       pairs, crp, rows, maps, st, bitmaps);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_symbolic_first(const spgemm_csr &A, const uint8_t *bins, const int4 *desc, const int2 *pairs,
                          int64_t *crp, int32_t *rows, int32_t *maps, DevState *st, bool bitmaps, int G, Ctx &c) {
    if (A.nrows == 0) return SPGEMM_OK;
    switch (G) {
        case 4: return run_first<4>(A, bins, desc, pairs, crp, rows, maps, st, bitmaps, c);
        case 8: return run_first<8>(A, bins, desc, pairs, crp, rows, maps, st, bitmaps, c);
        case 16: return run_first<16>(A, bins, desc, pairs, crp, rows, maps, st, bitmaps, c);
        default: return run_first<32>(A, bins, desc, pairs, crp, rows, maps, st, bitmaps, c);
    }
}

// ---------------------------------------------------------------- marked rows
// Column-set union of a row as a bitwise OR of compressed pairs into a bitmap
// of its span (Section 2.1), by a warp (NT = 32) or a block of NT threads per
// row.  The row's pairs are dealt out flat, 32 consecutive ones a step, as the
// products are in rank.cu: the entries of A are staged with the prefix sums of
// pairs(B_k), the entries that start within a step set a bit each, and a
// pair's entry is the number of bits up to its lane; BM_U steps' loads are in
// flight together.  A block's row meets long rows of B, so there a step that
// ends before the next entry starts reads on without looking anything up (in a
// warp's rows, of 18 pairs an entry, that cost 0.97 -> 1.10 ms).  Then the bitmap is counted and cleared 16 bytes at a time.
// What bounds it: instruction issue and, in rows of a few hundred pairs, the
// chain of loads A -> descriptors -> pairs.  Measured (one GB300, symbolic
// second pass and the first pass whose rows mostly failed it, before -> now):
// batch of 64 products of uniform rows (921,066 rows, 294 M products) 2.9 ->
// 0.94 ms; A*A of an R-MAT graph, scale 17 8.8 -> 2.15 ms (block hash maps of
// 8192 slots before; 2.8 without reading on, 2.2 with four loads in flight),
// scale 13 1.2 -> 0.11 ms (a warp walked rows of up to half a million pairs);
// 41,472 rows of 5,000 pairs 0.78 -> 0.35 ms.  The rows
// are listed and counted without a list length on the host, so the call waits
// for the device once instead of twice.
// MAP: rows over more blocks than the bitmap has (bw) put their pairs into a map
// in its place: what is cleared and counted is then two slots for every pair and
// not the span (internal.cuh has the rule and both sides).
constexpr int BM_U = 8, BM_WPB = 8;

struct BitmapP {
    const int64_t *arp; const int32_t *acol;
    const int4 *desc; const int2 *pairs; const int2 *rspan;
    const int32_t *rows, *maps;
    const uint8_t *bins;
    int64_t n;
    int64_t *crp;
    int bw;   // bitmap words (a multiple of 4)
};

// Adds a block's mask to a map of 2^L slots that is empty where all is zero
// (keys are the blocks plus one); false if full.
__device__ __forceinline__ bool sym_map_add(unsigned *keys, unsigned *masks, int L, int blk, unsigned m) {
    const unsigned key = (unsigned)blk + 1u, msk = (1u << L) - 1u;
    unsigned h = hash_slot(blk, L);
#pragma unroll 1
    for (unsigned probe = 0; probe <= msk; probe++) {
        unsigned k = ((volatile unsigned *)keys)[h];
        if (k == 0u) k = atomicCAS(&keys[h], 0u, key);
        if (k == 0u || k == key) {
            atomicOr(&masks[h], m);
            return true;
        }
        h = (h + 1u) & msk;
    }
    return false;
}

template <int NT>
struct BitmapSmem {   // words per row in flight: bitmap, starts of the entries (8 bytes each), their first pairs
    static constexpr int E = NT, extra = 2 * E + E + 40;
    static size_t bytes(int bw, int rows) { return (size_t)rows * (size_t)(bw + extra) * 4; }
};

template <int NT, bool MAP>
__device__ __forceinline__ void sym_rows(const BitmapP &a, DevState *st, unsigned *bm_smem, int *wsum, int *wcnt,
                                         long long &row_s) {
    constexpr bool WARP = NT == 32;
    constexpr int NW = NT / 32;
    constexpr bool RUNS = !WARP;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tid = WARP ? lane : (int)threadIdx.x, w = WARP ? 0 : wid;
    const unsigned below = (1u << lane) - 1u;
    unsigned *bits = bm_smem + (WARP ? (size_t)wid * (size_t)(a.bw + BitmapSmem<NT>::extra) : 0);
    long long *eq = (long long *)(bits + a.bw);   // start of B_k's pairs minus the entry's first pair
    int *pre = (int *)(eq + NT);                   // first pair of every entry
    auto sync = [] {
        if (WARP) __syncwarp();
        else __syncthreads();
    };
    const int64_t count = (int64_t) * (volatile unsigned long long *)(WARP ? &st->sym_warp : MAP ? &st->sym_map : &st->sym_block);
    if (count == 0) return;
    for (int x = tid; x < a.bw / 4; x += NT) ((uint4 *)bits)[x] = make_uint4(0u, 0u, 0u, 0u);
    int64_t t = WARP ? (int64_t)blockIdx.x * BM_WPB + wid : 0;
    bool fail = false;
    while (true) {
        if (!WARP) {   // rows of very different work: handed out one at a time
            if (tid == 0) row_s = (long long)atomicAdd(MAP ? &st->next_map : &st->next_row, 1ull);
            __syncthreads();
            t = row_s;
        }
        if (t >= count) break;
        const int i = WARP ? a.rows[t] : MAP ? a.maps[t] : a.rows[a.n - 1 - t];
        const int2 sp = a.rspan[i];
        const int lo = sp.x, nw = sp.y;
        const int64_t p0 = a.arp[i];
        const int64_t plen = a.arp[i + 1] - p0;
        // a row over more blocks than the bitmap has: a map by the bound on its blocks
        int L = 0;
        if (MAP && nw > a.bw) {
            const int b = a.bins[i];
            L = !WARP ? SYM_MAP_BLOCK_L : b <= 2 ? 7 : b == 3 ? 9 : SYM_MAP_L;
        }
        sync();
        for (int64_t pb = 0; pb < plen; pb += NT) {
            int len = 0;
            long long q0 = 0;
            if (pb + tid < plen) {
                const int4 d = a.desc[a.acol[p0 + pb + tid]];
                len = d.w;
                q0 = desc_start(d);
            }
            int incl = len;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            const unsigned some = __ballot_sync(0xffffffffu, len > 0);
            int base = 0, cb = 0, total, ne;
            if (WARP) {
                total = __shfl_sync(0xffffffffu, incl, 31);
                ne = __popc(some);
            } else {
                if (lane == 31) wsum[w] = incl;
                if (lane == 0) wcnt[w] = __popc(some);
                __syncthreads();
                const int nwu = (int)min((int64_t)NW, (plen - pb + 31) >> 5);
                const int s = lane < nwu ? wsum[lane] : 0, c = lane < nwu ? wcnt[lane] : 0;
                total = __reduce_add_sync(0xffffffffu, s);
                ne = __reduce_add_sync(0xffffffffu, c);
                base = __reduce_add_sync(0xffffffffu, lane < w ? s : 0);
                cb = __reduce_add_sync(0xffffffffu, lane < w ? c : 0);
            }
            if (len > 0) {
                const int pos = cb + __popc(some & below), first = base + incl - len;
                pre[pos] = first;
                eq[pos] = q0 - first;
            }
            for (int x = tid; x < 33; x += NT) pre[ne + x] = INT_MAX;   // a step looks 32 entries ahead
            sync();
            const int nch = (total + 31) >> 5, pw = (nch + NW - 1) / NW;
            int tc = w * pw * 32;
            const int tend = min(total, tc + pw * 32);
            int e0 = -1;
            if (tc < tend)
                for (int x = 0; x < ne; x += 32) {
                    const unsigned m = __ballot_sync(0xffffffffu, x + lane < ne && pre[x + lane] <= tc);
                    e0 += __popc(m);
                    if (m != 0xffffffffu) break;
                }
            // the entry of the step's first pair, and where the next one starts
            const int2 *row = a.pairs;
            int next = 0;
            if (RUNS && tc < tend) {
                row = a.pairs + eq[e0];
                next = pre[e0 + 1];
            }
            for (; tc < tend; tc += 32 * BM_U) {
                int2 pr[BM_U];
#pragma unroll
                for (int u = 0; u < BM_U; u++) {
                    const int tu = tc + 32 * u;
                    pr[u] = make_int2(lo, 0);
                    if (tu >= tend) continue;   // uniform in the warp
                    if (RUNS && tu + 32 < next) {   // (uniform) one row of B, and it goes on
                        if (tu + lane < total) pr[u] = row[tu + lane];
                        continue;
                    }
                    const int b = pre[e0 + 1 + lane] - tu;
                    const unsigned m = __reduce_or_sync(0xffffffffu, b < 32 ? 1u << b : 0u);
                    const int e = e0 + __popc(m & (2u * below + 1u));
                    e0 += __popc(__ballot_sync(0xffffffffu, b <= 32));
                    if (tu + lane < total) pr[u] = a.pairs[eq[e] + (tu + lane)];
                    if (RUNS) {
                        row = a.pairs + eq[e0];
                        next = pre[e0 + 1];
                    }
                }
                if (MAP && L) {
#pragma unroll 1
                    for (int u = 0; u < BM_U; u++) {
                        int2 x = pr[0];
#pragma unroll
                        for (int y = 1; y < BM_U; y++) if (u == y) x = pr[y];
                        if (x.y != 0 && !sym_map_add(bits + (1 << L), bits, L, x.x, (unsigned)x.y)) fail = true;
                    }
                    continue;
                }
#pragma unroll
                for (int u = 0; u < BM_U; u++) {
                    const unsigned wd = (unsigned)(pr[u].x - lo);
                    if (pr[u].y != 0 && wd < (unsigned)nw) atomicOr(&bits[wd], (unsigned)pr[u].y);
                }
            }
            sync();
        }
        int c = 0;
        const int used = MAP && L ? 1 << L : nw;   // words that hold bits
        for (int x = tid * 4; x < used; x += NT * 4) {
            const uint4 v = *(const uint4 *)&bits[x];
            c += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            *(uint4 *)&bits[x] = make_uint4(0u, 0u, 0u, 0u);
            if (MAP && L) *(uint4 *)&bits[used + x] = make_uint4(0u, 0u, 0u, 0u);
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (WARP) {
            if (lane == 0) a.crp[i + 1] = c;
            t += (int64_t)gridDim.x * BM_WPB;
        } else {
            if (lane == 0) wsum[w] = c;
            __syncthreads();
            if (tid == 0) {
                long long s = 0;
                for (int j = 0; j < NW; j++) s += wsum[j];
                a.crp[i + 1] = s;
            }
        }
        sync();
    }
    if (MAP && fail) atomicOr(&st->err, DERR_PROBE);
}

// The blocks' maps follow the warps' rows in the same launch (a launch of their
// own cost 5 us where B has no such row).
template <int NT, bool MAP>
__global__ void __launch_bounds__(NT == 32 ? BM_WPB * 32 : NT) k_sym_rows(BitmapP a, DevState *st) {
    constexpr int NW = NT == 32 ? BM_WPB : NT / 32;
    extern __shared__ __align__(16) unsigned bm_smem[];
    __shared__ int wsum[NW], wcnt[NW];
    __shared__ long long row_s;
    sym_rows<NT, MAP>(a, st, bm_smem, wsum, wcnt, row_s);
    if (MAP) {
        __syncthreads();
        a.bw = 2 << SYM_MAP_BLOCK_L;
        sym_rows<BM_WPB * 32, true>(a, st, bm_smem, wsum, wcnt, row_s);
    }
}

template <int NT, bool MAP>
static int run_bitmap(const BitmapP &p, DevState *st, const char *label, Ctx &c) {
    const int threads = NT == 32 ? BM_WPB * 32 : NT;
    const size_t smem = BitmapSmem<NT>::bytes(p.bw, NT == 32 ? BM_WPB : 1);
    static_assert(!MAP || BM_WPB * (SYM_WARP_WORDS + BitmapSmem<32>::extra) >= (2 << SYM_MAP_BLOCK_L) + BitmapSmem<BM_WPB * 32>::extra,
                  "a block's map fits where its warps' bitmaps do");
    int per_sm = 0;
    SG_TRY(kernel_blocks_per_sm((const void *)k_sym_rows<NT, MAP>, threads, smem, &per_sm));
    // (with maps a block takes a row too)
    const int64_t blocks = std::min<int64_t>(MAP ? p.n : (p.n * NT + threads - 1) / threads, (int64_t)per_sm * c.nsm);
    c.begin(label, p.n);
    k_sym_rows<NT, MAP><<<(unsigned)blocks, threads, smem, c.s>>>(p, st);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_symbolic_bitmaps(const spgemm_csr &A, const spgemm_csr &B, const int4 *desc, const int2 *pairs,
                            const int2 *rspan, const int32_t *rows, const int32_t *maps, const uint8_t *bins, int64_t *crp,
                            DevState *st, Ctx &c) {
    if (A.nrows == 0) return SPGEMM_OK;
    const int nwords = (int)((B.ncols + 31) / 32);
    BitmapP p{A.row_ptr, A.col_idx, desc, pairs, rspan, rows, maps, bins, A.nrows, crp, (std::min(nwords, SYM_WARP_WORDS) + 3) & ~3};
    if (nwords <= SYM_WARP_WORDS) SG_TRY((run_bitmap<32, false>(p, st, "symbolic.warp_rows", c)));
    else SG_TRY((run_bitmap<32, true>(p, st, "symbolic.warp_rows", c)));
    p.bw = (nwords + 3) & ~3;
    // a block's threads by the blocks that fit an SM beside its bitmap
    if (nwords <= 8192) return run_bitmap<256, false>(p, st, "symbolic.block_rows", c);
    if (nwords <= 24576) return run_bitmap<512, false>(p, st, "symbolic.block_rows", c);
    return run_bitmap<1024, false>(p, st, "symbolic.block_rows", c);
}

static const char *SYM_LABEL[NBINS] = {"", "", "symbolic.bin2", "symbolic.bin3",
                                       "symbolic.bin4", "symbolic.bin5", "symbolic.bin6", ""};

template <int S>
static int run_warp(const spgemm_csr &A, const int64_t *brp, const int32_t *ccnt, const int2 *pairs,
                    const int32_t *rows, int64_t count, int64_t *crp, int *err, int b, Ctx &c,
                    const int2 *rspan, int skip_span) {
    size_t smem = (size_t)8 * S * 8;
    SG_TRY(prep(k_sym_warp<S>, smem));
    int64_t blocks = (count + 7) / 8;
    blocks = blocks < (int64_t)c.nsm * 32 ? blocks : (int64_t)c.nsm * 32;
    c.begin(SYM_LABEL[b], count);
    k_sym_warp<S><<<(unsigned)blocks, 256, smem, c.s>>>(A.row_ptr, A.col_idx, brp, ccnt, pairs, rows,
                                                         count, crp, err, rspan, skip_span);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

template <int BS, int S>
static int run_block(const spgemm_csr &A, const int64_t *brp, const int32_t *ccnt, const int2 *pairs,
                     const int32_t *rows, int64_t count, int64_t *crp, int *err, int b, Ctx &c,
                     const int2 *rspan, int skip_span) {
    size_t smem = (size_t)S * 8;
    SG_TRY(prep(k_sym_block<BS, S>, smem));
    int64_t blocks = count < (int64_t)c.nsm * 16 ? count : (int64_t)c.nsm * 16;
    c.begin(SYM_LABEL[b], count);
    k_sym_block<BS, S><<<(unsigned)blocks, BS, smem, c.s>>>(A.row_ptr, A.col_idx, brp, ccnt, pairs,
                                                            rows, count, crp, err, rspan, skip_span);
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

static const char *SPAN_LABEL[NBINS] = {"", "", "symbolic.span2", "symbolic.span3",
                                        "symbolic.span4", "symbolic.span5", "", ""};
constexpr int SPAN_BW = 2048;

int launch_symbolic(const spgemm_csr &A, const spgemm_csr &B, const int2 *pairs,
                    const int32_t *ccnt, const int32_t *rows, const long long *counts,
                    int64_t *crp, int *err, void *gws, size_t gws_bytes, const int2 *rspan, Ctx &c) {
    const int nsm = c.nsm;
    int64_t off = 0;
    const int64_t *brp = B.row_ptr;
    for (int b = 2; b <= BIN_HUGE; b++) {
        int64_t cnt = counts[b];
        const int32_t *r = rows + off;
        off += cnt;
        if (cnt == 0) continue;
        if (b <= 5) {
            // rows spanning at most SPAN_BW column blocks: bitmap over the span
            constexpr int WPB = 8;
            const size_t smem = (size_t)WPB * SpanLayout<SPAN_BW, WPB>::words * 4;
            SG_TRY(prep(k_sym_span<SPAN_BW, WPB>, smem));
            int64_t blocks = (cnt + WPB - 1) / WPB;
            blocks = blocks < (int64_t)nsm * 32 ? blocks : (int64_t)nsm * 32;
            c.begin(SPAN_LABEL[b], cnt);
            k_sym_span<SPAN_BW, WPB><<<(unsigned)blocks, WPB * 32, smem, c.s>>>(
                A.row_ptr, A.col_idx, brp, ccnt, pairs, rspan, r, cnt, crp);
            c.end();
            SG_CUDA(cudaGetLastError());
        }
        switch (b) {
            case 2: SG_TRY((run_warp<128>(A, brp, ccnt, pairs, r, cnt, crp, err, b, c, rspan, SPAN_BW))); break;
            case 3: SG_TRY((run_warp<512>(A, brp, ccnt, pairs, r, cnt, crp, err, b, c, rspan, SPAN_BW))); break;
            case 4: SG_TRY((run_block<128, 2048>(A, brp, ccnt, pairs, r, cnt, crp, err, b, c, rspan, SPAN_BW))); break;
            case 5: SG_TRY((run_block<256, 8192>(A, brp, ccnt, pairs, r, cnt, crp, err, b, c, rspan, SPAN_BW))); break;
            default: {
                int64_t nwords = (B.ncols + 31) / 32;
                bool shared = nwords <= SMEM_BITMAP_WORDS;
                size_t smem = shared ? (size_t)nwords * 4 : 0;
                SG_TRY(prep(k_sym_bitmap<BITMAP_BS>, smem));
                int64_t blocks = cnt < (int64_t)nsm ? cnt : (int64_t)nsm;
                if (!shared && gws_bytes < (size_t)blocks * (size_t)nwords * 4) {
                    set_error("symbolic: global bitmap workspace too small");
                    return SPGEMM_ERR_INTERNAL;
                }
                c.begin(SYM_LABEL[b], cnt);
                k_sym_bitmap<BITMAP_BS><<<(unsigned)blocks, BITMAP_BS, smem, c.s>>>(
                    A.row_ptr, A.col_idx, brp, ccnt, pairs, r, cnt, crp, nwords,
                    shared ? nullptr : (unsigned *)gws);
                c.end();
                SG_CUDA(cudaGetLastError());
            }
        }
    }
    return SPGEMM_OK;
}

}  // namespace sg
