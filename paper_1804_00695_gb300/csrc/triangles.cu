// Triangle counting by a masked sparse product (the triangle-counting
// experiment of Section 4.1, with Wolf et al.'s formulation that the paper
// uses): the vertices of an undirected graph are relabelled in order of
// non-decreasing degree, L is the strictly lower triangle of the relabelled
// pattern, and the number of triangles is the sum of (L * L) masked by L: for
// every stored L_ik, the columns of L_k that are columns of L_i.
//
// Steps on the device: degrees and a histogram of them (one atomic per
// distinct degree of a warp); an exclusive scan (bucket starts); labels by
// atomic cursors per degree (vertices of equal degree in any order: the count
// does not depend on it, and the labels are returned); L, each row written
// where its vertex's row starts in the graph (it is no longer than that), so
// that its rows need no count of their own before; rows split by work: at most
// TRI_LIGHT_LEN entries and TRI_LIGHT_WORK columns to look up go to a warp each
// with a 256-slot map of row i's blocks (shared memory), the others to a block
// each with a dense bitmap of all columns (shared memory up to TRI_SMEM_WORDS
// words, else a bitmap per block in global memory), set from row i and cleared
// when the block meets another row.  The columns of the rows L_k are dealt out flat, 32
// consecutive ones a step, as the products are in rank.cu.
//
// The paper compresses the right-hand operand into (block, mask) pairs
// (Section 2.1).  The rows of L hold labels, which are not neighbours of one
// another when the vertices are (a pair per column on R-MAT graphs), so the
// pairs only cost their construction and twice the bytes.
//
// Measured (one GB300, R-MAT scale 18, 16 edges a vertex, 0.65e9 lookups): 4.5
// -> 1.1 ms.  Heavy rows 2.7 -> 0.79 ms (a warp took an entry k at a time, its
// lanes the pairs of an L_k that mostly has fewer than 32; 1.21 while a step
// inside one row L_k looked its entry up like any other, 0.81 with four loads
// of a lane in flight instead of six), L 1.02 -> 0.16 ms (counted, then filled,
// a hub's row by one warp 32 entries at a time), degrees and labels 0.19 -> 0.06
// ms (80,000 atomics on the bucket of degree 0).  Now instruction issue bounds
// it, some 14 cycles an SM for 32 lookups.  A hub's row as one block's work took
// 3.6 ms; tasks of 1024, 512 and 256 entries 1.65, 1.25 and 1.21; blocks of 256
// threads 1.29, of 1024 1.42 (these before the steps inside one row).
#include <climits>
#include "internal.cuh"

namespace sg {

constexpr int TRI_LIGHT_LEN = 64;
constexpr long long TRI_LIGHT_WORK = 32768;
constexpr int TRI_MAP_L = 8;             // 256 slots per light row
constexpr int TRI_WPB = 8;
constexpr int64_t TRI_SMEM_WORDS = 48 * 1024;   // 192 KB of bitmap in shared memory
constexpr int TRI_LONG = 1024;           // longer rows of the graph are taken by a block
constexpr int TRI_TASK = 256;            // entries of a heavy row that a block takes at once
constexpr int TRI_ROW_MAX = 1 << 20;     // 1024 rows of at most this many columns fit an int
constexpr int TRI_U = 6;                 // loads of a lane in flight together

// deg[u] (clamped to n - 1 for rows with repeated columns) and its histogram
// in hist[1 + deg] (hist[0] stays 0: the scan then gives bucket starts).
__global__ void k_tri_degree(int64_t n, const int64_t *__restrict__ rp, int32_t *__restrict__ deg,
                             int64_t *__restrict__ hist) {
    const int lane = threadIdx.x & 31;
    for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); u0 < n; u0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = u0 + lane;
        int d = -1;
        if (u < n) {
            d = (int)min(rp[u + 1] - rp[u], n - 1);
            deg[u] = d;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (d >= 0 && lane == __ffs(peers) - 1) atomicAdd((unsigned long long *)&hist[1 + d], (unsigned long long)__popc(peers));
    }
}

// Labels: lab[u] = start of u's degree bucket + its arrival in the bucket.
__global__ void k_tri_label(int64_t n, const int32_t *__restrict__ deg, int64_t *__restrict__ cursor,
                            int32_t *__restrict__ lab, int64_t *__restrict__ perm, int32_t *__restrict__ iperm) {
    const int lane = threadIdx.x & 31;
    for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); u0 < n; u0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = u0 + lane;
        const int d = u < n ? deg[u] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        long long at = 0;
        if (d >= 0 && lane == leader) at = (long long)atomicAdd((unsigned long long *)&cursor[d], (unsigned long long)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
        if (d >= 0) {
            lab[u] = (int32_t)at;
            if (perm) perm[u] = at;
            iperm[at] = (int32_t)u;
        }
    }
}

// Row lab[u] of L: the neighbours of u with a smaller label, in any order, from
// lcol[rp[u]] on; ldesc[label] = {start (int64), entries, 0}.  A warp per
// vertex, TRI_U * 32 entries a step; the vertices of more than TRI_LONG
// entries by the whole block afterwards (their places from a shared counter).
__global__ void __launch_bounds__(256) k_tri_lower(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                                                   const int32_t *__restrict__ lab, int32_t *__restrict__ lcol,
                                                   int4 *__restrict__ ldesc, int *err) {
    __shared__ int64_t longs[64];
    __shared__ int nlong, cnt_s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    if (threadIdx.x == 0) nlong = 0;
    __syncthreads();
    bool bad = false;
    // entries [p, p + 32 * TRI_U) of a row that ends at p1: the labels below pu
    auto take = [&](int64_t p, int64_t p1, int pu, int (&pv)[TRI_U]) {
        int v[TRI_U];
#pragma unroll
        for (int u = 0; u < TRI_U; u++) v[u] = p + 32 * u + lane < p1 ? col[p + 32 * u + lane] : -1;
#pragma unroll
        for (int u = 0; u < TRI_U; u++) {
            pv[u] = INT_MAX;
            if (p + 32 * u + lane >= p1) continue;
            if ((unsigned)v[u] >= (unsigned)n) bad = true;
            else pv[u] = lab[v[u]];
        }
    };
    const int64_t warps = (int64_t)gridDim.x * 8;
    for (int64_t u0 = (int64_t)blockIdx.x * 8; u0 < n; u0 += warps) {
        const int64_t u = u0 + w;
        if (u < n) {
            const int64_t p0 = rp[u], p1 = rp[u + 1];
            const int pu = lab[u];
            bool later = false;
            if (p1 - p0 > TRI_LONG) {
                int at = 64;
                if (lane == 0) at = atomicAdd(&nlong, 1);
                at = __shfl_sync(0xffffffffu, at, 0);
                later = at < 64;   // a full list: this warp takes the row
                if (later && lane == 0) longs[at] = u;
            }
            if (!later) {
                int64_t at = p0;
                for (int64_t p = p0; p < p1; p += 32 * TRI_U) {
                    int pv[TRI_U];
                    take(p, p1, pu, pv);
#pragma unroll
                    for (int x = 0; x < TRI_U; x++) {
                        const unsigned m = __ballot_sync(0xffffffffu, pv[x] < pu);
                        if (pv[x] < pu) lcol[at + __popc(m & below)] = pv[x];
                        at += __popc(m);
                    }
                }
                if (lane == 0) ldesc[pu] = make_int4((int)(unsigned)(uint64_t)p0, (int)((uint64_t)p0 >> 32), (int)(at - p0), 0);
            }
        }
    }
    __syncthreads();
    const int nl = min(nlong, 64);
    for (int t = 0; t < nl; t++) {
        const int64_t u = longs[t], p0 = rp[u], p1 = rp[u + 1];
        const int pu = lab[u];
        __syncthreads();
        if (threadIdx.x == 0) cnt_s = 0;
        __syncthreads();
        for (int64_t p = p0 + (int64_t)w * 32 * TRI_U; p < p1; p += 256 * TRI_U) {
            int pv[TRI_U];
            take(p, p1, pu, pv);
#pragma unroll
            for (int x = 0; x < TRI_U; x++) {
                const unsigned m = __ballot_sync(0xffffffffu, pv[x] < pu);
                int at = 0;
                if (lane == 0 && m) at = atomicAdd(&cnt_s, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (pv[x] < pu) lcol[p0 + at + __popc(m & below)] = pv[x];
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) ldesc[pu] = make_int4((int)(unsigned)(uint64_t)p0, (int)((uint64_t)p0 >> 32), cnt_s, 0);
    }
    if (bad) atomicOr(err, DERR_COL_RANGE);
}

// Rows of L with two entries or more (fewer close no triangle): to the light
// list (at most TRI_LIGHT_LEN entries and TRI_LIGHT_WORK columns of the rows
// they reach) or, in tasks of TRI_TASK entries {row, first entry}, the heavy
// list; counts in cnt[0], cnt[1].  Labels are taken from the top, where the heaviest rows are, so that those start first.  A
// warp hands on its light rows 32 at a time.
__global__ void k_tri_bins(int64_t n, const int32_t *__restrict__ lcol, const int4 *__restrict__ ldesc,
                           int32_t *__restrict__ light, int2 *__restrict__ heavy, unsigned long long *cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    int held = 0, row = 0;
    auto flush = [&]() {
        unsigned long long at = 0;
        if (lane == 0 && held) at = atomicAdd(&cnt[0], (unsigned long long)held);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (lane < held) light[at + lane] = row;
        held = 0;
    };
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < n; t += warps) {
        const int i = (int)(n - 1 - t);
        const int4 d = ldesc[i];
        if (d.z < 2) continue;
        const int64_t p0 = desc_start(d);
        long long wk = TRI_LIGHT_WORK + 1;
        if (d.z <= TRI_LIGHT_LEN) {
            int s = 0;
            for (int p = lane; p < d.z; p += 32) s += min(ldesc[lcol[p0 + p]].z, 2 * (int)TRI_LIGHT_WORK);
            wk = __reduce_add_sync(0xffffffffu, s);
        }
        if (wk > TRI_LIGHT_WORK) {
            const int k = (d.z + TRI_TASK - 1) / TRI_TASK;
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(&cnt[1], (unsigned long long)k);
            at = __shfl_sync(0xffffffffu, at, 0);
            for (int x = lane; x < k; x += 32) heavy[at + x] = make_int2(i, x * TRI_TASK);
        } else if (wk > 0) {
            if (lane == held) row = i;
            if (++held == 32) flush();
        }
    }
    flush();
}

// The columns of the rows L_k of a batch of entries k staged with the prefix
// sums of their lengths (pre, padded with 33 INT_MAX; eq: start less the first
// column's number), dealt out to a warp's share [tc, tend) of them, 32 a step:
// hit(column) for each, by TRI_U steps whose loads are in flight together.  Most
// rows of a hub's entries are longer than a step: a step that ends before the
// next row starts reads on in its row without looking anything up.
template <typename Hit>
__device__ __forceinline__ void tri_walk(const int *pre, const long long *eq, int ne, int tc, int tend, int total,
                                         const int32_t *__restrict__ lcol, int lane, Hit hit) {
    if (tc >= tend) return;
    const unsigned below = (1u << lane) - 1u;
    int e0 = -1;
    for (int x = 0; x < ne; x += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, x + lane < ne && pre[x + lane] <= tc);
        e0 += __popc(m);
        if (m != 0xffffffffu) break;
    }
    // the entry of the step's first column, and where the next one starts
    const int32_t *row = lcol + eq[e0];
    int next = pre[e0 + 1];
    for (; tc < tend; tc += 32 * TRI_U) {
        int c[TRI_U];
#pragma unroll
        for (int u = 0; u < TRI_U; u++) {
            const int tu = tc + 32 * u;
            c[u] = -1;
            if (tu >= tend) continue;   // uniform in the warp
            if (tu + 32 < next) {   // (uniform) the step lies in one row, and so does the next one's start
                if (tu + lane < total) c[u] = row[tu + lane];
                continue;
            }
            const int b = pre[e0 + 1 + lane] - tu;
            const unsigned m = __reduce_or_sync(0xffffffffu, b < 32 ? 1u << b : 0u);
            const int e = e0 + __popc(m & (2u * below + 1u));
            e0 += __popc(__ballot_sync(0xffffffffu, b <= 32));
            if (tu + lane < total) c[u] = lcol[eq[e] + (tu + lane)];
            row = lcol + eq[e0];
            next = pre[e0 + 1];
        }
#pragma unroll
        for (int u = 0; u < TRI_U; u++)
            if (c[u] >= 0) hit(c[u]);
    }
}

// Light rows: a warp per row.  Row i's column set goes into a map of 256
// slots, block -> OR of its bits (atomic CAS on the key, OR on the mask); then
// every column of the rows L_k is looked up in it.
__global__ void __launch_bounds__(TRI_WPB * 32) k_tri_light(
    const int32_t *__restrict__ rows, const unsigned long long *cnt, const int32_t *__restrict__ lcol,
    const int4 *__restrict__ ldesc, const int32_t *__restrict__ iperm, int64_t *__restrict__ vcount,
    unsigned long long *total_out, int *err) {
    constexpr int S = 1 << TRI_MAP_L;
    __shared__ int keys_all[TRI_WPB * S];
    __shared__ unsigned masks_all[TRI_WPB * S];
    __shared__ long long eq_all[TRI_WPB * 32];
    __shared__ int pre_all[TRI_WPB * 72];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int *keys = keys_all + w * S;
    unsigned *masks = masks_all + w * S;
    long long *eq = eq_all + w * 32;
    int *pre = pre_all + w * 72;
    const int64_t nrows = (int64_t)cnt[0];
    const int64_t warps = (int64_t)gridDim.x * TRI_WPB;
    unsigned long long wsum = 0;
    bool full = false;
    for (int64_t t = (int64_t)blockIdx.x * TRI_WPB + w; t < nrows; t += warps) {
        const int i = rows[t];
        for (int s = lane; s < S; s += 32) { keys[s] = -1; masks[s] = 0u; }
        __syncwarp();
        const int4 di = ldesc[i];
        const int64_t p0 = desc_start(di);
        for (int p = lane; p < di.z; p += 32) {
            const int c = lcol[p0 + p];
            full |= !sym_insert(keys, masks, TRI_MAP_L, c >> 5, 1u << (c & 31));
        }
        int rc = 0;
        for (int pb = 0; pb < di.z; pb += 32) {
            int4 d = make_int4(0, 0, 0, 0);
            if (pb + lane < di.z) d = ldesc[lcol[p0 + pb + lane]];
            int incl = d.z;
#pragma unroll
            for (int x = 1; x < 32; x <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, x);
                if (lane >= x) incl += y;
            }
            const unsigned some = __ballot_sync(0xffffffffu, d.z > 0);
            const int ne = __popc(some), total = __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
            if (d.z > 0) {
                const int pos = __popc(some & below);
                pre[pos] = incl - d.z;
                eq[pos] = desc_start(d) - (incl - d.z);
            }
            pre[ne + lane] = INT_MAX;
            if (lane == 0) pre[ne + 32] = INT_MAX;
            __syncwarp();
            tri_walk(pre, eq, ne, 0, total, total, lcol, lane, [&](int c) {
                const int blk = c >> 5;
                unsigned h = hash_slot(blk, TRI_MAP_L);
                int key = keys[h];
                for (int probe = 0; key != blk && key != -1 && probe < S; probe++) {
                    h = (h + 1) & (S - 1);
                    key = keys[h];
                }
                if (key == blk) rc += (masks[h] >> (c & 31)) & 1u;
            });
        }
        rc = __reduce_add_sync(0xffffffffu, rc);   // at most TRI_LIGHT_WORK
        if (lane == 0) {
            if (vcount) vcount[iperm[i]] = rc;
            wsum += (unsigned long long)rc;
        }
        __syncwarp();
    }
    if (full) atomicOr(err, DERR_PROBE);
    if (lane == 0 && wsum) atomicAdd(total_out, wsum);
}

// Heavy rows: a block per task (up to TRI_TASK entries k of a row: the row of a
// hub is several milliseconds of one block), handed out one at a time, with a
// bitmap of all columns (bm: shared memory, or this block's region of gbm): row
// i's bits are set and every column of the rows L_k is looked up.  A row's tasks
// come one after another, so a block keeps the bits of its row until it meets
// another one: they are set and cleared once for each block that works on the
// row, not once for each of its d / TRI_TASK tasks (a star of 8 million leaves,
// whose row has nothing to look up: 2264 -> 20 ms).
template <int T, bool SMEM>
__global__ void __launch_bounds__(T) k_tri_heavy(
    const int2 *__restrict__ tasks, unsigned long long *cnt, const int32_t *__restrict__ lcol,
    const int4 *__restrict__ ldesc, const int32_t *__restrict__ iperm, int64_t *__restrict__ vcount,
    unsigned long long *total_out, int64_t nwords, unsigned *gbm) {
    constexpr int NW = T / 32;
    extern __shared__ unsigned tri_smem[];
    __shared__ unsigned long long red[NW];
    __shared__ long long eq[T], row_s;
    __shared__ int pre[T + 40], wsum[NW], wcnt[NW];
    unsigned *bm = SMEM ? tri_smem : gbm + (int64_t)blockIdx.x * nwords;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int64_t nrows = (int64_t)cnt[1];
    if (nrows == 0) return;
    for (int64_t x = threadIdx.x; x < nwords; x += T) bm[x] = 0u;
    unsigned long long bsum = 0;
    int held = -1;   // the row whose bits are set
    while (true) {
        if (threadIdx.x == 0) row_s = (long long)atomicAdd(&cnt[2], 1ull);
        __syncthreads();   // (and the last task's lookups are through)
        if (row_s >= nrows) break;
        const int2 task = tasks[row_s];
        const int i = task.x;
        const int4 di = ldesc[i];
        const int64_t p0 = desc_start(di);
        if (i != held) {
            if (held >= 0) {
                const int4 dh = ldesc[held];
                const int64_t h0 = desc_start(dh);
                for (int p = threadIdx.x; p < dh.z; p += T) bm[lcol[h0 + p] >> 5] = 0u;
            }
            __syncthreads();
            for (int p = threadIdx.x; p < di.z; p += T) {
                const int c = lcol[p0 + p];
                atomicOr(&bm[c >> 5], 1u << (c & 31));
            }
            held = i;
        }
        unsigned long long rc = 0;
        const int pend = min(di.z, task.y + TRI_TASK);
        for (int pb = task.y; pb < pend; pb += T) {
            int4 d = make_int4(0, 0, 0, 0);
            if (pb + (int)threadIdx.x < pend) d = ldesc[lcol[p0 + pb + threadIdx.x]];
            if (__syncthreads_or(d.z > TRI_ROW_MAX)) {   // the batch's columns might not fit an int: row by row
                for (int p = pb; p < min(pend, pb + T); p++) {
                    const int4 dk = ldesc[lcol[p0 + p]];
                    const int64_t q0 = desc_start(dk);
                    for (int q = threadIdx.x; q < dk.z; q += T) {
                        const int c = lcol[q0 + q];
                        rc += (bm[c >> 5] >> (c & 31)) & 1u;
                    }
                }
                __syncthreads();
                continue;
            }
            int incl = d.z;
#pragma unroll
            for (int x = 1; x < 32; x <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, x);
                if (lane >= x) incl += y;
            }
            const unsigned some = __ballot_sync(0xffffffffu, d.z > 0);
            if (lane == 31) wsum[w] = incl;
            if (lane == 0) wcnt[w] = __popc(some);
            __syncthreads();
            const int s = lane < NW ? wsum[lane] : 0, k = lane < NW ? wcnt[lane] : 0;
            const int total = __reduce_add_sync(0xffffffffu, s), ne = __reduce_add_sync(0xffffffffu, k);
            const int base = __reduce_add_sync(0xffffffffu, lane < w ? s : 0), cb = __reduce_add_sync(0xffffffffu, lane < w ? k : 0);
            if (d.z > 0) {
                const int pos = cb + __popc(some & below), first = base + incl - d.z;
                pre[pos] = first;
                eq[pos] = desc_start(d) - first;
            }
            if (threadIdx.x < 33) pre[ne + threadIdx.x] = INT_MAX;
            __syncthreads();
            const int per = (((total + 31) >> 5) + NW - 1) / NW * 32;   // whole steps, the same for all warps
            unsigned hits = 0;
            tri_walk(pre, eq, ne, w * per, min(total, (w + 1) * per), total, lcol, lane,
                     [&](int c) { hits += (bm[c >> 5] >> (c & 31)) & 1u; });
            rc += hits;
            __syncthreads();
        }
        for (int x = 16; x > 0; x >>= 1) rc += __shfl_xor_sync(0xffffffffu, rc, x);
        if (lane == 0) red[w] = rc;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long s = 0;
            for (int x = 0; x < NW; x++) s += red[x];
            if (vcount && s) atomicAdd((unsigned long long *)&vcount[iperm[i]], s);
            bsum += s;
        }
    }
    if (threadIdx.x == 0 && bsum) atomicAdd(total_out, bsum);
}

size_t triangles_ws(int64_t n, int64_t nnz, int nsm) {
    const int64_t nwords = (n + 31) / 32;
    size_t b = 0;
    auto add = [&](size_t x) { b += (x + 255) & ~(size_t)255; };
    add((size_t)n * 4);              // deg
    add((size_t)(n + 1) * 8);        // hist / cursor
    add((size_t)n * 4);              // labels
    add((size_t)n * 4);              // iperm
    add((size_t)n * 16);             // ldesc
    add((size_t)nnz * 4);            // lcol
    add((size_t)n * 4);              // light list
    add((size_t)(n + nnz / TRI_TASK) * 8);   // heavy tasks
    add(64);                         // counters
    add(scan_tmp_bytes(n));
    if (nwords > TRI_SMEM_WORDS) add((size_t)nsm * (size_t)nwords * 4);
    return b;
}

int launch_triangles(const spgemm_csr &A, void *ws, int64_t *perm_out, int64_t *vcount, unsigned long long *total,
                     int *err, Ctx &c) {
    const int64_t n = A.nrows, nnz = A.nnz, nwords = (n + 31) / 32;
    char *w = (char *)ws;
    auto take = [&](size_t x) { char *p = w; w += (x + 255) & ~(size_t)255; return p; };
    int32_t *deg = (int32_t *)take((size_t)n * 4);
    int64_t *hist = (int64_t *)take((size_t)(n + 1) * 8);
    int32_t *lab = (int32_t *)take((size_t)n * 4);
    int32_t *iperm = (int32_t *)take((size_t)n * 4);
    int4 *ldesc = (int4 *)take((size_t)n * 16);
    int32_t *lcol = (int32_t *)take((size_t)nnz * 4);
    int32_t *light = (int32_t *)take((size_t)n * 4);
    int2 *heavy = (int2 *)take((size_t)(n + nnz / TRI_TASK) * 8);
    unsigned long long *cnt = (unsigned long long *)take(64);   // light rows, heavy tasks, heavy tasks handed out
    void *tmp = take(scan_tmp_bytes(n));
    unsigned *gbm = (unsigned *)w;
    const unsigned g1 = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c.nsm * 16);
    const unsigned gw = (unsigned)std::min<int64_t>((n + 7) / 8, (int64_t)c.nsm * 32);
    SG_CUDA(cudaMemsetAsync(hist, 0, (size_t)(n + 1) * 8, c.s));
    SG_CUDA(cudaMemsetAsync(cnt, 0, 64, c.s));
    SG_CUDA(cudaMemsetAsync(total, 0, sizeof(unsigned long long), c.s));
    if (vcount) SG_CUDA(cudaMemsetAsync(vcount, 0, (size_t)n * 8, c.s));
    c.begin("triangles.degree", n);
    k_tri_degree<<<g1, 256, 0, c.s>>>(n, A.row_ptr, deg, hist);
    c.end();
    SG_TRY(launch_scan_counts(hist, n, (long long *)(cnt + 4), tmp, c));   // hist -> bucket starts
    c.begin("triangles.label", n);
    k_tri_label<<<g1, 256, 0, c.s>>>(n, deg, hist, lab, perm_out, iperm);
    c.end();
    c.begin("triangles.lower", n);
    k_tri_lower<<<(unsigned)std::min<int64_t>((n + 7) / 8, resident_blocks(k_tri_lower, 256, c.nsm)), 256, 0, c.s>>>(
        n, A.row_ptr, A.col_idx, lab, lcol, ldesc, err);
    c.end();
    c.begin("triangles.bins", n);
    k_tri_bins<<<gw, 256, 0, c.s>>>(n, lcol, ldesc, light, heavy, cnt);
    c.end();
    c.begin("triangles.light", n);
    k_tri_light<<<(unsigned)((int64_t)c.nsm * 8), TRI_WPB * 32, 0, c.s>>>(light, cnt, lcol, ldesc, iperm, vcount, total, err);
    c.end();
    // a block's threads by the blocks that fit an SM beside its bitmap
    auto heavy_rows = [&](auto kern, int T, bool smem) -> int {
        const size_t bytes = smem ? (size_t)nwords * 4 : 0;
        int per_sm = 1;
        if (smem) SG_TRY(kernel_blocks_per_sm((const void *)kern, T, bytes, &per_sm));
        c.begin("triangles.heavy", n);
        kern<<<(unsigned)((int64_t)c.nsm * per_sm), T, bytes, c.s>>>(heavy, cnt, lcol, ldesc, iperm, vcount, total, nwords, gbm);
        c.end();
        SG_CUDA(cudaGetLastError());
        return SPGEMM_OK;
    };
    if (nwords <= 24576) return heavy_rows(k_tri_heavy<512, true>, 512, true);
    if (nwords <= TRI_SMEM_WORDS) return heavy_rows(k_tri_heavy<1024, true>, 1024, true);
    return heavy_rows(k_tri_heavy<512, false>, 512, false);
}

}  // namespace sg
