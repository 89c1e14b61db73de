// Rows of C with many products over their column span, rows of B sorted: a
// block per row with a dense accumulator (the dense accumulator of Section
// 3.1) over windows of W columns held in shared memory.  Every window's part
// of each row of B is found in a table of split offsets made once per call,
// so the products of a window are dealt out evenly over the block's warps
// whatever the lengths of the rows of B: whole strips of 64 entries of one
// row of B to a warp each, with nothing to look up inside, and the last 1 to
// 64 entries of every part flat, 32 consecutive products a step (found as in
// rank.cu); either way the loads of B are coalesced.
//
// A slot that no product has reached holds -0.0, which no sum of products
// can give: a product that is -0.0 is added as +0.0, and a sum is -0.0 only
// if every term is.  So a slot says by itself whether it is an entry of C,
// and a product costs one shared-memory update (a bitmap of touched columns
// would cost a second one, on a word that neighbouring lanes share).  The
// window's entries leave in column order, compacted by ballots.
//
// What bounds it: shared-memory updates and the loads that feed them, about
// 27 cycles an SM for 32 products where the update alone takes 9.4 (random
// words), and 5 of the 13.9 ms below for staging and writing out windows.
// Measured (one GB300, FP32, A*A of an R-MAT graph of scale 17: 3.3e9
// products in 39,071 rows of 8192 to 131,072 outputs): 40.8 -> 13.9 ms
// against a window kernel in which one lane walked each short part (loads of
// a warp on 32 lines) and every product marked a bitmap. Of that: even dealing
// 19.4, permuted slots 16.7, rows handed out one at a time 14.7, two blocks
// of 512 threads an SM and strips of 64 14.4, the flat products loaded in
// place 13.9. Blocks of 256 threads over 44 KB took 19.4 before the last
// three. Everything flat, steps inside one part read on without a lookup,
// takes 15.1 (and 5.8 for 6.3 ms on 41,448 FP64 rows of 16,000 products whose
// parts have about 50), strips of 128 14.0 (6.7).
#include <climits>
#include "internal.cuh"

namespace sg {

__device__ __forceinline__ float dense_empty(float) { return __int_as_float(0x80000000); }
__device__ __forceinline__ double dense_empty(double) { return __hiloint2double(0x80000000, 0); }
__device__ __forceinline__ bool dense_has(float v) { return __float_as_uint(v) != 0x80000000u; }
__device__ __forceinline__ bool dense_has(double v) {
    return __double2loint(v) != 0 || (unsigned)__double2hiint(v) != 0x80000000u;
}
// a*b with -0.0 as +0.0 (in FP64 by the words: an addition would take a
// second operation of the few FP64 units)
__device__ __forceinline__ float dense_prod(float a, float b) { return __fadd_rn(__fmul_rn(a, b), 0.f); }
__device__ __forceinline__ double dense_prod(double a, double b) {
    const double p = __dmul_rn(a, b);
    return dense_has(p) ? p : 0.0;
}

// A column's slot: the 32 slots of a run of 32 columns are permuted by the
// run's number, which keeps neighbouring columns on different banks and
// spreads columns whose low bits repeat (in R-MAT graphs a quarter of all
// entries have five zero low bits).
__device__ __forceinline__ int dense_perm(int run) { return (run ^ (run >> 5)) & 31; }
__device__ __forceinline__ unsigned dense_slot(unsigned x) { return x ^ (unsigned)dense_perm((int)(x >> 5)); }

// split[k * (nwin - 1) + j]: entries of B_k below column (j + 1) * W.
__global__ void k_dense_split(int64_t nrows, const int64_t *__restrict__ brp, const int32_t *__restrict__ bcol, int W,
                              int nwin, int32_t *__restrict__ split) {
    const int64_t total = nrows * (nwin - 1);
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = x / (nwin - 1);
        const int64_t lim = (x - k * (nwin - 1) + 1) * W;
        const int64_t q0 = brp[k];
        int64_t lo = q0, hi = brp[k + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (bcol[mid] < lim) lo = mid + 1;
            else hi = mid;
        }
        split[x] = (int32_t)(lo - q0);
    }
}

template <typename V>
struct DenseP {
    const int64_t *arp; const int32_t *acol; const V *aval;
    const int32_t *bcol; const V *bval;
    const int64_t *crp; int32_t *ccol; V *cval;
    const int4 *bdesc; const int2 *rspan; const int32_t *rows; const int32_t *split;
    int64_t count;
    int W, nwin;
    unsigned long long *next;   // rows handed out so far
    V *fold;                    // W sums for every block (null: none)
};

// In FP32 a slot takes the terms of at most DENSE_FOLD batches of a row's
// entries (1024 with blocks of 256 threads, 2048 with 512) before the window is added to sums of its own in global memory (L2):
// a hub's entries are sums of tens of thousands of terms, and the rounding of
// one long chain of additions grows with its length.  A*A of an R-MAT graph of
// scale 17 against 64 bits (2-norms): 3.6e-7 to 1.2e-6 -> 1.6e-7, for 13.9 ->
// 14.2 ms.  FP64 goes without: its registers would spill (6.3 -> 7.1 ms at
// scale 16), and its chains keep far more digits than the result needs.
constexpr int DENSE_FOLD = 4;

template <typename V, int T>
struct DenseSmem {
    size_t acc, eq, ea, pre, str, bytes;
    __host__ __device__ explicit DenseSmem(int W) {
        size_t o = 0;
        auto take = [&](size_t b) { const size_t p = o; o += (b + 15) & ~(size_t)15; return p; };
        acc = take((size_t)W * sizeof(V));
        eq = take((size_t)T * 8);
        ea = take((size_t)T * sizeof(V));
        pre = take((size_t)(T + 40) * 4);
        str = take((size_t)(T + 1) * 4);
        bytes = o;
    }
};

constexpr int DENSE_STRIP_L = 6, DENSE_STRIP = 1 << DENSE_STRIP_L;   // entries of B a warp takes at once

template <typename V, int T, int MINB>
__global__ void __launch_bounds__(T, MINB) k_num_dense(DenseP<V> a, int *err) {
    constexpr int NW = T / 32, U = DENSE_STRIP / 32, F = 2, VW = 16 / (int)sizeof(V);   // values per 16 bytes
    constexpr bool FOLDS = sizeof(V) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int wsum[NW], wcnt[NW], wstr[NW];
    __shared__ long long row_s;
    const DenseSmem<V, T> L(a.W);
    V *acc = (V *)(smem_raw + L.acc);
    // per part of a row of B: where its flat products start, less the first
    // of them; a_ik; its first flat product; its first strip
    long long *eq = (long long *)(smem_raw + L.eq);
    V *ea = (V *)(smem_raw + L.ea);
    int *pre = (int *)(smem_raw + L.pre);
    int *str = (int *)(smem_raw + L.str);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const unsigned below = (1u << lane) - 1u;
    const int32_t *__restrict__ bcol = a.bcol;
    const V *__restrict__ bval = a.bval;
    const int W = a.W, runs = W / 32 / NW;   // runs of 32 columns that a warp writes out
    for (int x = tid; x < W; x += T) acc[x] = dense_empty(V(0));
    int flag = 0;
    __syncthreads();
    // rows are handed out one at a time: their products differ by orders of
    // magnitude, and the heavy rows of a power-law graph come first
    while (true) {
        if (tid == 0) row_s = (long long)atomicAdd(a.next, 1ull);
        __syncthreads();
        const int64_t t = row_s;
        if (t >= a.count) break;
        const int i = a.rows[t];
        const int2 sp = a.rspan[i];
        const int64_t out = a.crp[i], expect = a.crp[i + 1] - out;
        const int64_t p0 = a.arp[i];
        const int plen = (int)(a.arp[i + 1] - p0);
        if (sp.y <= 0 || plen <= 0) {   // A changed since the symbolic phase
            flag |= DERR_COUNT;
            __syncthreads();
            continue;
        }
        const int j0 = (int)((int64_t)sp.x * 32 / W), j1 = (int)(((int64_t)(sp.x + sp.y) * 32 - 1) / W);
        int64_t written = 0;
        // this thread's entry of a batch: a_ik, the start and length of B_k,
        // its splits; kept from window to window when the row is one batch,
        // the next split loaded a window ahead
        V av = V(0);
        int blen = 0, s0 = 0, s1 = 0;
        long long bq = 0;
        const int32_t *sk = nullptr;
        auto entry = [&](int idx, int j) {
            blen = s0 = s1 = 0;
            if (idx < plen) {
                const int k = a.acol[p0 + idx];
                const int4 d = a.bdesc[k];
                sk = a.split + (int64_t)k * (a.nwin - 1);
                av = a.aval[p0 + idx];
                blen = d.z;
                bq = desc_start(d);
                s0 = j == 0 ? 0 : sk[j - 1];
                s1 = j == a.nwin - 1 ? blen : sk[j];
            }
        };
        const bool single = plen <= T;
        if (single) entry(tid, j0);
        for (int j = j0; j <= j1 && j < a.nwin; j++) {
            const int64_t w0 = (int64_t)j * W;
            bool folded = false;
            V *sums = FOLDS && a.fold ? a.fold + (int64_t)blockIdx.x * W : nullptr;
            for (int pb = 0; pb < plen; pb += T) {
                // stage the parts of up to T rows of B inside the window (empty ones left out)
                if (!single) entry(pb + tid, j);
                const int len = s1 - s0;
                const long long q0 = bq + s0;
                if (single) {   // the next window's split
                    s0 = s1;
                    if (blen > 0) s1 = j + 1 >= a.nwin - 1 ? blen : sk[j + 1];
                }
                // 1 to DENSE_STRIP flat products after whole strips
                const int ns = len > 0 ? (len - 1) >> DENSE_STRIP_L : 0, flat = len - (ns << DENSE_STRIP_L);
                int incl = flat, sincl = ns;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, d), z = __shfl_up_sync(0xffffffffu, sincl, d);
                    if (lane >= d) { incl += y; sincl += z; }
                }
                const unsigned some = __ballot_sync(0xffffffffu, len > 0);
                if (lane == 31) { wsum[w] = incl; wstr[w] = sincl; }
                if (lane == 0) wcnt[w] = __popc(some);
                __syncthreads();
                int base, cb, sb, total, ne, strips;
                {
                    const int nwu = min(NW, (plen - pb + 31) >> 5);
                    const int s = lane < nwu ? wsum[lane] : 0, c = lane < nwu ? wcnt[lane] : 0,
                              z = lane < nwu ? wstr[lane] : 0;
                    total = __reduce_add_sync(0xffffffffu, s);
                    ne = __reduce_add_sync(0xffffffffu, c);
                    strips = __reduce_add_sync(0xffffffffu, z);
                    base = __reduce_add_sync(0xffffffffu, lane < w ? s : 0);
                    cb = __reduce_add_sync(0xffffffffu, lane < w ? c : 0);
                    sb = __reduce_add_sync(0xffffffffu, lane < w ? z : 0);
                }
                if (len > 0) {
                    const int pos = cb + __popc(some & below), first = base + incl - flat;
                    pre[pos] = first;
                    str[pos] = sb + sincl - ns;
                    eq[pos] = q0 + (ns << DENSE_STRIP_L) - first;
                    ea[pos] = av;
                }
                for (int x = tid; x < 33; x += T) pre[ne + x] = INT_MAX;   // a step looks 32 parts ahead
                if (tid == 0) str[ne] = strips;
                __syncthreads();
                // The strips are loaded one ahead of the updates: a warp would
                // otherwise wait for its loads, then for its updates, in turn
                // (few rows show it: 2148 of them 0.23 against 0.27 ms).  The
                // flat products are not: what they find their parts with and
                // hold a step ahead costs more than the wait.
                auto add = [&](const int (&cc)[U], const V (&vv)[U], V av1) {
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const unsigned at = (unsigned)cc[u] - (unsigned)w0;
                        if (at < (unsigned)W) atomicAdd(&acc[dense_slot(at)], dense_prod(av1, vv[u]));
                        else flag |= DERR_COUNT;
                    }
                };
                // whole strips, the same number to every warp
                {
                    const int per = (strips + NW - 1) / NW;
                    int x = w * per;
                    const int xend = min(strips, x + per);
                    int e = -1, next = -1;
                    long long qb = 0;
                    V ae = V(0);
                    auto load = [&](int y, int (&cc)[U], V (&vv)[U], V &av1) {
                        if (y >= next) {   // uniform in the warp
                            while (str[e + 1] <= y) e++;
                            next = str[e + 1];
                            qb = eq[e] + pre[e] - ((long long)next << DENSE_STRIP_L) + lane;
                            ae = ea[e];
                        }
                        const int32_t *pc = bcol + (qb + ((long long)y << DENSE_STRIP_L));
                        const V *pv = bval + (qb + ((long long)y << DENSE_STRIP_L));
                        av1 = ae;
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            cc[u] = pc[32 * u];
                            vv[u] = pv[32 * u];
                        }
                    };
                    if (x < xend) {
                        for (int y = 0; y < ne; y += 32) {
                            const unsigned m = __ballot_sync(0xffffffffu, y + lane < ne && str[y + lane] <= x);
                            e += __popc(m);
                            if (m != 0xffffffffu) break;
                        }
                        int c0[U], c1[U];
                        V v0[U], v1[U], a0, a1 = V(0);
                        load(x, c0, v0, a0);
                        for (; x < xend; x += 2) {
                            if (x + 1 < xend) load(x + 1, c1, v1, a1);
                            add(c0, v0, a0);
                            if (x + 2 < xend) load(x + 2, c0, v0, a0);
                            if (x + 1 < xend) add(c1, v1, a1);
                        }
                    }
                }
                // the flat products: the same number of whole steps of 32 to every warp
                {
                    const int nch = (total + 31) >> 5, pw = (nch + NW - 1) / NW;
                    int tc = w * pw * 32;
                    const int tend = min(total, tc + pw * 32);
                    int e0 = -1;
                    if (tc < tend) {
                        for (int x = 0; x < ne; x += 32) {
                            const unsigned m = __ballot_sync(0xffffffffu, x + lane < ne && pre[x + lane] <= tc);
                            e0 += __popc(m);
                            if (m != 0xffffffffu) break;
                        }
                    }
                    for (; tc < tend; tc += 32 * F) {
                        int c[F];
                        V v[F], av1[F];
#pragma unroll
                        for (int u = 0; u < F; u++) {
                            const int tu = tc + 32 * u;
                            c[u] = -1;
                            if (tu >= tend) continue;   // uniform in the warp
                            const int b = pre[e0 + 1 + lane] - tu;
                            const unsigned m = __reduce_or_sync(0xffffffffu, b < 32 ? 1u << b : 0u);
                            const int e = e0 + __popc(m & (2u * below + 1u));
                            e0 += __popc(__ballot_sync(0xffffffffu, b <= 32));
                            if (tu + lane < total) {
                                const long long q = eq[e] + (tu + lane);
                                c[u] = bcol[q];
                                v[u] = bval[q];
                                av1[u] = ea[e];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < F; u++) {
                            if (c[u] < 0) continue;
                            const unsigned at = (unsigned)c[u] - (unsigned)w0;
                            if (at < (unsigned)W) atomicAdd(&acc[dense_slot(at)], dense_prod(av1[u], v[u]));
                            else flag |= DERR_COUNT;
                        }
                    }
                }
                __syncthreads();
                // (an empty slot is -0.0, which an addition leaves as it is)
                if (FOLDS && sums && pb + T < plen && (pb / T + 1) % DENSE_FOLD == 0) {
                    for (int x = tid; x < W; x += T) {
                        sums[x] = folded ? sums[x] + acc[x] : acc[x];
                        acc[x] = dense_empty(V(0));
                    }
                    folded = true;
                    __syncthreads();
                }
            }
            if (FOLDS && folded) {
                for (int x = tid; x < W; x += T) acc[x] = sums[x] + acc[x];
                __syncthreads();
            }
            // entries of each warp's runs, then their places
            int n = 0;
            for (int x = w * runs * 32 + lane * VW; x < (w + 1) * runs * 32; x += 32 * VW) {
                union { uint4 u; V v[VW]; } q;
                q.u = *(const uint4 *)&acc[x];
#pragma unroll
                for (int y = 0; y < VW; y++) n += dense_has(q.v[y]);
            }
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) wsum[w] = n;
            __syncthreads();
            const int s = lane < NW ? wsum[lane] : 0;
            const int tot = __reduce_add_sync(0xffffffffu, s);
            int64_t r = out + written + __reduce_add_sync(0xffffffffu, lane < w ? s : 0);
            const bool fits = written + tot <= expect;
            if (!fits) flag |= DERR_COUNT;   // not the pattern of the symbolic phase
            int32_t *oc = a.ccol + r;
            V *ov = a.cval + r;
#pragma unroll 4
            for (int x = w * runs; x < (w + 1) * runs; x++) {
                const int at = x * 32 + (lane ^ dense_perm(x));
                const V v = acc[at];
                acc[at] = dense_empty(V(0));
                const bool has = dense_has(v);
                const unsigned m = __ballot_sync(0xffffffffu, has);
                if (has && fits) {
                    const int p = __popc(m & below);
                    oc[p] = (int)w0 + x * 32 + lane;
                    ov[p] = v;
                }
                oc += __popc(m);
                ov += __popc(m);
            }
            written += tot;
            __syncthreads();
        }
        if (written != expect) flag |= DERR_COUNT;
    }
    if (flag) atomicOr(err, flag);
}

// Columns of a window: the span of B's columns in as few windows as fit
// `most` columns, equal ones, a multiple of 4096.
static void dense_windows(int64_t ncols, int64_t most, int &W, int &nwin) {
    const int64_t n = std::max<int64_t>(1, (ncols + most - 1) / most);
    W = (int)(((ncols + n - 1) / n + 4095) / 4096 * 4096);
    nwin = (int)std::max<int64_t>(1, (ncols + W - 1) / W);
}
// Columns that fit a window: 88 KB of accumulators (96 once rounded up)
// beside 10-12 KB of staging, two blocks an SM.
template <typename V>
constexpr int64_t dense_most() { return DENSE_BYTES / (int64_t)sizeof(V); }

size_t dense_ws(int64_t nrows_b, int64_t ncols_b) {
    int W, nwin;
    dense_windows(ncols_b, dense_most<double>(), W, nwin);
    return ((size_t)nrows_b * (size_t)(nwin - 1) * 4 + 255) & ~(size_t)255;
}
// The windows' sums of all blocks that fit the chip (no more than its shared
// memory), when a row of A has more than the batches of one fold.
static_assert(DENSE_FOLD_ALEN == 256 * DENSE_FOLD, "the shortest row of A that is folded");
size_t dense_fold_ws(int64_t max_alen, int nsm) { return max_alen > DENSE_FOLD_ALEN ? (size_t)nsm * (228 << 10) : 0; }

template <typename V>
static int num_dense(const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc, const int2 *rspan,
                     const int32_t *rows, int64_t count, int64_t max_alen, void *ws, size_t ws_bytes,
                     unsigned long long *next, int *err, Ctx &c) {
    int W, nwin;
    dense_windows(B.ncols, dense_most<V>(), W, nwin);
    int32_t *split = (int32_t *)ws;
    const int64_t cells = B.nrows * (nwin - 1);
    if ((size_t)cells * 4 > ws_bytes) {
        set_error("numeric: split table workspace too small");
        return SPGEMM_ERR_INTERNAL;
    }
    if (cells > 0) {
        c.begin("numeric.dense_split", B.nrows);
        k_dense_split<<<(unsigned)std::min<int64_t>((cells + 255) / 256, (int64_t)c.nsm * 16), 256, 0, c.s>>>(
            B.nrows, B.row_ptr, B.col_idx, W, nwin, split);
        c.end();
        SG_CUDA(cudaGetLastError());
    }
    DenseP<V> p{A.row_ptr, A.col_idx, (const V *)A.values, B.col_idx, (const V *)B.values, C.row_ptr, C.col_idx,
                (V *)C.values, bdesc, rspan, rows, split, count, W, nwin, next, nullptr};
    const size_t used = ((size_t)cells * 4 + 255) & ~(size_t)255;
    SG_CUDA(cudaMemsetAsync(next, 0, sizeof(*next), c.s));
    auto go = [&](auto kern, int T, size_t smem) -> int {
        int per_sm = 0;
        SG_TRY(kernel_blocks_per_sm((const void *)kern, T, smem, &per_sm));
        const int64_t blocks = std::min<int64_t>(count, (int64_t)per_sm * c.nsm);
        if (sizeof(V) == 4 && max_alen > (int64_t)T * DENSE_FOLD) {
            if (used + (size_t)blocks * W * sizeof(V) > ws_bytes) {
                set_error("numeric: workspace of the folded windows too small");
                return SPGEMM_ERR_INTERNAL;
            }
            p.fold = (V *)((char *)ws + used);
        }
        c.begin("numeric.dense", count);
        kern<<<(unsigned)blocks, T, smem, c.s>>>(p, err);
        c.end();
        SG_CUDA(cudaGetLastError());
        return SPGEMM_OK;
    };
    // Windows of up to 40 KB leave room for four blocks of 256 threads an SM, which wait
    // less at their barriers: 2000 FP32 rows of 6500 products over 4096 columns, rows of B
    // of 100, 56 us (two blocks of 512: 70), 8000 of 40,000 over 8192, rows of B of 200, 615
    // (693).  (100 of those rows alone 40 us, by 512 threads 27.)
    if ((size_t)W * sizeof(V) <= 40 * 1024) return go(k_num_dense<V, 256, 4>, 256, DenseSmem<V, 256>(W).bytes);
    return go(k_num_dense<V, 512, 2>, 512, DenseSmem<V, 512>(W).bytes);
}

int launch_num_dense(int dtype, const spgemm_csr &A, const spgemm_csr &B, spgemm_csr &C, const int4 *bdesc,
                     const int2 *rspan, const int32_t *rows, int64_t count, int64_t max_alen, void *ws,
                     size_t ws_bytes, unsigned long long *next, int *err, Ctx &c) {
    if (count <= 0) return SPGEMM_OK;
    return dtype == SPGEMM_F32 ? num_dense<float>(A, B, C, bdesc, rspan, rows, count, max_alen, ws, ws_bytes, next, err, c)
                               : num_dense<double>(A, B, C, bdesc, rspan, rows, count, max_alen, ws, ws_bytes, next, err, c);
}

}  // namespace sg
