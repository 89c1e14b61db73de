// Gradients of a sparse product with respect to the stored values of its
// operands.  With L a scalar function of C = A*B and dC = dL/dC given on the
// pattern of C, the product is bilinear, so
//     dA_ik = sum over stored b_kj of dC_ij * b_kj        (dC * B^T on pattern(A))
//     dB_kj = sum over stored a_ik of a_ik * dC_ij        (A^T * dC on pattern(B))
// Both come out of one pass over the same products as the forward product:
// for each stored a_ik and each stored b_kj, dC_ij is found in row i of C
// (columns ascending) by binary search; the dA terms of a_ik are summed by
// the lanes walking B_k (a segmented sum across the lanes, one update per
// a_ik and step), and the dB terms are added atomically into the slot of
// b_kj (its position in B is the loop index).  No dense intermediate.
// Rows of C with at most BWD_CAP entries are searched in a copy of their
// columns in shared memory (a warp per row, products dealt out over the
// lanes); longer rows are searched in global memory.
#include <climits>
#include "internal.cuh"

namespace sg {

// Position of column j in the sorted row col[c0, c1), or -1.
__device__ __forceinline__ int64_t find_col(const int32_t *__restrict__ col, int64_t c0, int64_t c1, int j) {
    int64_t lo = c0, hi = c1;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (col[mid] < j) lo = mid + 1;
        else hi = mid;
    }
    return (lo < c1 && col[lo] == j) ? lo : -1;
}

// A warp per row of A whose row of C has at most BWD_CAP entries: the
// columns of C_i are copied to shared memory, the products a_ik * b_kj of
// the row are dealt out over the lanes through prefix sums of nnz(B_k)
// (stored a_ik staged BWD_E at a time; a step's entries from the starts
// within it, as in rank.cu), each lane finds dC_ij by binary search in the
// copy, adds its dA term into the staged entry's accumulator and its dB term
// atomically into db.
// What bounds it: the chain B's column -> search -> dC.  U steps go through it
// together: their loads of B, then their searches (as many halvings for every
// lane), then their loads of dC.  Measured (one GB300, FP32): 20,001 rows of about
// 320 products 101 -> 80 us with four steps together (two 87, six 95).  Where the
// rows have 32 products or fewer in the mean, or 64, most have one step, or two,
// and the others only cost: 200,000 rows of 9 products 153 us with four, 134 with
// one, of 25 164 and 139; of 36 202 with four, 182 with two, of 64 227 and 215.
constexpr int BWD_CAP = 1024, BWD_WPB = 8, BWD_E = 32;
constexpr int BWD_ROW_MAX = 1 << 20;   // entries of a row of B taken (32 of them fit an int; a row of C holds fewer)

template <typename V, int U>
__global__ void __launch_bounds__(BWD_WPB * 32) k_backward_rows(
    int64_t nrows, const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const V *__restrict__ aval, const int64_t *__restrict__ brp, const int32_t *__restrict__ bcol,
    const V *__restrict__ bval, const int64_t *__restrict__ crp, const int32_t *__restrict__ ccol,
    const V *__restrict__ dc, V *__restrict__ da, V *__restrict__ db, int *err) {
    __shared__ int cs_all[BWD_WPB * BWD_CAP];
    __shared__ long long eq0_all[BWD_WPB * BWD_E];
    __shared__ V ea_all[BWD_WPB * BWD_E];
    __shared__ V dacc_all[BWD_WPB * BWD_E];
    __shared__ int pre_all[BWD_WPB * BWD_E];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *cs = cs_all + w * BWD_CAP;
    long long *eq0 = eq0_all + w * BWD_E;
    V *ea = ea_all + w * BWD_E;
    V *dacc = dacc_all + w * BWD_E;
    int *pre = pre_all + w * BWD_E;
    const unsigned below = (1u << lane) - 1u, upto = 2u * below + 1u;
    bool missing = false;
    for (int64_t i = (int64_t)blockIdx.x * BWD_WPB + w; i < nrows; i += (int64_t)gridDim.x * BWD_WPB) {
        const int64_t c0 = crp[i];
        const int64_t nc64 = crp[i + 1] - c0;
        if (nc64 > BWD_CAP) continue;   // searched in global memory by k_backward
        const int nc = (int)nc64;
        const int64_t p0 = arp[i];
        const int plen = (int)(arp[i + 1] - p0);
        if (plen == 0) continue;
        for (int x = lane; x < nc; x += 32) cs[x] = ccol[c0 + x];
        __syncwarp();
        for (int pb = 0; pb < plen; pb += BWD_E) {
            int len = 0;
            int64_t q0 = 0;
            if (pb + lane < plen) {
                const int k = acol[p0 + pb + lane];
                q0 = brp[k];
                len = (int)min(brp[k + 1] - q0, (int64_t)BWD_ROW_MAX);
            }
            dacc[lane] = V(0);
            int incl = len;
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            // the entries with a row of B, in order
            const unsigned some = __ballot_sync(0xffffffffu, len > 0);
            const int pos = __popc(some & below), ne = __popc(some);
            if (len > 0) {
                pre[pos] = incl - len;
                eq0[pos] = q0 - (incl - len);
                ea[pos] = aval ? aval[p0 + pb + lane] : V(0);
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
            const int at = lane < ne ? pre[lane] : INT_MAX;   // first product of entry `lane`
            for (int t0 = 0; t0 < total; t0 += 32 * U) {
                long long q[U];
                int e[U], j[U], lo[U];
                unsigned m[U];
                V bv[U], g[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int tc = t0 + 32 * u;
                    e[u] = -1;
                    j[u] = lo[u] = 0;
                    bv[u] = V(0);
                    if (tc >= total) continue;   // uniform in the warp
                    const int b = at - tc;
                    m[u] = __reduce_or_sync(0xffffffffu, (unsigned)b < 32u ? 1u << b : 0u);
                    const int ee = __popc(__ballot_sync(0xffffffffu, b < 0)) + __popc(m[u] & upto) - 1;
                    if (tc + lane < total) {
                        e[u] = ee;
                        q[u] = eq0[ee] + (tc + lane);
                        j[u] = bcol[q[u]];
                        if (bval) bv[u] = bval[q[u]];
                    }
                }
                for (int n = nc; n > 1;) {
                    const int half = n >> 1;
#pragma unroll
                    for (int u = 0; u < U; u++) lo[u] += cs[lo[u] + half - 1] < j[u] ? half : 0;
                    n -= half;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    g[u] = V(0);
                    if (e[u] < 0) continue;
                    if (lo[u] < nc && cs[lo[u]] < j[u]) lo[u]++;
                    if (lo[u] < nc && cs[lo[u]] == j[u]) {
                        g[u] = dc[c0 + lo[u]];
                    } else {
                        missing = true;
                        e[u] = -1 - e[u] - 1;   // (no term, but still of its entry)
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int tc = t0 + 32 * u;
                    if (tc >= total) break;
                    if (db && e[u] >= 0) atomicAdd(&db[q[u]], ea[e[u]] * g[u]);
                    if (bval) {
                        // the lanes of one staged a_ik are consecutive: a segmented
                        // sum over them leaves its dA term in the segment's first
                        // lane, which alone updates the entry's accumulator
                        V term = e[u] >= 0 ? g[u] * bv[u] : V(0);
                        const unsigned after = m[u] & ~upto;
                        const int last = after ? __ffs(after) - 2 : min(31, total - 1 - tc);
                        for (int d = 1; d < 32; d <<= 1) {
                            const V y = __shfl_down_sync(0xffffffffu, term, d);
                            if (lane + d <= last) term += y;
                        }
                        const int ee = e[u] >= 0 ? e[u] : -2 - e[u];
                        if (tc + lane < total && (lane == 0 || (m[u] >> lane & 1u))) dacc[ee] += term;
                        __syncwarp();
                    }
                }
            }
            __syncwarp();
            if (da && pb + lane < plen) da[p0 + pb + lane] = len > 0 ? dacc[pos] : V(0);
            __syncwarp();
        }
    }
    if (missing) atomicOr(err, DERR_COUNT);
}

// G lanes per row of A whose row of C has more than skip_cap entries: for
// each stored a_ik in turn the lanes walk B_k, each looks up dC_ij in global
// memory, and the group reduces the dA term.
template <typename V, int G>
__global__ void __launch_bounds__(256, 4) k_backward(
    int64_t nrows, const int64_t *__restrict__ arp, const int32_t *__restrict__ acol,
    const V *__restrict__ aval, const int64_t *__restrict__ brp, const int32_t *__restrict__ bcol,
    const V *__restrict__ bval, const int64_t *__restrict__ crp, const int32_t *__restrict__ ccol,
    const V *__restrict__ dc, V *__restrict__ da, V *__restrict__ db, int *err, int64_t skip_cap) {
    const int gl = threadIdx.x % G;
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1) << ((threadIdx.x & 31) & ~(G - 1)));
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
    bool missing = false;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; i < nrows; i += groups) {
        const int64_t c0 = crp[i], c1 = crp[i + 1];
        if (c1 - c0 <= skip_cap) continue;
        for (int64_t p = arp[i]; p < arp[i + 1]; p++) {
            const int k = acol[p];
            const V a = aval ? aval[p] : V(0);
            V acc = V(0);
            for (int64_t q = brp[k] + gl; q < brp[k + 1]; q += G) {
                const int64_t pos = find_col(ccol, c0, c1, bcol[q]);
                if (pos < 0) {
                    missing = true;
                    continue;
                }
                const V g = dc[pos];
                if (bval) acc += g * bval[q];
                if (db) atomicAdd(&db[q], a * g);
            }
            for (int d = G / 2; d > 0; d >>= 1) acc += __shfl_xor_sync(gmask, acc, d, G);
            if (da && gl == 0) da[p] = acc;
        }
    }
    if (missing) atomicOr(err, DERR_COUNT);
}

template <typename V>
static int run_bwd(const spgemm_csr &A, const spgemm_csr &B, const spgemm_csr &C, void *da, void *db,
                   int *err, int G, Ctx &c) {
    if (db) SG_CUDA(cudaMemsetAsync(db, 0, (size_t)B.nnz * sizeof(V), c.s));
    if (A.nrows == 0) return SPGEMM_OK;
    int64_t rblocks = (A.nrows + BWD_WPB - 1) / BWD_WPB;
    rblocks = rblocks < (int64_t)c.nsm * 16 ? rblocks : (int64_t)c.nsm * 16;
    auto rows = [&](auto kern) {
        c.begin("backward", A.nrows);
        kern<<<(unsigned)rblocks, BWD_WPB * 32, 0, c.s>>>(
            A.nrows, A.row_ptr, A.col_idx, (const V *)A.values, B.row_ptr, B.col_idx,
            da ? (const V *)B.values : nullptr, C.row_ptr, C.col_idx, (const V *)C.values, (V *)da, (V *)db, err);
        c.end();
    };
    const double products = (double)A.nnz * (double)B.nnz / ((double)A.nrows * (double)std::max<int64_t>(B.nrows, 1));
    if (products <= 32.0) rows(k_backward_rows<V, 1>);
    else if (products <= 64.0) rows(k_backward_rows<V, 2>);
    else rows(k_backward_rows<V, 4>);
    SG_CUDA(cudaGetLastError());
    int64_t blocks = (A.nrows * G + 255) / 256;
    blocks = blocks < (int64_t)c.nsm * 32 ? blocks : (int64_t)c.nsm * 32;
    c.begin("backward_long", A.nrows);
#define SG_BWD(GG)                                                                                   \
    k_backward<V, GG><<<(unsigned)blocks, 256, 0, c.s>>>(                                            \
        A.nrows, A.row_ptr, A.col_idx, (const V *)A.values, B.row_ptr, B.col_idx,                   \
        da ? (const V *)B.values : nullptr, C.row_ptr, C.col_idx, (const V *)C.values, (V *)da,      \
        (V *)db, err, (int64_t)BWD_CAP)
    switch (G) {
        case 4: SG_BWD(4); break;
        case 8: SG_BWD(8); break;
        case 16: SG_BWD(16); break;
        default: SG_BWD(32);
    }
#undef SG_BWD
    c.end();
    SG_CUDA(cudaGetLastError());
    return SPGEMM_OK;
}

int launch_backward(int dtype, const spgemm_csr &A, const spgemm_csr &B, const spgemm_csr &C, void *da,
                    void *db, int *err, Ctx &c) {
    const double mean_b = B.nrows ? (double)B.nnz / (double)B.nrows : 1.0;
    int G = 4;
    while (G < 32 && 2 * G <= mean_b) G *= 2;
    return dtype == SPGEMM_F64 ? run_bwd<double>(A, B, C, da, db, err, G, c)
                               : run_bwd<float>(A, B, C, da, db, err, G, c);
}

}  // namespace sg
