// Stage 4 (Section 4.1, "arranging data"): the sizes nnz(c_i) are summed by an
// exclusive prefix sum into C.row_ptr (int64), C is allocated by the host, and
// the rows are copied from the temporary matrix C~ into C.  Rows of bin 1 hold a
// single product, which is computed here directly; rows of bin 0 need nothing.
// Bins 2..36 are copied by one warp per row, bin 37 by one CTA per row (all
// column slices of a split row, in column order).
#include "internal.h"
#include "scan.cuh"

namespace spg {

struct LoadNnzc {
    const int32_t *nnzc;
    SPG_DEV int64_t operator()(int64_t i) const { return (int64_t)nnzc[i]; }
};
struct StoreRp {
    int64_t *rp;
    SPG_DEV void operator()(int64_t i, int64_t v) const { rp[i] = v; }
};

int row_scan_launches(int64_t m) { return scan_launches(m, true); }
int64_t row_scan_partials(int64_t m) { return scan_blocks(m) + 1; }

cudaError_t launch_row_scan(int64_t m, const int32_t *nnzc, int64_t *c_rp, int64_t *partial,
                            cudaStream_t st, int64_t *host, const int64_t *err) {
    return device_exclusive_scan(m, LoadNnzc{nnzc}, StoreRp{c_rp}, partial, c_rp + m, st, host, err);
}

constexpr int ARR_NT = 256;

// G lanes per row (about the entries of an average row, so that short rows fill their warps);
// the groups stride over the rows (one pass when the grid covers them).  A streaming copy: 12
// bytes read and written per entry.  A*P of the 27-point operator on 64^3 (262,144 rows of 7.6
// entries) took 70 us with a warp per row.
template <int G>
__global__ void __launch_bounds__(ARR_NT)
k_arrange_short(StageArgs a, RowSet R, const uint8_t *__restrict__ bin,
                const int64_t *__restrict__ c_rp, int32_t *__restrict__ c_col, val_t *__restrict__ c_val) {
    if (gated(a.gate)) return;
    const int32_t *rows;
    int64_t nrows;
    rowset_range(R, rows, nrows);
    constexpr int UN = 4;
    const int gl = threadIdx.x & (G - 1), sh = lane_id() & ~(G - 1);
    const unsigned gm = G == 32 ? SPG_FULL : ((1u << (G & 31)) - 1u) << sh;
    for (int64_t wg = ((int64_t)blockIdx.x * ARR_NT + threadIdx.x) / G; wg < nrows;
         wg += (int64_t)gridDim.x * (ARR_NT / G)) {
        const int row = rows[wg];
        const int64_t o = c_rp[row];
        if (bin[row] == 1) {
            // exactly one A entry of this row selects a B row of length 1
            const int64_t a0 = a.A.rp[row], a1 = a.A.rp[row + 1];
            for (int64_t base = a0; base < a1; base += G) {
                const int64_t p = base + gl;
                int64_t b0 = 0;
                bool hit = false;
                if (p < a1) {
                    const int32_t j = a.A.col[p];
                    b0 = a.B.rp[j];
                    hit = (a.B.rp[j + 1] - b0) > 0;
                }
                const unsigned m = __ballot_sync(gm, hit) & gm;
                if (m) {
                    if (lane_id() == __ffs(m) - 1 && SPG_IN(o < c_rp[row + 1], 103)) {
                        c_col[o] = a.B.col[b0];
                        c_val[o] = a.A.val[p] * a.B.val[b0];
                    }
                    break;
                }
            }
            continue;
        }
        const int64_t n = c_rp[row + 1] - o;
        const int64_t src = a.ctil_rp[row];
        if (!SPG_IN(src + n <= a.ctil_rp[row + 1], 104)) continue;  // C~ holds the row
        for (int64_t t = gl; t < n; t += UN * G) {
            int32_t c[UN];
            val_t v[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u)
                if (t + u * G < n) c[u] = __ldcs(a.ctil_col + src + t + u * G);
#pragma unroll
            for (int u = 0; u < UN; ++u)
                if (t + u * G < n) v[u] = __ldcs(a.ctil_val + src + t + u * G);
#pragma unroll
            for (int u = 0; u < UN; ++u)
                if (t + u * G < n) {
                    c_col[o + t + u * G] = c[u];
                    c_val[o + t + u * G] = v[u];
                }
        }
    }
}

cudaError_t launch_arrange_short(const StageArgs &a, const RowSet &R, const uint8_t *bin, const int64_t *c_rp,
                                 int32_t *c_col, val_t *c_val, int64_t avg_nnz, cudaStream_t st) {
    if (R.n <= 0) return cudaSuccess;
    auto go = [&](auto kern, int g) {
        const int64_t need = (R.n * g + ARR_NT - 1) / ARR_NT;
        const int64_t grid = R.dev_lo ? persistent_blocks((const void *)kern, ARR_NT, 0, need) : need;
        if (grid <= 0) return cudaErrorInvalidValue;
        kern<<<(unsigned)grid, ARR_NT, 0, st>>>(a, R, bin, c_rp, c_col, c_val);
        return cudaGetLastError();
    };
    if (avg_nnz <= 6) return go(k_arrange_short<4>, 4);
    if (avg_nnz <= 12) return go(k_arrange_short<8>, 8);
    if (avg_nnz <= 40) return go(k_arrange_short<16>, 16);
    return go(k_arrange_short<32>, 32);
}

// The rows of bin 1 alone (a replay, the precise method): the one entry of A that selects a row of B that is not
// empty is searched by G lanes, one entry each at first, several in a row that turns out long.  Bound by
// the gathers of B's row pointers, so few registers and many warps.  A launch on rows of bin 1 among 200,000 rows
// of A of 256 and of 3 entries, 100 rows of 200,000: by four lanes with the copy's registers 100 us, 64 us and 13.1 ms,
// here 69 us, 51 us and 0.83 ms (a warp per row: 69 us, 264 us and 1.5 ms).
template <int G>
__global__ void __launch_bounds__(ARR_NT, 8)
k_single(StageArgs a, RowSet R, const int64_t *__restrict__ c_rp, int32_t *__restrict__ c_col,
         val_t *__restrict__ c_val) {
    if (gated(a.gate)) return;
    const int32_t *rows;
    int64_t nrows;
    rowset_range(R, rows, nrows);
    constexpr int UN = 4;
    const int gl = threadIdx.x & (G - 1);
    const unsigned gm = G == 32 ? SPG_FULL : ((1u << (G & 31)) - 1u) << (lane_id() & ~(G - 1));
    for (int64_t wg = ((int64_t)blockIdx.x * ARR_NT + threadIdx.x) / G; wg < nrows;
         wg += (int64_t)gridDim.x * (ARR_NT / G)) {
        const int row = rows[wg];
        const int64_t a0 = a.A.rp[row], a1 = a.A.rp[row + 1];
        auto hit = [&](int32_t j) { return a.B.rp[j + 1] > a.B.rp[j]; };
        int64_t p = -1;
        for (int64_t base = a0 + gl; base - gl < a1;) {
            if (base - a0 < 16 * G) {
                if (base < a1 && hit(a.A.col[base])) p = base;
                base += G;
            } else {
                int32_t j[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (base + u * G < a1) j[u] = a.A.col[base + u * G];
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (base + u * G < a1 && hit(j[u])) p = base + u * G;
                base += UN * G;
            }
            if (__any_sync(gm, p >= 0)) break;
        }
        if (p >= 0) {
            const int64_t o = c_rp[row], b0 = a.B.rp[a.A.col[p]];
            if (SPG_IN(o < c_rp[row + 1], 116)) {
                c_col[o] = a.B.col[b0];
                c_val[o] = a.A.val[p] * a.B.val[b0];
            }
        }
    }
}

cudaError_t launch_single(const StageArgs &a, const RowSet &R, const int64_t *c_rp, int32_t *c_col, val_t *c_val,
                          cudaStream_t st) {
    if (R.n <= 0) return cudaSuccess;
    auto go = [&](auto kern, int g) {
        const int64_t need = (R.n * g + ARR_NT - 1) / ARR_NT;
        const int64_t grid = R.dev_lo ? persistent_blocks((const void *)kern, ARR_NT, 0, need) : need;
        if (grid <= 0) return cudaErrorInvalidValue;
        kern<<<(unsigned)grid, ARR_NT, 0, st>>>(a, R, c_rp, c_col, c_val);
        return cudaGetLastError();
    };
    const int64_t half = a.A.nnz / (2 * (a.A.nrows > 0 ? a.A.nrows : 1));  // of an average row of A
    if (half <= 4) return go(k_single<4>, 4);
    if (half <= 12) return go(k_single<8>, 8);
    if (half <= 24) return go(k_single<16>, 16);
    return go(k_single<32>, 32);
}

// One thread: whether C (c_rp[m] entries) fits the cap entries allocated for it.
__global__ void k_gate(const int64_t *c_rp, int64_t m, int64_t cap, int64_t *gate, int64_t *err) {
    const bool over = c_rp[m] > cap;
    *gate = over ? 1 : 0;
    if (over) atomicExch((unsigned long long *)err, 8ull);
}

// A C that does not fit becomes the empty matrix (all row pointers 0), so that nothing
// downstream -- a chained product reading it as its B -- reads beyond its arrays.
__global__ void k_gate_clear(int64_t *c_rp, int64_t m, const int64_t *gate) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= m && *gate != 0) c_rp[i] = 0;
}

cudaError_t launch_gate(int64_t *c_rp, int64_t m, int64_t cap, int64_t *gate, int64_t *err, cudaStream_t st) {
    k_gate<<<1, 1, 0, st>>>(c_rp, m, cap, gate, err);
    k_gate_clear<<<(unsigned)((m + 1 + 255) / 256), 256, 0, st>>>(c_rp, m, gate);
    return cudaGetLastError();
}

// One CTA per bin-37 row: its leaves (column slices) are visited in column order
// (a walk of the split tree, left child first) and copied back to back.
// Rows of the dense-slice kernels are already in C.
__global__ void __launch_bounds__(ARR_NT)
k_arrange_long(MergeItems it, const int64_t *__restrict__ c_rp, int32_t *__restrict__ c_col,
               val_t *__restrict__ c_val) {
    constexpr int LEAF_BUF = 128;
    __shared__ int leaves[LEAF_BUF];
    __shared__ int nleaves, cursor;
    const int j = blockIdx.x;
    if (it.child[j] == ITEM_DENSE) return;  // written into C by the dense-slice kernel
    int64_t o = c_rp[it.row[j]];
    if (threadIdx.x == 0) cursor = split_first_leaf(it, j);
    __syncthreads();
    while (true) {
        if (threadIdx.x == 0) {
            int n = 0, x = cursor;
            while (x >= 0 && n < LEAF_BUF) {
                leaves[n++] = x;
                x = split_next_leaf(it, j, x);
            }
            cursor = x;
            nleaves = n;
        }
        __syncthreads();
        const int nl = nleaves;
        if (nl == 0) break;
        for (int l = 0; l < nl; ++l) {
            const int x = leaves[l];
            const int64_t n = it.len[x];
            const int32_t *sc = it.home_col[x];
            const val_t *sv = it.home_val[x];
            if (!SPG_IN(o + n <= c_rp[it.row[j] + 1], 105)) break;  // the leaves fill the row of C exactly
            constexpr int UN = 4;  // loads in flight per thread
            for (int64_t t = threadIdx.x; t < n; t += UN * ARR_NT) {
                int32_t c[UN];
                val_t v[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (t + u * ARR_NT < n) c[u] = __ldcs(sc + t + u * ARR_NT);
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (t + u * ARR_NT < n) v[u] = __ldcs(sv + t + u * ARR_NT);
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (t + u * ARR_NT < n) {
                        c_col[o + t + u * ARR_NT] = c[u];
                        c_val[o + t + u * ARR_NT] = v[u];
                    }
            }
            o += n;
        }
        __syncthreads();
    }
}

cudaError_t launch_arrange_long(const MergeItems &it, int64_t n37, const int64_t *c_rp, int32_t *c_col,
                                val_t *c_val, cudaStream_t st) {
    if (n37 <= 0) return cudaSuccess;
    k_arrange_long<<<(unsigned)n37, ARR_NT, 0, st>>>(it, c_rp, c_col, c_val);
    return cudaGetLastError();
}

}  // namespace spg
