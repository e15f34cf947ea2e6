// Stage 3, bin group 5, for the rows whose products cover a large part of B's
// column range (and, in the precise method, for every bin-37 row): an accumulator
// over column slices instead of the merge of Section 4.1.
//
// B's columns are cut into K slices of W columns (W a multiple of 32, at most
// DENSE_W_MAX, K W >= ncols).  A slice of a row is one CTA's item.  The counting pass marks
// the columns of the row's products in the slice in a shared bitmap and counts its
// bits, and may leave the bitmap in device memory.  The fill pass reads it back (or marks
// the columns again when it was not kept), ranks the bitmap (set bits before each word),
// and adds every product into the sum at its column's rank: clearing and writing out cost
// the slice's entries, not its width, and the sums come out in column order.  There are no
// misses, no merges and no capacity to outgrow.  The part of each B row that falls in slice
// s is read from a table of per-row slice boundaries, built once per call.
//
// Because the rows are counted first, they need no temporary result rows: their sizes
// go into the row counts of C with the other rows', and the values are written
// straight into C once its row pointers exist (the kept bitmaps, W / 8 bytes per
// (row, slice), are the only temporary, and an optional one).  The same launch recomputes the values
// for a values-only replay.
//
// Measured (count + fill launches of C = A*A, double, one GB300, before -> after the product
// walk below replaced a search per product, the sums moved from shared memory into C, and the fill
// was split by size): R-MAT 2^18 x 8, every bin-37 row, bitmaps not kept: 24.4 -> 10.5 ms; R-MAT 2^20 x
// 8, kept: 129.8 -> 66.0 ms.
#include "internal.h"
#include "common.cuh"
#include "dynamic_smem.h"

#include <algorithm>
#include <type_traits>

namespace spg {

// ---- per-B-row slice boundaries ----

__global__ void k_dense_bounds(DevCSR B, int K, int W, int32_t *bnd) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B.nrows * (K + 1)) return;
    const int64_t k = i / (K + 1);
    const int s = (int)(i - k * (K + 1));
    const int64_t rs = B.rp[k];
    const int n = (int)(B.rp[k + 1] - rs);
    int v;
    if (s == 0) v = 0;
    else if (s == K) v = n;
    else v = lower_bound_i32(B.col + rs, n, (int32_t)((int64_t)s * W));
    bnd[i] = v;
}

cudaError_t launch_dense_bounds(const DevCSR &B, int K, int W, int32_t *bnd, cudaStream_t st) {
    const int64_t n = B.nrows * (K + 1);
    if (n <= 0 || K <= 1) return cudaSuccess;
    k_dense_bounds<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(B, K, W, bnd);
    return cudaGetLastError();
}

// ---- selection of the dense rows among the bin-37 rows ----
// A dense row's bucket is 64 kind + the leading zeros of u, so that larger rows come first.  Kind 0
// takes a CTA per slice: the rows of more than DENSE_MID_W columns, and narrower ones whose parts
// (products per entry of A) a warp would take one by one with most lanes idle, or whose parts are
// long but scattered.  Kinds 1 and 2, more and at most DENSE_NARROW_W columns, take a warp per row, but
// for the rows that would outlast the others (k_dense_select_starts).  DENSE_BUCKETS for the rows
// that are not dense.  order[0..nd) lists the dense items, order[nd..n37) the rest.
//
// Product of 30,000 rows by a warp each / by CTAs, ms.  Double, consecutive parts in ranges of 200
// columns: parts of 2, u = 600 1.44 / 0.92, u = 32,000 66.6 / 16.2; of 8, u = 600 0.55 / 0.75, u = 2,000
// 1.30 / 0.93; of 16, u = 4,500 1.60 / 1.48 (single precision 1.26 / 1.51), u = 8,000 2.68 / 2.00; of 32
// and 80, u = 32,000 5.2 / 6.6 and 4.4 / 6.2.  Single precision, scattered parts of 80, u = 2,000, 8,000 and
// 32,000: of 200 columns 0.84 / 0.97, 2.65 / 1.92 and 9.5 / 5.8, of 1,000 0.69 / 0.97, 1.83 / 1.84 and 5.84 / 5.22.

constexpr int DENSE_BUCKETS = 3 * 64;
constexpr int64_t DENSE_SCATTERED = 32;  // products per column from which scattered parts take a CTA
SPG_DEV int dense_bucket(const DevCSR &A, const DevCSR &B, int row, int64_t u, int32_t width) {
    const int c = __clzll((long long)u);
    if (width > DENSE_MID_W) return c;
    const int64_t a0 = A.rp[row], nA = A.rp[row + 1] - a0;
    if (u < 4 * nA || (u >= 1536 && u < 12 * nA) || (u >= 6144 && u < 18 * nA)) return c;
    if (u >= 4096 && u >= DENSE_SCATTERED * width) {  // the part in the middle stands for all
        const int32_t k = A.col[a0 + nA / 2];
        const int64_t b0 = B.rp[k], b1 = B.rp[k + 1];
        if (b1 > b0 && B.col[b1 - 1] - B.col[b0] != b1 - b0 - 1) return c;
    }
    return (width > DENSE_NARROW_W ? 64 : 128) + c;
}

__global__ void k_dense_select_count(DevCSR A, DevCSR B, const int32_t *bin_rows, int64_t m, BinSummary *summary,
                                     const int64_t *u, const uint8_t *flag, const int32_t *lo, const int32_t *hi,
                                     int32_t *cls_of, int32_t *count) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n37 = summary->bin_count[BIN_MERGE];
    if (j >= n37) return;
    const int32_t row = bin_rows[m - n37 + j];
    const int64_t uu = u[row];
    const int g = flag[row] ? dense_bucket(A, B, row, uu, hi[row] - lo[row]) : DENSE_BUCKETS;
    cls_of[j] = g;
    // one add per bucket and warp: most rows fall into few buckets
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, g);
    if (lane_id() == __ffs(peers) - 1) atomicAdd(&count[g], __popc(peers));
    // A's entries in the rows of kind 0 (fewer than 2^31 in a row: summed in halves of 16 bits)
    const uint32_t nA = g < 64 ? (uint32_t)(A.rp[row + 1] - A.rp[row]) : 0u;
    const uint32_t low = __reduce_add_sync(act, nA & 0xffffu), high = __reduce_add_sync(act, nA >> 16);
    if (lane_id() == __ffs(act) - 1 && (low | high) != 0u)
        atomicAdd((unsigned long long *)&summary->dense_entries, ((unsigned long long)high << 16) + low);
}

// The buckets' places, a thread per size.  A warp per row is as fast as the chip is full of them,
// about DENSE_FEW_ROWS of equal length.  A row of 2^DENSE_FEW_LOG products or more that is longer than
// a DENSE_FEW_ROWS-th of all such rows' products takes a CTA per slice.  Product of R rows of u products
// in parts of 80 consecutive columns out of 200 by a warp each / by CTAs, ms, double: R = 150, u = 2,000 0.15 /
// 0.19, u = 8,000 0.21 / 0.21, u = 128,000 2.03 / 0.57; R = 1,000 0.15 / 0.19, 0.25 / 0.24 and 2.03 / 1.27; R = 3,000
// 0.17 / 0.26, 0.28 / 0.39 and 2.06 / 2.69.  A^T A of 10^6 x 64 with 8 entries a row: 97 / 6.3.
constexpr int DENSE_FEW_ROWS = 2048, DENSE_FEW_LOG = 13;

__global__ void __launch_bounds__(64)
k_dense_select_starts(const int32_t *count, int32_t *start, int32_t *cursor, BinSummary *summary) {
    __shared__ int64_t scratch[3];
    __shared__ double narrow[2];
    const int z = threadIdx.x;
    int32_t n[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        n[k] = count[64 * k + z];
        cursor[64 * k + z] = 0;
    }
    const double size = ldexp(1.0, 63 - z);
    const double t = warp_reduce_sum(size * (n[1] + n[2]));
    if (lane_id() == 0) narrow[warp_id()] = t;
    __syncthreads();
    const bool cta = 63 - z >= DENSE_FEW_LOG && DENSE_FEW_ROWS * size > narrow[0] + narrow[1];
    // kind 0 (with the moved rows), then kind 1, then kind 2
    const int64_t w = (int64_t)n[0] + (cta ? n[1] + n[2] : 0);
    const int64_t rest = cta ? 0 : ((int64_t)n[1] << 32) | n[2];
    int64_t nw, nr;
    const int32_t pw = (int32_t)block_exclusive_scan<64>(w, scratch, nw);
    const int64_t pr = block_exclusive_scan<64>(rest, scratch, nr);
    const int32_t e0 = (int32_t)nw, e1 = e0 + (int32_t)(nr >> 32), e2 = e1 + (int32_t)(nr & 0xffffffff);
    start[z] = pw;
    start[64 + z] = cta ? pw + n[0] : e0 + (int32_t)(pr >> 32);
    start[128 + z] = cta ? pw + n[0] + n[1] : e1 + (int32_t)(pr & 0xffffffff);
    if (z == 0) {
        start[DENSE_BUCKETS] = e2;
        cursor[DENSE_BUCKETS] = 0;
        summary->dense_count = e2;
        summary->dense_end[0] = e0;
        summary->dense_end[1] = e1;
    }
}

__global__ void k_dense_select_scatter(const int32_t *bin_rows, int64_t m, const BinSummary *summary,
                                       const int32_t *cls_of, const int32_t *start, int32_t *cursor,
                                       const int32_t *lo, const int32_t *hi, int32_t *order, int32_t *rows,
                                       int32_t *rlo, int32_t *rhi) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n37 = summary->bin_count[BIN_MERGE];
    if (j >= n37) return;
    const int g = cls_of[j];
    const unsigned peers = __match_any_sync(__activemask(), g);
    const int leader = __ffs(peers) - 1;
    int32_t pos = lane_id() == leader ? start[g] + atomicAdd(&cursor[g], __popc(peers)) : 0;
    pos = __shfl_sync(peers, pos, leader) + __popc(peers & ((1u << lane_id()) - 1u));
    order[pos] = (int32_t)j;
    if (g < DENSE_BUCKETS) {
        const int32_t row = bin_rows[m - n37 + j];
        rows[pos] = row;
        rlo[pos] = lo[row];
        rhi[pos] = hi[row];
    }
}

int64_t dense_select_scratch(int64_t m) { return 3 * (DENSE_BUCKETS + 1) + m; }

cudaError_t launch_dense_select(const DevCSR &A, const DevCSR &B, const int32_t *bin_rows, BinSummary *summary,
                                const int64_t *u, const uint8_t *flag, const int32_t *lo, const int32_t *hi,
                                int32_t *scratch, int32_t *order, int32_t *rows, int32_t *rlo, int32_t *rhi, cudaStream_t st) {
    const int64_t m = A.nrows;
    if (m <= 0) return cudaSuccess;
    int32_t *count = scratch, *start = count + DENSE_BUCKETS + 1, *cursor = start + DENSE_BUCKETS + 1,
            *cls_of = cursor + DENSE_BUCKETS + 1;
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int32_t) * (DENSE_BUCKETS + 1), st);
    if (e != cudaSuccess) return e;
    const unsigned g = (unsigned)((m + 255) / 256);
    k_dense_select_count<<<g, 256, 0, st>>>(A, B, bin_rows, m, summary, u, flag, lo, hi, cls_of, count);
    k_dense_select_starts<<<1, 64, 0, st>>>(count, start, cursor, summary);
    k_dense_select_scatter<<<g, 256, 0, st>>>(bin_rows, m, summary, cls_of, start, cursor, lo, hi, order, rows, rlo,
                                              rhi);
    return cudaGetLastError();
}

// ---- the products of a (row, slice) ----
// The A entries of the row are taken NT at a time.  The entries of one window that select a
// non-empty part of a B row (its entries inside slice s) are compacted into a table: each
// part's first product in the window's sequence of products, and its place in B.  Every warp
// then takes one contiguous range of that sequence, 32 products at a time, without a barrier:
// the lanes look at the next 32 part starts, the starts that fall into the 32 products become
// a bit mask (one warp-wide OR), and a lane's part is the number of mask bits at or below it.
// So parts of any length -- most are a few entries long, a hub's has thousands -- keep all
// lanes busy, and a product costs no search.  (A binary search per product, and whole-CTA
// passes with a barrier per part for the long parts, held the 2^16-row R-MAT to a quarter of
// the rate of the shared-memory atomics.)
constexpr int DENSE_UN = 4;  // groups of 32 products in flight per warp
constexpr int DENSE_STAGE = 256;  // columns of 32 words (of 1,024) that a warp stages before it writes them to C

template <int NT>
struct DenseWin {
    int64_t base[NT];        // place in B of the part's first entry, minus start
    int64_t scan[NT / 32 + 1];
    val_t av[NT];            // a_ik
    int32_t start[NT + 32];  // first product of the part; INT_MAX past the last part
};

// Builds the table of the entries [e, min(e + NT, a1)); returns the number of products (a
// part has at most DENSE_W_MAX entries, so the window's products fit 32 bits).  Its first
// barrier ends the use of the previous window; the table is ready when it returns.
template <int NT, bool VALS, bool TAB>
SPG_DEV int dense_window(const DevCSR &A, const DevCSR &B, const DenseArgs &D, int s, int64_t e, int64_t a1,
                         DenseWin<NT> &w) {
    static_assert((int64_t)NT * DENSE_W_MAX < INT32_MAX, "products of a window");
    int64_t bs = 0;
    int len = 0;
    val_t av = val_t(0);
    const int64_t i = e + threadIdx.x;
    if (i < a1) {
        const int32_t k = A.col[i];
        if (VALS) av = A.val[i];
        const int64_t rs = B.rp[k];
        if (TAB && D.K > 1) {
            const int32_t *bk = D.bnd + (int64_t)k * (D.K + 1) + s;
            const int32_t b0 = bk[0];
            bs = rs + b0;
            len = bk[1] - b0;
        } else if (!TAB) {  // the part is searched for
            const int n = (int)(B.rp[k + 1] - rs);
            const int b0 = s > 0 ? lower_bound_i32(B.col + rs, n, (int32_t)((int64_t)s * D.W)) : 0;
            bs = rs + b0;
            len = s + 1 < D.K ? lower_bound_i32(B.col + bs, n - b0, (int32_t)((int64_t)(s + 1) * D.W)) : n - b0;
        } else {
            bs = rs;
            len = (int)(B.rp[k + 1] - rs);
        }
    }
    int64_t tot;
    const int64_t ex = block_exclusive_scan<NT, int64_t, false>(len > 0 ? (int64_t(1) << 32) | len : 0, w.scan, tot);
    const int np = (int)(tot >> 32);
    if (len > 0) {
        const int q = (int)(ex >> 32), st = (int)(ex & 0xffffffff);
        w.start[q] = st;
        w.base[q] = bs - st;
        if (VALS) w.av[q] = av;
    }
    if ((int)threadIdx.x >= np) w.start[threadIdx.x] = INT_MAX;
    if (threadIdx.x < 32) w.start[NT + threadIdx.x] = INT_MAX;
    __syncthreads();
    return (int)(tot & 0xffffffff);
}

// f(p, a, ok, full): DENSE_UN entry positions p[] of B, the a_ik that multiply them (VALS) and
// which are valid, called by whole warps.  Each access of a warp reads consecutive entries of few
// B rows.  Where the DENSE_UN groups lie inside one part (full = true_type: consecutive entries,
// all valid, one a_ik), nothing is looked up at all: 4 instructions a group instead of 16.
template <int NT, bool VALS, typename F>
SPG_DEV void dense_walk(const DenseWin<NT> &w, int T, F f) {
    constexpr int NW = NT / 32, ST = NT / 32;
    const int lane = lane_id(), wid = warp_id();
    const int64_t G = (T + 31) >> 5;
    const int g0 = (int)(G * wid / NW), g1 = (int)(G * (wid + 1) / NW);
    if (g0 >= g1) return;
    const int end = min(T, g1 << 5);
    // the part of product 32 g0: among every ST-th start, then among the ST after it
    const int c = __popc(__ballot_sync(SPG_FULL, w.start[lane * ST] <= (g0 << 5))) - 1;
    int t = c * ST - 1 + __popc(__ballot_sync(SPG_FULL, lane < ST && w.start[c * ST + (lane < ST ? lane : 0)] <= (g0 << 5)));
    const unsigned le = (2u << lane) - 1u;  // the lanes up to this one
    for (int q0 = g0 << 5; q0 < end; q0 += 32 * DENSE_UN) {
        int64_t p[DENSE_UN];
        val_t a[DENSE_UN];
        bool ok[DENSE_UN];
        if (min(w.start[t + 1], end) - q0 >= 32 * DENSE_UN) {
#pragma unroll
            for (int u = 0; u < DENSE_UN; ++u) {
                p[u] = w.base[t] + (q0 + lane) + 32 * u;
                if (VALS) a[u] = w.av[t];
                ok[u] = true;
            }
            f(p, a, ok, std::true_type());
            // the next products may begin a part
            if (w.start[t + 1] == q0 + 32 * DENSE_UN) ++t;
            continue;
        }
#pragma unroll
        for (int u = 0; u < DENSE_UN; ++u) {
            const int q = q0 + 32 * u;
            const bool on = q < end;
            const unsigned d = (unsigned)(w.start[t + 1 + lane] - q);
            const unsigned m = __reduce_or_sync(SPG_FULL, (on && d < 32u) ? 1u << d : 0u);
            const int pt = t + __popc(m & le);
            ok[u] = on && q + lane < T;
            p[u] = w.base[pt] + (q + lane);
            if (VALS) a[u] = w.av[pt];
            t += __popc(m);
        }
        f(p, a, ok, std::false_type());
    }
}

// ---- the column bitmap of a (row, slice) ----

// The next (item, slice) of a CTA: blockIdx.x, then + gridDim.x (a grid that covers the
// items takes one each), or, with a work counter, the counter's next ticket (a persistent
// grid over a count read on the device).  All threads call it; its barrier ends the
// previous item's use of shared memory.
SPG_DEV int64_t dense_next(unsigned long long *counter, int64_t cur, bool first, int64_t *s_b) {
    __syncthreads();
    if (counter == nullptr) return first ? (int64_t)blockIdx.x : cur + gridDim.x;
    if (threadIdx.x == 0) *s_b = (int64_t)atomicAdd(counter, 1ull);
    __syncthreads();
    return *s_b;
}

// Starts moving `bytes` (a multiple of 16) at p (16-byte aligned) from memory into L2; the
// copy completes on its own, nothing waits for it.
SPG_DEV void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The (row, slice) items of the wide rows.
SPG_DEV int64_t dense_items(const DenseArgs &D) { return (D.dev_end != nullptr ? D.dev_end[0] : D.n_wide) * (int64_t)D.K; }

// The columns of slice s that row d of the dense items can reach: [lo, lo + span).
SPG_DEV int dense_span(const DevCSR &B, const DenseArgs &D, int64_t d, int s, int64_t &lo) {
    lo = max((int64_t)s * D.W, (int64_t)D.clo[d]);
    return (int)(min(min((int64_t)(s + 1) * D.W, B.ncols), (int64_t)D.chi[d]) - lo);
}

// Marks the column offset x of every product of the row in the slice with mark(x).  Returns
// whether a column lay outside [lo, lo + span) (cannot happen: the slice boundaries select
// the columns); a barrier must follow before the marks are read.
template <int NT, bool TAB, typename M>
SPG_DEV bool dense_mark_columns(const DevCSR &A, const DevCSR &B, const DenseArgs &D, int row, int s, int64_t lo,
                                int span, DenseWin<NT> &win, M mark) {
    bool bad = false;
    const int64_t a0 = A.rp[row], a1 = A.rp[row + 1];
    for (int64_t e = a0; e < a1; e += NT) {
        const int T = dense_window<NT, false, TAB>(A, B, D, s, e, a1, win);
        dense_walk<NT, false>(win, T, [&](const int64_t *p, const val_t *, const bool *ok, auto full) {
            int32_t c[DENSE_UN];
#pragma unroll
            for (int u = 0; u < DENSE_UN; ++u)
                if (full || ok[u]) c[u] = __ldg(B.col + p[u]);
#pragma unroll
            for (int u = 0; u < DENSE_UN; ++u) {
                if (!full && !ok[u]) continue;
                const int x = (int)(c[u] - lo);
                if ((unsigned)x < (unsigned)span) mark(x);
                else bad = true;
            }
        });
    }
    return bad;
}

// ---- pass 1: the number of columns of every (row, slice) ----
// Shared memory: the slice's column bitmap (one bit per column), then its popcount.  Bound by
// the gather of B's columns and the shared atomics on the bitmap.
template <int NT, bool TAB>
SPG_DEV void dense_count_item(const DevCSR &A, const DevCSR &B, const DenseArgs &D, int64_t b, int64_t *err) {
    extern __shared__ __align__(16) uint32_t dc_bm[];
    __shared__ DenseWin<NT> win;
    __shared__ int32_t scan32[NT / 32 + 1];
    const int64_t d = b / D.K;
    const int s = (int)(b - d * D.K);
    int64_t lo;
    const int span = dense_span(B, D, d, s, lo);
    if (span <= 0) {
        if (threadIdx.x == 0) D.cnt[b] = 0;
        return;
    }
    const int ng = (((span + 31) >> 5) + 3) >> 2;  // 16-byte groups of bitmap words
    uint4 *b4 = reinterpret_cast<uint4 *>(dc_bm);
    for (int q = threadIdx.x; q < ng; q += NT) b4[q] = make_uint4(0u, 0u, 0u, 0u);
    // (the first window's barriers come before the first mark)
    const bool bad = dense_mark_columns<NT, TAB>(A, B, D, D.rows[d], s, lo, span, win,
                                            [&](int x) { atomicOr(&dc_bm[x >> 5], 1u << (x & 31)); });
    __syncthreads();
    int n = 0;
    uint4 *k4 = D.keep != nullptr ? reinterpret_cast<uint4 *>(D.keep + b * (int64_t)D.keep_words) : nullptr;
    for (int q = threadIdx.x; q < ng; q += NT) {
        const uint4 v = b4[q];
        n += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        if (k4 != nullptr) k4[q] = v;  // for the fill (whole groups: the words past the span are clear)
    }
    n = block_reduce_sum<NT, int>(n, scan32);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicExch((unsigned long long *)err, 5ull);
    if (threadIdx.x == 0) D.cnt[b] = n;
}

template <int NT, bool TAB>
__global__ void __launch_bounds__(NT, 1536 / NT)
k_dense_count(DevCSR A, DevCSR B, DenseArgs D, int64_t *err) {
    __shared__ int64_t s_b;
    unsigned long long *q = D.dev_end != nullptr ? D.queue : nullptr;
    const int64_t nb = dense_items(D);
    for (int64_t b = dense_next(q, 0, true, &s_b); b < nb; b = dense_next(q, b, false, &s_b))
        dense_count_item<NT, TAB>(A, B, D, b, err);
}

// One thread per dense item: the slices' offsets inside the row and the row's length.
__global__ void k_dense_rows(MergeItems it, DenseArgs D) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= D.n) return;
    int32_t acc = 0;
    for (int s = 0; s < D.K; ++s) {
        D.soff[d * D.K + s] = acc;
        acc += D.cnt[d * D.K + s];
    }
    const int j = D.items[d];
    it.len[j] = acc;
    it.src_len[j] = 0;
    it.home_cap[j] = 0;
    it.home_col[j] = nullptr;
    it.home_val[j] = nullptr;
    it.child[j] = ITEM_DENSE;
}

// ---- pass 2: the values, written into C ----
// Shared memory: per 32-column word of the slice the pair (bits, set bits in the words before
// it).  A product's column x has the position rank + popc(bits below x) among the slice's
// columns, i.e. its place in the row of C, so one 8-byte shared load leads from a column to
// its sum.  The columns are written and the sums cleared first, straight in C; in double
// precision every product is then added in C itself (an atomic add performed in L2, which
// holds the slice just cleared): no buffer of sums, so a CTA needs 42 KB for the widest slice,
// four CTAs of 256 threads share an SM and any number of entries takes one pass.  Measured over the chip
// with random addresses: 214-280 G adds/s in L2 against 288-372 G/s for fp64 atomics in shared
// memory, which would leave one or two CTAs per SM.  In single precision the sums are kept in
// shared memory (SHV: 786-1,171 G adds/s, and global float atomics flush denormals), one per
// column of the result, in pieces when a slice has more entries than the buffer holds.

__host__ __device__ inline int dense_nw4(int W) { return ((W + 31) / 32 + 4) & ~3; }

// Turns the words of a slice's bitmap into the index: the groups of four words from src(g)
// are counted, ranked and written as pairs.  Unless enter(number of set bits) is false (the
// caller must then return), put(w) is called by whole warps for every 32 words from w on, once
// their pairs are written.  The index is complete after the caller's next barrier.
template <int NT, typename S, typename E, typename P>
SPG_DEV bool dense_index(uint2 *idx, int nwords, int32_t *scan32, S src, E enter, P put) {
    constexpr int NW = NT / 32, RG = (DENSE_W_MAX / 128 + NT - 1) / NT;
    const int lane = lane_id(), wid = warp_id();
    const int ng = (nwords + 3) >> 2;
    const int per = (ng + NT - 1) / NT;  // at most RG: each warp takes per * 32 consecutive groups
    uint4 b[RG];
    int mine = 0;
#pragma unroll
    for (int i = 0; i < RG; ++i) {
        const int g = (wid * per + i) * 32 + lane;
        b[i] = (i < per && g < ng) ? src(g) : make_uint4(0u, 0u, 0u, 0u);
        mine += __popc(b[i].x) + __popc(b[i].y) + __popc(b[i].z) + __popc(b[i].w);
    }
    mine = warp_reduce_sum(mine);
    if (lane == 0) scan32[wid] = mine;
    __syncthreads();
    int run = 0, tot = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        const int c = scan32[k];
        if (k < wid) run += c;
        tot += c;
    }
    if (!enter(tot)) return false;
#pragma unroll
    for (int i = 0; i < RG; ++i) {
        if (i >= per) break;
        const int g = (wid * per + i) * 32 + lane;
        const int c0 = __popc(b[i].x), c1 = c0 + __popc(b[i].y), c2 = c1 + __popc(b[i].z), c3 = c2 + __popc(b[i].w);
        const int inc = warp_inclusive_scan(c3);
        const int ex = run + inc - c3;
        run += __shfl_sync(SPG_FULL, inc, 31);
        if (g < ng) {
            uint4 *o4 = reinterpret_cast<uint4 *>(idx + 4 * g);
            o4[0] = make_uint4(b[i].x, (unsigned)ex, b[i].y, (unsigned)(ex + c0));
            o4[1] = make_uint4(b[i].z, (unsigned)(ex + c1), b[i].w, (unsigned)(ex + c2));
        }
        __syncwarp();
        for (int w = 4 * (g - lane); w < nwords && w < 4 * (g - lane) + 128; w += 32) put(w);
    }
    return true;
}

// REPLAY: values-only replay; C's columns are already in place, so the bitmap is built
// from the slice's known entries of C and only the values are written.
template <int NT, bool REPLAY, bool SHV, bool TAB>
SPG_DEV void dense_fill_item(const DevCSR &A, const DevCSR &B, const DenseArgs &D, int64_t b, const int64_t *c_rp,
                             int32_t *c_col, val_t *c_val, int64_t *err, int vcap) {
    extern __shared__ __align__(16) unsigned char df_smem[];
    __shared__ DenseWin<NT> win;
    __shared__ int32_t scan32[NT / 32 + 1];
    __shared__ uint16_t stage[NT / 32][DENSE_STAGE];
    const int expected = D.cnt[b];  // > 0
    const int64_t d = b / D.K;
    const int s = (int)(b - d * D.K);
    const int row = D.rows[d];
    // the slice's columns that the row can reach (non-empty: the slice has columns of the row)
    int64_t lo;
    const int span = dense_span(B, D, d, s, lo);
    const int nwords = (span + 31) >> 5;
    const int64_t o = c_rp[row] + D.soff[b];  // the slice's first entry in C
    uint2 *idx = reinterpret_cast<uint2 *>(df_smem);
    val_t *V = reinterpret_cast<val_t *>(idx + dense_nw4(D.W));
    bool bad = false;
    // ---- the slice's columns ----
    const bool kept = !REPLAY && D.keep != nullptr;
    if (!kept) {
        uint4 *i4 = reinterpret_cast<uint4 *>(idx);
        for (int q = threadIdx.x; q < 2 * ((nwords + 3) >> 2); q += NT) i4[q] = make_uint4(0u, 0u, 0u, 0u);
        auto mark = [&](int x) { atomicOr(&idx[x >> 5].x, 1u << (x & 31)); };
        if (REPLAY) {
            __syncthreads();
            for (int t = threadIdx.x; t < expected; t += NT) {
                const int x = (int)(c_col[o + t] - lo);
                if ((unsigned)x < (unsigned)span) mark(x);
                else bad = true;  // C's columns were changed since the product
            }
        } else {
            bad = dense_mark_columns<NT, TAB>(A, B, D, row, s, lo, span, win, mark);
        }
        __syncthreads();
    }
    const uint4 *k4 = kept ? reinterpret_cast<const uint4 *>(D.keep + b * (int64_t)D.keep_words) : nullptr;
    const uint4 *i4 = reinterpret_cast<const uint4 *>(idx);
    const bool match = dense_index<NT>(
        idx, nwords, scan32,
        [&](int g) {
            if (kept) return __ldg(k4 + g);
            const uint4 p = i4[2 * g], q = i4[2 * g + 1];
            return make_uint4(p.x, p.z, q.x, q.z);
        },
        [&](int tot) { return tot == expected; },
        [&](int w) {
            // C's columns of 32 words, a word per lane
            if (REPLAY) return;
            const int lane = lane_id();
            const uint2 wd = w + lane < nwords ? idx[w + lane] : make_uint2(0u, 0u);
            uint32_t bits = wd.x;
            const unsigned some = __ballot_sync(SPG_FULL, bits != 0u);
            if (some == 0u) return;
            const int last = 31 - __clz(some);
            const int r0 = __shfl_sync(SPG_FULL, (int)wd.y, __ffs(some) - 1);
            const int n = __shfl_sync(SPG_FULL, (int)wd.y + __popc(bits), last) - r0;
            if (!SPG_IN(r0 + n <= expected, 110)) return;  // the slice's entries of C
            const int32_t base = (int32_t)(lo + ((int64_t)w << 5));
            if (n <= DENSE_STAGE) {
                // few columns per word: staged, so that the warp's stores are contiguous (lane by
                // lane every store would touch a sector of its own)
                uint16_t *sg = stage[warp_id()];
                for (int q = (int)wd.y - r0; bits; bits &= bits - 1u) sg[q++] = (uint16_t)((lane << 5) + __ffs(bits) - 1);
                __syncwarp();
                for (int t = lane; t < n; t += 32) c_col[o + r0 + t] = base + sg[t];
                __syncwarp();
            } else {
                int64_t q = o + (int)wd.y;
                for (; bits; bits &= bits - 1u) c_col[q++] = base + (lane << 5) + __ffs(bits) - 1;
            }
        });
    if (!match) {  // the counting pass saw other columns: cannot happen
        if (threadIdx.x == 0) atomicExch((unsigned long long *)err, 6ull);
        return;
    }
    if (!SHV)
        for (int t = threadIdx.x; t < expected; t += NT) c_val[o + t] = val_t(0);
    // ---- the sums: in C at once, or in pieces of at most vcap entries in V ----
    const int64_t a0 = A.rp[row], a1 = A.rp[row + 1];
    for (int w0 = 0; w0 < nwords;) {
        int w1 = nwords, e0 = 0, n = expected;
        if (SHV) {
            __syncthreads();  // the index is complete, and V is free
            auto rank_at = [&](int w) { return w < nwords ? (int)idx[w].y : expected; };
            // the last word end w1 with rank_at(w1) - e0 <= vcap (a word holds <= 32 <= vcap entries)
            e0 = rank_at(w0);
            if (expected - e0 > vcap) {
                int l = w0 + 1, h = nwords;
                while (l < h) {
                    const int mid = (l + h + 1) >> 1;
                    if (rank_at(mid) - e0 <= vcap) l = mid; else h = mid - 1;
                }
                w1 = l;
            }
            n = rank_at(w1) - e0;
            for (int k = threadIdx.x; k < n; k += NT) V[k] = val_t(0);
        }
        const int x0 = w0 << 5, x1 = min(span, w1 << 5);
        for (int64_t e = a0; e < a1; e += NT) {
            const int T = dense_window<NT, true, TAB>(A, B, D, s, e, a1, win);
            dense_walk<NT, true>(win, T, [&](const int64_t *p, const val_t *a, const bool *ok, auto full) {
                int32_t c[DENSE_UN];
                val_t v[DENSE_UN];
#pragma unroll
                for (int u = 0; u < DENSE_UN; ++u)
                    if (full || ok[u]) c[u] = __ldg(B.col + p[u]);
#pragma unroll
                for (int u = 0; u < DENSE_UN; ++u)
                    if (full || ok[u]) v[u] = __ldg(B.val + p[u]);
#pragma unroll
                for (int u = 0; u < DENSE_UN; ++u) {
                    if (!full && !ok[u]) continue;
                    const int x = (int)(c[u] - lo);
                    if (SHV && (x < x0 || x >= x1)) continue;  // another piece's
                    const bool in = (unsigned)x < (unsigned)span;
                    const uint2 wd = in ? idx[x >> 5] : make_uint2(0u, 0u);
                    if (!((wd.x >> (x & 31)) & 1u)) {
                        bad = true;  // a column the bitmap does not hold (the structure changed)
                        continue;
                    }
                    const int q = (int)wd.y + __popc(wd.x & ((1u << (x & 31)) - 1u));
                    if (!SPG_IN(q >= e0 && q - e0 < n, 109)) continue;
                    if (SHV) atomicAdd(&V[q - e0], a[u] * v[u]);
                    else atomicAdd(&c_val[o + q], a[u] * v[u]);
                }
            });
        }
        if (SHV) {
            __syncthreads();
            if (SPG_IN(e0 + n <= expected, 111))
                for (int k = threadIdx.x; k < n; k += NT) c_val[o + e0 + k] = V[k];
        }
        w0 = w1;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicExch((unsigned long long *)err, 6ull);
}

// Ticket t of a grid of `ctas`: the first item of its run and the run's length.  The first four
// tickets per CTA are single items (the list begins with the heaviest rows), the next four are
// pairs, and so on up to runs of 32.
SPG_DEV int64_t dense_run(int64_t t, int64_t ctas, int &len) {
    const int64_t c = 4 * ctas;
    const int64_t l = min(t / c, (int64_t)5);
    len = 1 << l;
    return c * (len - 1) + (t - l * c) * len;
}

// A persistent grid over the items whose count lies in (cmin, cmax].  A CTA takes a run of
// consecutive items from the work counter, looks at all their counts at once and fills the
// ones that are its own.
template <int NT, int MINB, bool REPLAY, bool SHV, bool TAB>
__global__ void __launch_bounds__(NT, MINB)
k_dense_fill(DevCSR A, DevCSR B, DenseArgs D, const int64_t *c_rp, int32_t *c_col, val_t *c_val, int64_t *err,
             const int64_t *gate, int vcap, unsigned long long *counter, int cmin, int cmax) {
    __shared__ int64_t s_base;
    __shared__ unsigned s_mask;
    if (gated(gate)) return;
    const int64_t nb = dense_items(D);
    while (true) {
        if (threadIdx.x < 32) {
            int64_t t = 0;
            if (threadIdx.x == 0) t = (int64_t)atomicAdd(counter, 1ull);
            int run;
            const int64_t base = dense_run(__shfl_sync(SPG_FULL, t, 0), gridDim.x, run);
            const int64_t i = base + threadIdx.x;
            const int c = ((int)threadIdx.x < run && i < nb) ? D.cnt[i] : 0;
            const unsigned m = __ballot_sync(SPG_FULL, c > cmin && c <= cmax);
            if (threadIdx.x == 0) {
                s_base = base;
                s_mask = m;
            }
        }
        __syncthreads();
        const int64_t base = s_base;
        unsigned mask = s_mask;
        if (base >= nb) return;
        while (mask) {
            const int64_t b = base + __ffs(mask) - 1;
            mask &= mask - 1u;
            // the next item's kept bitmap (written by the counting pass, long out of L2) is on its
            // way into L2 while this item is filled
            if (threadIdx.x == 0 && !REPLAY && D.keep != nullptr && mask)
                prefetch_l2(D.keep + (base + __ffs(mask) - 1) * (int64_t)D.keep_words, 4u * (uint32_t)D.keep_words);
            dense_fill_item<NT, REPLAY, SHV, TAB>(A, B, D, b, c_rp, c_col, c_val, err, vcap);
            __syncthreads();  // the item's shared memory is free
        }
        __syncthreads();  // every thread has read the run before the next one
    }
}

// ---- rows that reach few columns: a warp per row ----
// A band, a block or a stencil's neighbourhood: at most W columns, whatever B's width.  One
// warp holds a sum per column in shared memory and takes the B rows one after another, 32
// entries at a time: their columns are distinct, so plain fused multiply-adds suffice, and no
// barrier wider than the warp is needed.  A*A of a band matrix of 50,021 rows and width 40 (80 M
// products, single precision) takes 404 us as a whole, 73 of them for the count; 490 us with all
// sums in shared memory, 3.39 ms with a CTA per row and 1.75 ms with the product walk above.
// Bound by shared memory (issue where registers hold the sums) and, in double precision, the
// FP64 pipe.
// The columns are a bitmap, a word per lane.  A B row whose entries are consecutive columns
// (last - first + 1 = length, as in a band or a block) sets its bits and finds its columns
// without reading them, and 32 such rows (a window of A) are summed in registers: lane l holds
// the sums of columns l, l + 32, ..., and no sum passes through shared memory.
constexpr int DN_WARPS = 8;
constexpr int DN_AHEAD = 4;  // steps of 32 products whose loads are in flight
// Register steps (a word of the range for one part) taken for one shared-memory step of 32
// products.  Float: bands of 24 to 100 entries 334-1619 -> 312-1239 us for the product, a band
// of 201 times one of 3 is better left in shared memory (1364 against 1974 us).  Double: FMAs of
// lanes outside a part cost as much as the others (a band of 64: 893 us in shared memory, 1090
// in registers), so only where the parts fill their words (blocks of 64: 905 -> 755 us).
constexpr int DN_REG_PER_STEP = sizeof(val_t) == 4 ? 4 : 1;

struct __align__(16) DensePart {
    int64_t p0;  // first entry in B
    int32_t x0;  // first column - lo
    int32_t len; // entries; negative: consecutive columns
};
struct DenseParts {  // per warp: 32 B rows
    DensePart part[32];
    val_t a[32];     // a_ik
    uint32_t bits[32];
};

// FILL: sums and C's row (REPLAY: its values only); else the row's count per slice.
template <int W, bool FILL, bool REPLAY>
__global__ void __launch_bounds__(DN_WARPS * 32)
k_dense_narrow(DevCSR A, DevCSR B, DenseArgs D, const int64_t *__restrict__ c_rp, int32_t *__restrict__ c_col,
               val_t *__restrict__ c_val, int64_t *err, const int64_t *gate) {
    static_assert(W % 32 == 0 && W <= 1024, "a bitmap word per lane");
    __shared__ DenseParts parts[DN_WARPS];
    extern __shared__ __align__(16) unsigned char dn_smem[];
    if (FILL && gated(gate)) return;
    const int lane = lane_id();
    DenseParts &S = parts[warp_id()];
    val_t *V = reinterpret_cast<val_t *>(dn_smem) + (FILL ? warp_id() * W : 0);
    const int64_t i0 = D.dev_end ? D.dev_end[0] : (W == DENSE_MID_W ? D.n_wide : D.n_mid);
    // with the counts on the device, one launch (of the wider kernel) takes all of them
    const int64_t i1 = D.dev_end ? *D.dev_n : (W == DENSE_MID_W ? D.n_mid : D.n);
    for (int64_t d = i0 + (int64_t)blockIdx.x * DN_WARPS + warp_id(); d < i1; d += (int64_t)gridDim.x * DN_WARPS) {
        const int row = D.rows[d];
        const int32_t lo = D.clo[d];
        const int span = min(D.chi[d] - lo, W);
        uint32_t known = 0;       // replay: the columns of C's row
        bool bad = D.chi[d] - lo > W;  // cannot happen: the items were chosen by their width
        S.bits[lane] = 0;
        int64_t o = 0;
        int n = 0;
        if (FILL) {
            o = c_rp[row];
            n = (int)(c_rp[row + 1] - o);
            for (int x = lane; x < span; x += 32) V[x] = val_t(0);
        }
        __syncwarp();
        if (REPLAY) {
            for (int t = lane; t < n; t += 32) {
                const int x = c_col[o + t] - lo;
                if ((unsigned)x < (unsigned)span) atomicOr(&S.bits[x >> 5], 1u << (x & 31));
                else bad = true;  // C's columns were changed since the product
            }
            __syncwarp();
            known = S.bits[lane];
            __syncwarp();
            S.bits[lane] = 0;
            __syncwarp();
        }
        uint32_t mine = 0;  // bits of columns [32 lane, 32 lane + 32) set by consecutive parts
        constexpr int REGS = FILL && W <= 256 ? W / 32 : 0;
        val_t acc[REGS > 0 ? REGS : 1];
#pragma unroll
        for (int r = 0; r < REGS; ++r) acc[r] = val_t(0);
        const int64_t a0 = A.rp[row], a1 = A.rp[row + 1];
        for (int64_t e = a0; e < a1; e += 32) {
            int len = 0, x0 = 0;
            bool run = false;
            int64_t rs = 0;
            val_t av = val_t(0);
            if (e + lane < a1) {
                const int32_t k = A.col[e + lane];
                if (FILL) av = A.val[e + lane];
                rs = B.rp[k];
                len = (int)(B.rp[k + 1] - rs);
                if (len > 0) {
                    const int32_t f = B.col[rs], l = B.col[rs + len - 1];
                    x0 = f - lo;
                    run = l - f + 1 == len;
                    // cannot happen: [lo, hi) covers the columns of the row's parts
                    if (x0 < 0 || l - lo >= span) {
                        bad = true;
                        len = 0;
                    }
                }
            }
            const unsigned nz = __ballot_sync(SPG_FULL, len > 0);
            const int np = __popc(nz);
            if (len > 0) {
                const int q = __popc(nz & ((1u << lane) - 1u));
                S.part[q] = DensePart{rs, x0, run ? -len : len};
                if (FILL) S.a[q] = av;
            }
            // every column of the range is asked for every part: not for parts much shorter
            const bool runs = FILL && REGS > 0 && !__any_sync(SPG_FULL, len > 0 && !run) &&
                              DN_REG_PER_STEP * (int)__reduce_add_sync(SPG_FULL, (unsigned)(len + 31) >> 5) >= np * ((span + 31) >> 5);
            __syncwarp();
            // the columns
            for (int t = 0; t < np; ++t) {
                const int ln = S.part[t].len, f = S.part[t].x0;
                if (ln < 0) {
                    const int b0 = max(f - 32 * lane, 0), b1 = min(f - ln - 32 * lane, 32);
                    if (b0 < b1) mine |= (b1 - b0 == 32 ? ~0u : ((1u << (b1 - b0)) - 1u) << b0);
                } else {
                    const int64_t p = S.part[t].p0;
                    for (int i = lane; i < ln; i += 32) {
                        const int x = __ldg(B.col + p + i) - lo;
                        if ((unsigned)x < (unsigned)span) atomicOr(&S.bits[x >> 5], 1u << (x & 31));
                        else bad = true;
                    }
                }
            }
            if (runs) {
#pragma unroll
                for (int r = 0; r < REGS; ++r) {
                    if (32 * r >= span) break;
                    const int x = 32 * r + lane;
                    for (int t = 0; t < np; t += DN_AHEAD) {
                        val_t v[DN_AHEAD];
                        bool ok[DN_AHEAD];
#pragma unroll
                        for (int u = 0; u < DN_AHEAD; ++u) {
                            ok[u] = false;
                            if (t + u < np) {
                                const DensePart q = S.part[t + u];
                                ok[u] = (unsigned)(x - q.x0) < (unsigned)-q.len;
                                if (ok[u]) v[u] = __ldg(B.val + q.p0 + (x - q.x0));
                            }
                        }
#pragma unroll
                        for (int u = 0; u < DN_AHEAD; ++u)
                            if (ok[u]) acc[r] = fma(S.a[t + u], v[u], acc[r]);
                    }
                }
            } else if (FILL) {
                // steps (part t, entries i0..i0+31), their loads DN_AHEAD steps ahead
                val_t v[DN_AHEAD];
                int32_t c[DN_AHEAD];
                int lt = 0, li = 0;  // the next step to load
                auto load = [&](val_t &vv, int32_t &cc) {
                    if (lt >= np) return;
                    const DensePart q = S.part[lt];
                    const int ln = q.len, m = ln < 0 ? -ln : ln;
                    const int64_t p = q.p0 + li + lane;
                    if (li + lane < m) {
                        vv = __ldg(B.val + p);
                        cc = ln < 0 ? q.x0 + li + lane : __ldg(B.col + p) - lo;
                    }
                    li += 32;
                    if (li >= m) {
                        li = 0;
                        ++lt;
                    }
                };
#pragma unroll
                for (int u = 0; u < DN_AHEAD; ++u) load(v[u], c[u]);
                for (int t = 0, i = 0; t < np;) {
#pragma unroll
                    for (int u = 0; u < DN_AHEAD; ++u) {
                        if (t < np) {
                            const int ln = S.part[t].len, m = ln < 0 ? -ln : ln;
                            if (i + lane < m && (unsigned)c[u] < (unsigned)span) V[c[u]] = fma(S.a[t], v[u], V[c[u]]);
                            i += 32;
                            if (i >= m) {
                                i = 0;
                                ++t;
                            }
                            __syncwarp();  // the next B row may add into the same columns
                            load(v[u], c[u]);
                        }
                    }
                }
            }
            __syncwarp();  // the table is reused
        }
        const uint32_t bits = mine | S.bits[lane];
        if (!FILL) {
            // the columns of every slice the range touches, and zeros elsewhere
            for (int s = lane; s < D.K; s += 32) D.cnt[d * D.K + s] = 0;
            __syncwarp();
            const int s0 = lo / D.W, s1 = (lo + span - 1) / D.W;
            for (int s = s0; s <= s1 && s < D.K; ++s) {
                const int64_t b = (int64_t)s * D.W - lo - 32 * lane;  // the slice's first column in this lane's word
                const int b0 = (int)max(min(b, (int64_t)32), (int64_t)0), b1 = (int)max(min(b + D.W, (int64_t)32), (int64_t)0);
                const uint32_t m = b1 > b0 ? (b1 - b0 == 32 ? ~0u : ((1u << (b1 - b0)) - 1u) << b0) : 0u;
                const int c = __reduce_add_sync(SPG_FULL, __popc(bits & m));
                if (lane == 0) D.cnt[d * D.K + s] = c;
            }
            if (__any_sync(SPG_FULL, bad) && lane == 0) atomicExch((unsigned long long *)err, 5ull);
        } else {
            const int cw = __popc(bits);
            const int inc = warp_inclusive_scan(cw);
            // every product's column is in C, and (but in a replay) C holds nothing else
            if (REPLAY ? (bits & ~known) != 0u : __shfl_sync(SPG_FULL, inc, 31) != n) bad = true;
            if (__any_sync(SPG_FULL, bad)) {
                if (lane == 0) atomicExch((unsigned long long *)err, 6ull);
                __syncwarp();
                continue;
            }
#pragma unroll
            for (int r = 0; r < REGS; ++r)
                if (32 * r + lane < span) V[32 * r + lane] += acc[r];
            __syncwarp();
            const uint32_t out = REPLAY ? known : bits;
            const int ow = __popc(out);
            const int before = warp_inclusive_scan(ow) - ow;
            unsigned words = __ballot_sync(SPG_FULL, out != 0u);
            while (words) {  // a word's columns are consecutive entries of C
                const int w = __ffs(words) - 1;
                words &= words - 1u;
                const uint32_t wd = __shfl_sync(SPG_FULL, out, w);
                const int r = __shfl_sync(SPG_FULL, before, w);
                if ((wd >> lane) & 1u) {
                    const int q = r + __popc(wd & ((1u << lane) - 1u));
                    if (!SPG_IN(q < n, 113)) continue;  // the row's entries of C
                    if (!REPLAY) c_col[o + q] = lo + 32 * w + lane;
                    c_val[o + q] = V[32 * w + lane];
                }
            }
            __syncwarp();  // the sums are cleared for the next row
        }
    }
}

template <int W, bool FILL, bool REPLAY>
static cudaError_t launch_narrow(const DevCSR &A, const DevCSR &B, const DenseArgs &D, const int64_t *c_rp,
                                 int32_t *c_col, val_t *c_val, int64_t *err, const int64_t *gate, cudaStream_t st) {
    const int64_t n = D.dev_end != nullptr ? D.n : (W == DENSE_MID_W ? D.n_mid - D.n_wide : D.n - D.n_mid);
    if (n <= 0) return cudaSuccess;
    auto kern = k_dense_narrow<W, FILL, REPLAY>;
    const int smem = FILL ? DN_WARPS * W * (int)sizeof(val_t) : 0;
    cudaError_t e = allow_dynamic_smem((const void *)kern, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    const int64_t need = (n + DN_WARPS - 1) / DN_WARPS;
    const int64_t grid = D.dev_end != nullptr ? persistent_blocks((const void *)kern, DN_WARPS * 32, smem, need) : need;
    if (grid <= 0 || grid > INT32_MAX) return cudaErrorInvalidValue;
    kern<<<(unsigned)grid, DN_WARPS * 32, smem, st>>>(A, B, D, c_rp, c_col, c_val, err, gate);
    return cudaGetLastError();
}

template <bool FILL, bool REPLAY>
static cudaError_t launch_narrow_rows(const DevCSR &A, const DevCSR &B, const DenseArgs &D, const int64_t *c_rp,
                                      int32_t *c_col, val_t *c_val, int64_t *err, const int64_t *gate,
                                      cudaStream_t st) {
    cudaError_t e = launch_narrow<DENSE_MID_W, FILL, REPLAY>(A, B, D, c_rp, c_col, c_val, err, gate, st);
    if (e == cudaSuccess && D.dev_end == nullptr)
        e = launch_narrow<DENSE_NARROW_W, FILL, REPLAY>(A, B, D, c_rp, c_col, c_val, err, gate, st);
    return e;
}

// One thread per dense item (precise method): the slices' offsets inside the row and the
// row's size nnz(c_i), the sum of its slices' counts.
__global__ void k_dense_rowsum(DenseArgs D, int32_t *nnzc) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n = D.dev_n != nullptr ? *D.dev_n : D.n;
    if (d >= n) return;
    int32_t acc = 0;
    for (int s = 0; s < D.K; ++s) {
        D.soff[d * D.K + s] = acc;
        acc += D.cnt[d * D.K + s];
    }
    nnzc[D.rows[d]] = acc;
}

constexpr int DENSE_NT = 256;
constexpr int DENSE_FEW = 4096;  // entries of a (row, slice) filled by the smaller CTAs in double

// The parts' places come from the table (or one slice holds whole rows), else from searches.
static bool dense_tabled(const DenseArgs &D) { return D.K == 1 || D.bnd != nullptr; }

int dense_keep_words(int W) { return dense_nw4(W); }  // a multiple of 4: every item's bitmap starts on a 16-byte boundary

static cudaError_t dense_check(const DevCSR &B, const DenseArgs &D) {
    if (D.n * D.K > INT32_MAX || D.W % 32 != 0 || D.W > DENSE_W_MAX || (int64_t)D.K * D.W < B.ncols || D.queue == nullptr)
        return cudaErrorInvalidValue;
    if (D.keep != nullptr && (D.keep_words < dense_nw4(D.W) || D.keep_words % 4 != 0)) return cudaErrorInvalidValue;
    return cudaSuccess;
}

cudaError_t launch_dense_count(const DevCSR &A, const DevCSR &B, const DenseArgs &D, int64_t *err, cudaStream_t st) {
    if (D.n <= 0) return cudaSuccess;
    const int64_t nb = (D.dev_end != nullptr ? D.n : D.n_wide) * D.K;
    cudaError_t e = dense_check(B, D);
    if (e == cudaSuccess) e = launch_narrow_rows<false, false>(A, B, D, nullptr, nullptr, nullptr, err, nullptr, st);
    if (e != cudaSuccess || nb <= 0) return e;
    const int smem = (int)(sizeof(uint32_t) * dense_nw4(D.W));
    auto kern = dense_tabled(D) ? k_dense_count<DENSE_NT, true> : k_dense_count<DENSE_NT, false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    int64_t grid = nb;
    if (D.dev_end != nullptr) {  // persistent grid over the items counted on the device
        e = cudaMemsetAsync(D.queue, 0, sizeof(unsigned long long), st);
        if (e != cudaSuccess) return e;
        grid = persistent_blocks((const void *)kern, DENSE_NT, smem, nb);
        if (grid <= 0) return cudaErrorInvalidValue;
    }
    kern<<<(unsigned)grid, DENSE_NT, smem, st>>>(A, B, D, err);
    return cudaGetLastError();
}

cudaError_t launch_dense_rowsum(const DenseArgs &D, int32_t *nnzc, cudaStream_t st) {
    if (D.n <= 0) return cudaSuccess;
    k_dense_rowsum<<<(unsigned)((D.n + 127) / 128), 128, 0, st>>>(D, nnzc);
    return cudaGetLastError();
}

cudaError_t launch_dense_rows(const MergeItems &it, const DenseArgs &D, cudaStream_t st) {
    if (D.n <= 0) return cudaSuccess;
    k_dense_rows<<<(unsigned)((D.n + 127) / 128), 128, 0, st>>>(it, D);
    return cudaGetLastError();
}

template <bool TAB>
static cudaError_t launch_fill(const DevCSR &A, const DevCSR &B, const DenseArgs &D, const int64_t *c_rp, int32_t *c_col,
                               val_t *c_val, int64_t *err, cudaStream_t st, bool replay, const int64_t *gate) {
    if (D.n <= 0) return cudaSuccess;
    cudaError_t e = dense_check(B, D);
    if (e == cudaSuccess)
        e = replay ? launch_narrow_rows<true, true>(A, B, D, c_rp, c_col, c_val, err, gate, st)
                   : launch_narrow_rows<true, false>(A, B, D, c_rp, c_col, c_val, err, gate, st);
    const int64_t nb = (D.dev_end != nullptr ? D.n : D.n_wide) * D.K;
    if (e != cudaSuccess || nb <= 0) return e;
    e = cudaMemsetAsync(D.queue + 1, 0, sizeof(unsigned long long) * (DENSE_QUEUES - 1), st);
    if (e != cudaSuccess) return e;
    // a persistent grid of nt threads per CTA over the items with counts in (cmin, cmax]
    auto go = [&](auto kern, int nt, int smem, int vcap, unsigned long long *q, int cmin, int cmax) -> cudaError_t {
        cudaError_t x = allow_dynamic_smem((const void *)kern, smem);
        if (x == cudaSuccess) x = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (x != cudaSuccess) return x;
        const int grid = persistent_blocks((const void *)kern, nt, smem, nb);
        if (grid <= 0) return cudaErrorInvalidValue;
        kern<<<(unsigned)grid, nt, smem, st>>>(A, B, D, c_rp, c_col, c_val, err, gate, vcap, q, cmin, cmax);
        return cudaGetLastError();
    };
    const int index = (int)(sizeof(uint2) * (size_t)dense_nw4(D.W));
    if constexpr (sizeof(val_t) == 8) {
        // few entries: four CTAs of 256 threads per SM.  Many: two of 512, half as many rows of C
        // in flight, since their sums must stay in L2 while they are added to (16 k entries per
        // row, R-MAT 2^16 x 16: 1.62 ms at 304 CTAs, 2.34 at 608, 2.90 at 760; 3.2 k entries, 2^18 x
        // 8: 10.2 ms at 304, 8.8 at 608)
        e = replay ? go(k_dense_fill<256, 4, true, false, TAB>, 256, index, 0, D.queue + 1, 0, DENSE_FEW)
                   : go(k_dense_fill<256, 4, false, false, TAB>, 256, index, 0, D.queue + 1, 0, DENSE_FEW);
        if (e != cudaSuccess || D.W <= DENSE_FEW) return e;  // a slice has at most W entries
        return replay ? go(k_dense_fill<512, 2, true, false, TAB>, 512, index, 0, D.queue + 2, DENSE_FEW, INT32_MAX)
                      : go(k_dense_fill<512, 2, false, false, TAB>, 512, index, 0, D.queue + 2, DENSE_FEW, INT32_MAX);
    } else {
        // sums in shared memory: the items whose entries fit a quarter of an SM's shared memory at
        // four CTAs of 256 threads per SM, those that fit a half at two of 512, the rest at one of 1,024
        auto room = [&](int per_sm, int nt) {  // sums that fit beside the index
            const int fixed = 1024 + 512 + nt * (int)(sizeof(int64_t) + sizeof(val_t) + sizeof(int32_t)) + nt / 4 +
                          nt / 32 * DENSE_STAGE * (int)sizeof(uint16_t);
            return (std::min(227 * 1024, 228 * 1024 / per_sm) - fixed - index) / (int)sizeof(val_t) & ~31;
        };
        const int v4 = room(4, 256), v2 = room(2, 512), v1 = room(1, 1024);
        if (v4 < 32) return cudaErrorInvalidValue;
        const int fs = (int)sizeof(val_t);
        e = replay ? go(k_dense_fill<256, 4, true, true, TAB>, 256, index + v4 * fs, v4, D.queue + 1, 0, v4)
                   : go(k_dense_fill<256, 4, false, true, TAB>, 256, index + v4 * fs, v4, D.queue + 1, 0, v4);
        if (e != cudaSuccess) return e;
        if (D.W <= v4) return e;  // a slice has at most W entries
        e = replay ? go(k_dense_fill<512, 2, true, true, TAB>, 512, index + v2 * fs, v2, D.queue + 2, v4, v2)
                   : go(k_dense_fill<512, 2, false, true, TAB>, 512, index + v2 * fs, v2, D.queue + 2, v4, v2);
        if (e != cudaSuccess) return e;
        if (D.W <= v2) return e;
        return replay ? go(k_dense_fill<1024, 1, true, true, TAB>, 1024, index + v1 * fs, v1, D.queue + 3, v2, INT32_MAX)
                      : go(k_dense_fill<1024, 1, false, true, TAB>, 1024, index + v1 * fs, v1, D.queue + 3, v2, INT32_MAX);
    }
}

cudaError_t launch_dense_fill(const DevCSR &A, const DevCSR &B, const DenseArgs &D, const int64_t *c_rp,
                              int32_t *c_col, val_t *c_val, int64_t *err, cudaStream_t st, bool replay,
                              const int64_t *gate) {
    return dense_tabled(D) ? launch_fill<true>(A, B, D, c_rp, c_col, c_val, err, st, replay, gate)
                           : launch_fill<false>(A, B, D, c_rp, c_col, c_val, err, st, replay, gate);
}

}  // namespace spg
