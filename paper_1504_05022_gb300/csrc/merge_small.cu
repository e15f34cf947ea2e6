// Stage 3, bin group 5, for the rows whose products fit the registers of a CTA (u_i up to 16 per
// thread): the result of the merge method without its batches.
//
// The CTA loads the columns of all products of the row once, 16 per thread, and keeps them in
// registers while they find their places: a bitmap of the occupied 32-column words of
// B (one bit per word) and its rank directory number the words; a bitmap per occupied word and
// the ranks over those give every column its position in the row.  Then the values are read and
// added into one sum per column.  Fifteen barriers in all, and no capacity to outgrow before the
// size is known: a row longer than its home is listed as overflowed with its exact size (its
// length in the work-item table) before any value is read, and later rounds pass it on until
// their capacity fits.
//
// The batched kernel (merge_bm.cu) searches each product's B row in a table, buffers the products
// whose columns are new and merges them by rank, with a barrier per batch and a dozen per merge;
// at 230 KB of shared memory per CTA it leaves 16 warps on an SM.  Here a CTA needs 8 bytes per
// product and per 1,024 columns of B: 28 to 32 warps per SM up to 1.2 million columns (3.5 million for
// the CTAs of 512 threads), 16 to 24 at the 4,194,304 that the index takes.  Shared-memory latency
// and instruction issue bound it.
//
// Measured (kernel time of all bin-37 merge launches, one GB300, before -> after): R-MAT 2^20 x 8, its
// 180 k rows of 513..8,191 products, 23.3 -> 9.2 ms; R-MAT 2^16 x 16 1.68 -> 1.19 ms; R-MAT 30,011 x 8
// in single precision under the hybrid policy (five rounds) 0.89 -> 0.70 ms.  50,000 rows of 576 and of 2,025
// products, the whole product by the upper-bound policy: B of 200,000 columns 3.92 -> 1.34 and 5.85 ->
// 2.04 ms, of 4,194,304 4.45 -> 2.23 and 6.53 -> 3.10.  The line lies at 8,192 products because 512
// threads of 16 are the most that share an SM twice.
#include "internal.h"
#include "common.cuh"
#include "dynamic_smem.h"

namespace spg {

constexpr int MS_PPT = 16;  // products per thread

// 2 A entries per thread make the window, so a row has at most 2 NT of them.
template <int NT>
struct MsWin {
    int64_t base[2 * NT];        // place in B of the part's first entry, minus start
    int64_t scan[NT / 32 + 1];
    val_t av[2 * NT];
    int32_t start[2 * NT + 32];  // first product of the part; INT_MAX past the last part
};

// Words of the level-1 bitmap (a bit per 32 columns), and the shared memory of a CTA: per
// product a word and its rank, later its sum; then the level-1 bitmap and its ranks.
static int ms_words(int64_t ncols) { return (int)((ncols + 1023) / 1024); }
static int ms_smem(int nt, int64_t ncols) {
    return nt * MS_PPT * 8 + 2 * 4 * ((ms_words(ncols) + 4) & ~3) + 64;
}

template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_merge_small(StageArgs a, MergeItems it, MergeLaunch L, int nw1) {
    extern __shared__ __align__(16) unsigned char ms_smem_raw[];
    __shared__ MsWin<NT> win;
    __shared__ int32_t scan32[NT / 32 + 1];
    constexpr int NW = NT / 32, UMAX = NT * MS_PPT;
    uint32_t *Wb = reinterpret_cast<uint32_t *>(ms_smem_raw);  // bits of the occupied words
    int32_t *Wr = reinterpret_cast<int32_t *>(Wb + UMAX);      // and columns before them
    val_t *V = reinterpret_cast<val_t *>(ms_smem_raw);         // then the sums, in their place
    uint32_t *T = reinterpret_cast<uint32_t *>(Wr + UMAX);
    int32_t *Tr = reinterpret_cast<int32_t *>(T + ((nw1 + 4) & ~3));
    static_assert(sizeof(val_t) <= 8, "the sums take the words' place");

    const int64_t w = blockIdx.x;
    const int j = L.work ? L.work[w] : (int)(L.work_base + w);
    const int row = it.row[j];
    const int64_t a0 = a.A.rp[row];
    const int nA = (int)min(a.A.rp[row + 1] - a0, (int64_t)INT_MAX);
    const int64_t uu = L.u[row];
    if (merge_small_threads(uu, nA, L.small_u) != NT || !merge_fresh(it, j)) return;
    // where this launch writes the item, as in k_merge_bm
    int32_t *dst_col = it.home_col[j];
    val_t *dst_val = it.home_val[j];
    int64_t dst_cap = it.home_cap[j];
    int cap = L.cap;
    if (dst_cap < cap) {
        if (L.pool_col != nullptr) {
            dst_col = L.pool_col + w * L.pool_cap;
            dst_val = L.pool_val + w * L.pool_cap;
            dst_cap = L.pool_cap;
        } else {
            cap = (int)dst_cap;
        }
    }
    auto overflow = [&](int nnz) {
        if (threadIdx.x == 0) {
            it.len[j] = nnz;
            L.ovf_list[atomicAdd(L.ovf_count, 1)] = j;
        }
    };
    const int known = it.len[j];  // its size, when an earlier round computed it
    if (known > cap) {
        overflow(known);
        return;
    }
    for (int t = threadIdx.x; t < nw1; t += NT) T[t] = 0u;

    // ---- the row's parts ----
    int len[2] = {0, 0};
    int64_t bs[2];
    val_t av2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int e = 2 * (int)threadIdx.x + h;
        if (e < nA) {
            const int32_t k = a.A.col[a0 + e];
            bs[h] = a.B.rp[k];
            len[h] = (int)(a.B.rp[k + 1] - bs[h]);
            av2[h] = a.A.val[a0 + e];
        }
    }
    int64_t tot;
    const int64_t ex = block_exclusive_scan<NT, int64_t, false>(
        ((int64_t)((len[0] > 0) + (len[1] > 0)) << 32) + len[0] + len[1], win.scan, tot);
    const int np = (int)(tot >> 32), U = (int)(tot & 0xffffffff);
    {
        int q = (int)(ex >> 32), st = (int)(ex & 0xffffffff);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (len[h] > 0) {
                win.start[q] = st;
                win.base[q] = bs[h] - st;
                win.av[q] = av2[h];
                ++q;
                st += len[h];
            }
        }
    }
    for (int t = np + (int)threadIdx.x; t < 2 * NT + 32; t += NT) win.start[t] = INT_MAX;
    __syncthreads();
    if (U > UMAX) {  // cannot happen: U = u_i
        if (threadIdx.x == 0) atomicExch((unsigned long long *)L.err, 1ull);
        return;
    }

    // ---- the products: warp w's contiguous groups of 32, one per register slot ----
    const int lane = lane_id(), wid = warp_id();
    const int G = (U + 31) >> 5;
    const int g0 = G * wid / NW, g1 = G * (wid + 1) / NW;
    int t0 = 0;  // the part of product 32 g0
    for (int lo = 0, hi = np - 1; lo < hi;) {
        const int mid = (lo + hi + 1) >> 1;
        if (win.start[mid] <= (g0 << 5)) lo = mid; else hi = mid - 1;
        t0 = lo;
    }
    const unsigned le = (2u << lane) - 1u;
    // slot k's part (the next group's in t) and place in B; false without a product
    auto product = [&](int k, int &t, int &pt, int64_t &p) {
        const int q = (g0 + k) << 5;
        const bool on = g0 + k < g1;
        const unsigned d = (unsigned)(win.start[t + 1 + lane] - q);
        const unsigned m = __reduce_or_sync(SPG_FULL, (on && d < 32u) ? 1u << d : 0u);
        pt = t + __popc(m & le);
        t += __popc(m);
        p = win.base[pt] + (q + lane);
        return on && q + lane < U;
    };
    int32_t c[MS_PPT];  // column, -1: none
    bool bad = false;
    {
        int t = t0;
#pragma unroll
        for (int k = 0; k < MS_PPT; ++k) {
            int pt;
            int64_t p;
            c[k] = product(k, t, pt, p) ? __ldg(a.B.col + p) : -1;
        }
    }
    // ---- level 1: the occupied words ----
#pragma unroll
    for (int k = 0; k < MS_PPT; ++k) {
        if (c[k] == -1) continue;
        if ((unsigned)c[k] >= (unsigned)a.B.ncols) {  // bad input
            bad = true;
            c[k] = -1;
            continue;
        }
        atomicOr(&T[c[k] >> 10], 1u << ((c[k] >> 5) & 31));
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0) atomicExch((unsigned long long *)L.err, 5ull);
        return;
    }
    const int nocc = bitmap_rank<NT>(T, Tr, nw1, scan32);
    for (int t = threadIdx.x; t < nocc; t += NT) Wb[t] = 0u;
    __syncthreads();
    // ---- level 2: the columns of every occupied word ----
    int pos[MS_PPT];
#pragma unroll
    for (int k = 0; k < MS_PPT; ++k) {
        if (c[k] < 0) continue;
        pos[k] = Tr[c[k] >> 10] + __popc(T[c[k] >> 10] & ((1u << ((c[k] >> 5) & 31)) - 1u));
        if (!SPG_IN(pos[k] < nocc, 114)) {
            c[k] = -1;
            continue;
        }
        atomicOr(&Wb[pos[k]], 1u << (c[k] & 31));
    }
    __syncthreads();
    const int nnz = bitmap_rank<NT>(Wb, Wr, nocc, scan32);
    if (nnz > cap) {
        overflow(nnz);
        return;
    }
#pragma unroll
    for (int k = 0; k < MS_PPT; ++k)
        if (c[k] >= 0) pos[k] = Wr[pos[k]] + __popc(Wb[pos[k]] & ((1u << (c[k] & 31)) - 1u));
    __syncthreads();  // the words have been read: their space holds the sums
    for (int t = threadIdx.x; t < nnz; t += NT) V[t] = val_t(0);
    __syncthreads();
    {
        int t = t0;
        constexpr int UN = 4;
#pragma unroll
        for (int k0 = 0; k0 < MS_PPT; k0 += UN) {
            val_t v[UN], av[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                int pt;
                int64_t p;
                if (product(k0 + u, t, pt, p)) {
                    v[u] = __ldg(a.B.val + p);
                    av[u] = win.av[pt];
                }
            }
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                const int k = k0 + u;
                if (c[k] < 0 || !SPG_IN(pos[k] < nnz, 117)) continue;
                atomicAdd(&V[pos[k]], av[u] * v[u]);
                dst_col[pos[k]] = c[k];  // the same column from every product of the position
            }
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nnz; t += NT) dst_val[t] = V[t];
    if (threadIdx.x == 0) {
        it.home_col[j] = dst_col;
        it.home_val[j] = dst_val;
        it.home_cap[j] = dst_cap;
        it.len[j] = nnz;
    }
}

template <int NT, int MINB>
static cudaError_t launch_ms(const StageArgs &a, const MergeItems &s, const MergeLaunch &L, cudaStream_t st) {
    auto kern = k_merge_small<NT, MINB>;
    const int smem = ms_smem(NT, a.B.ncols);
    cudaError_t e = allow_dynamic_smem((const void *)kern, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)L.nwork, NT, smem, st>>>(a, s, L, ms_words(a.B.ncols));
    return cudaGetLastError();
}

cudaError_t launch_merge_small(const StageArgs &a, const MergeItems &s, const MergeLaunch &L, cudaStream_t st) {
    if (L.nwork <= 0 || L.small_u <= 0) return cudaSuccess;
    cudaError_t e = launch_ms<128, 7>(a, s, L, st);
    if (e == cudaSuccess) e = launch_ms<256, 4>(a, s, L, st);
    if (e == cudaSuccess) e = launch_ms<512, 2>(a, s, L, st);
    return e;
}

}  // namespace spg
