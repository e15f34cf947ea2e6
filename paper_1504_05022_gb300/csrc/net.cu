// Stage 3, bin group 3 (u_i = 2..32) and its counting pass, for launches of many rows: a thread per
// row, and the expand-sort-compress of esc.cu with a sorting network in registers.
//
// The thread expands its row's products into its own column of shared memory (slot-major, so a
// warp touches consecutive words), loads the keys -- column and slot in one word, as in esc.cu --
// into registers, sorts them with Batcher's odd-even merge network (19, 63 or 191
// compare-exchanges for 8, 16 or 32 keys, two instructions each, no data moved between threads)
// and sums equal columns in order.  The groups of esc.cu take 820 instructions for two rows of 27
// products; they stay for launches of few rows, where a thread per row would leave the SMs idle.
// Bound by the dependent gathers (A's column, B's row, its entries) and instruction issue.
//
// Measured (kernel time, double, one GB300; esc.cu -> here): A*P of the 7-point operator on 80^3 (512,000
// rows of up to 7 products) 82 -> 38 us, its count 47 -> 18 us; A*P of the 27-point operator on 64^3
// (262,144 rows of up to 27) 134 -> 104 us.
#include "internal.h"
#include "common.cuh"

namespace spg {

constexpr int NET_NT = 64;

// Batcher's odd-even merge sort, ascending.  The steps are template arguments, so that every
// loop unrolls and the keys stay in registers.
template <int P, int D, int N, typename K>
SPG_DEV void net_step(K (&x)[N]) {
#pragma unroll
    for (int j = D % P; j <= N - 1 - D; j += 2 * D) {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            if (i + j + D < N && (i + j) / (2 * P) == (i + j + D) / (2 * P)) {
                const K a = x[i + j], b = x[i + j + D];
                x[i + j] = a < b ? a : b;
                x[i + j + D] = a < b ? b : a;
            }
        }
    }
    if constexpr (D > 1) net_step<P, D / 2, N, K>(x);
}
template <int N, typename K, int P = 1>
SPG_DEV void net_sort(K (&x)[N]) {
    net_step<P, P, N, K>(x);
    if constexpr (2 * P < N) net_sort<N, K, 2 * P>(x);
}

// The threads stride over the rows (one pass when the grid covers them).  COUNT: nnz(c_i) only.
template <int N, typename K, bool COUNT>
__global__ void __launch_bounds__(NET_NT)
k_net(StageArgs a, RowSet R) {
    constexpr int LB = COUNT ? 0 : (sizeof(K) == 8 ? 32 : N == 8 ? 3 : N == 16 ? 4 : 5);
    static_assert(COUNT || sizeof(K) == 8 || (1 << LB) == N, "N is a power of two up to 32");
    constexpr K PAD = ~K(0);
    __shared__ K sk[N * NET_NT];
    __shared__ val_t sv[COUNT ? 1 : N * NET_NT];
    if (!COUNT && gated(a.gate)) return;
    const int32_t *rows;
    int64_t nrows;
    rowset_range(R, rows, nrows);
    for (int64_t t = (int64_t)blockIdx.x * NET_NT + threadIdx.x; t < nrows; t += (int64_t)gridDim.x * NET_NT) {
        const int row = rows[t];
        const int64_t a0 = a.A.rp[row], a1 = a.A.rp[row + 1];
        int n = 0;
        auto put = [&](int32_t c, val_t v) {
            if (n >= N) return;  // cannot happen: n <= u_i
            sk[n * NET_NT + threadIdx.x] = COUNT ? (K)(uint32_t)c : ((K)(uint32_t)c << (LB & (8 * sizeof(K) - 1))) | (K)n;
            if (!COUNT) sv[n * NET_NT + threadIdx.x] = v;
            ++n;
        };
        constexpr int UN = 4;  // entries of A, then of a B row, whose loads are in flight together
        for (int64_t p = a0; p < a1; p += UN) {
            int64_t bs[UN];
            int32_t len[UN];
            val_t av[UN];
            bool single = true;
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                len[u] = 0;
                if (p + u < a1) {
                    const int32_t j = a.A.col[p + u];
                    bs[u] = a.B.rp[j];
                    len[u] = (int32_t)(a.B.rp[j + 1] - bs[u]);
                    if (!COUNT) av[u] = a.A.val[p + u];
                }
                single = single && len[u] <= 1;
            }
            if (single) {
                int32_t c[UN];
                val_t v[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (len[u] > 0) {
                        c[u] = __ldg(a.B.col + bs[u]);
                        if (!COUNT) v[u] = __ldg(a.B.val + bs[u]);
                    }
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (len[u] > 0) put(c[u], COUNT ? val_t(0) : av[u] * v[u]);
                continue;
            }
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                for (int q = 0; q < len[u]; q += UN) {
                    int32_t c[UN];
                    val_t v[UN];
#pragma unroll
                    for (int w = 0; w < UN; ++w)
                        if (q + w < len[u]) {
                            c[w] = __ldg(a.B.col + bs[u] + q + w);
                            if (!COUNT) v[w] = __ldg(a.B.val + bs[u] + q + w);
                        }
#pragma unroll
                    for (int w = 0; w < UN; ++w)
                        if (q + w < len[u]) put(c[w], COUNT ? val_t(0) : av[u] * v[w]);
                }
            }
        }
        K key[N];
#pragma unroll
        for (int e = 0; e < N; ++e) key[e] = e < n ? sk[e * NET_NT + threadIdx.x] : PAD;
        net_sort<N, K>(key);
        if constexpr (COUNT) {
            int cnt = 0;
#pragma unroll
            for (int e = 0; e < N; ++e) cnt += (key[e] != PAD && (e == 0 || key[e] != key[e > 0 ? e - 1 : 0])) ? 1 : 0;
            a.nnzc[row] = cnt;
        } else {
            const int64_t o = a.ctil_rp[row];
            int cnt = 0;
            uint32_t col = 0;
            val_t sum = val_t(0);
            auto out = [&] {
                if (SPG_IN(o + cnt < a.ctil_rp[row + 1], 115)) {  // the row's space in C~ (or C)
                    a.ctil_col[o + cnt] = (int32_t)col;
                    a.ctil_val[o + cnt] = sum;
                }
                ++cnt;
            };
#pragma unroll
            for (int e = 0; e < N; ++e) {
                if (e < n) {
                    const uint32_t c = (uint32_t)(key[e] >> (LB & (8 * sizeof(K) - 1)));
                    const val_t v = sv[(int)(key[e] & (K)(N - 1)) * NET_NT + threadIdx.x];
                    if (e > 0 && c == col) {
                        sum += v;
                    } else {
                        if (e > 0) out();
                        col = c;
                        sum = v;
                    }
                }
            }
            if (n > 0) out();
            a.nnzc[row] = cnt;
        }
    }
}

template <int N, typename K, bool COUNT>
static cudaError_t net_go(const StageArgs &a, const RowSet &R, cudaStream_t st) {
    const int64_t need = (R.n + NET_NT - 1) / NET_NT;
    auto kern = k_net<N, K, COUNT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    const int64_t grid = R.dev_lo ? persistent_blocks((const void *)kern, NET_NT, 0, need) : need;
    if (grid <= 0) return cudaErrorInvalidValue;
    kern<<<(unsigned)grid, NET_NT, 0, st>>>(a, R);
    return cudaGetLastError();
}

template <int N>
static cudaError_t net_pick(const StageArgs &a, const RowSet &R, bool count_only, cudaStream_t st) {
    if (count_only) return net_go<N, uint32_t, true>(a, R, st);
    // the packed key must hold column and slot, and stay below the pad
    if (a.B.ncols * N < (int64_t(1) << 32)) return net_go<N, uint32_t, false>(a, R, st);
    return net_go<N, uint64_t, false>(a, R, st);
}

cudaError_t launch_net_set(const StageArgs &a, const RowSet &R, int max_u, bool count_only, cudaStream_t st) {
    if (R.n <= 0) return cudaSuccess;
    if (max_u <= 8) return net_pick<8>(a, R, count_only, st);
    if (max_u <= 16) return net_pick<16>(a, R, count_only, st);
    return max_u <= 32 ? net_pick<32>(a, R, count_only, st) : cudaErrorInvalidValue;
}

}  // namespace spg
