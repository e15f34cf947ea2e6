// Stage 3, bin groups 3 and 4 (u_i = 2..512): the expand-sort-compress method of Section 4.1
// with a bitonic network, on packed keys.
//
// A group of G lanes takes a row of at most N = G*E products.  It expands the products into
// shared memory, sorts them by column and sums equal columns.  The network moves one word per
// product: the column and the product's number among the N, packed into 32 bits when B has
// fewer than 2^(32 - log2 N) columns and into 64 bits otherwise.  The values stay where they
// were expanded and are fetched once, by that number, after the sort.  (A network that carries
// the value along needs three shuffles per step instead of one; A*A of an Erdos-Renyi matrix
// with 100,003 rows of 16 spent 0.76 ms in it.)  Element i = lane*E + e, so compare-exchange
// distances below E stay inside a thread and the others are one shuffle.
//
// A product's part is found without a search: the starts of the next G
// parts (non-empty B rows) that fall into the G products at hand become a bit mask, and a
// lane's part is the number of mask bits at or below it.  Rows of at most 8, 16 and 32
// products take groups of 8, 8 and 16 lanes, so that a warp has four or two rows' dependent
// loads in flight; longer ones take a warp.  Latency and issue slots bound it.
//
// Measured (one GB300, kernel time, double; before -> after): A*A of that Erdos-Renyi matrix (25.6 M
// products, bin 35) 764 -> 265 us; A*P of the 27-point operator on 64^3 (6.9 M products, bins
// 2..27), the heap kernel with one thread per row 262 us -> 152 us, and a values-only replay of
// R*(A*P) 234 -> 157 us; A*A of a 64 x 64 5-point Laplacian, heap 63 us -> 13 us.  The heap kernel
// runs only where opts.heap_max_u asks for it.
#include "internal.h"
#include "common.cuh"

namespace spg {

constexpr int ESC_NT = 128;
// Launches of at least so many rows of u <= 32 take a thread per row (net.cu): below, there are fewer
// warps than SMs can hold and a row's serial loads show (3,600 rows of 25 products: 11 us against
// 7 here; 262,144 rows of 27: 104 us against 134 here; 512,000 rows of 7: 38 against 82).
constexpr int64_t ESC_NET_ROWS = 16384;
// And only where A's rows average at most so many entries: in longer ones most entries select empty
// rows of B, and a thread looks at them one after another (200,000 rows of 512 entries and 16 products,
// precise: 5.8 ms against 2.3 here, 5.7 by the heap and a warp per row before them).
constexpr int64_t ESC_NET_ENTRIES = 32;

template <int G, typename T>
SPG_DEV T group_inclusive_scan(unsigned gm, int gl, T v) {
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        const T n = __shfl_up_sync(gm, v, d, G);
        if (gl >= d) v += n;
    }
    return v;
}

template <int G>
SPG_DEV unsigned group_or(unsigned gm, unsigned v) {
    if constexpr (G == 32) {
        return __reduce_or_sync(gm, v);
    } else {
#pragma unroll
        for (int d = 1; d < G; d <<= 1) v |= __shfl_xor_sync(gm, v, d, G);
        return v;
    }
}

template <int G, int E, typename K, bool COUNT>
struct EscSmem {
    static constexpr int N = G * E;
    K key[N];
    val_t val[COUNT ? 1 : N];
    int64_t base[G];        // place in B of the part's first entry, minus start
    val_t av[COUNT ? 1 : G];
    int32_t start[2 * G];   // first product of the part; INT_MAX past the last part
};

// The groups of a warp lie 4 G bytes apart modulo the 128 bytes of the banks, so that their
// accesses do not meet in the same banks.
template <int G, int E, typename K, bool COUNT>
struct EscGroup : EscSmem<G, E, K, COUNT> {
    static constexpr int RAW = (int)sizeof(EscSmem<G, E, K, COUNT>);
    static constexpr int GAP = ((4 * G - RAW) % 128 + 128) % 128;
    unsigned char gap[GAP == 0 ? 128 : GAP];
};

// COUNT: the counting pass of the precise method (Section 3.1): the same expansion and sort
// on the columns alone, and nnz(c_i) = the number of distinct columns, written to a.nnzc.
// The groups stride over the rows (one pass when the grid covers them).
template <int G, int E, typename K, bool COUNT>
__global__ void __launch_bounds__(ESC_NT)
k_esc(StageArgs a, RowSet R) {
    constexpr int N = G * E, GROUPS = ESC_NT / G;
    // bits of a product's number below its column
    constexpr int LB = COUNT ? 0 : (sizeof(K) == 8 ? 32 : (N == 8 ? 3 : N == 16 ? 4 : N == 32 ? 5 : N == 64 ? 6 : N == 128 ? 7 : N == 256 ? 8 : 9));
    static_assert(N <= 512 && (COUNT || sizeof(K) == 8 || (1 << LB) == N), "N is a power of two");
    constexpr K PAD = ~K(0);
    constexpr int U = E < 4 ? E : 4;  // groups of G products in flight
    using Smem = EscGroup<G, E, K, COUNT>;
    __shared__ Smem smem[GROUPS];
    if (!COUNT && gated(a.gate)) return;
    const int32_t *rows;
    int64_t nrows;
    rowset_range(R, rows, nrows);
    const int gl = threadIdx.x & (G - 1);
    const unsigned gm = G == 32 ? SPG_FULL : ((1u << (G & 31)) - 1u) << (lane_id() & ~(G - 1));
    const unsigned le = (2u << gl) - 1u;
    Smem &S = smem[threadIdx.x / G];
    for (int64_t t = (int64_t)blockIdx.x * GROUPS + threadIdx.x / G; t < nrows; t += (int64_t)gridDim.x * GROUPS) {
        const int row = rows[t];
        // ---- expand ----
        int filled = 0;
        const int64_t a0 = a.A.rp[row], a1 = a.A.rp[row + 1];
        for (int64_t ch = a0; ch < a1; ch += G) {
            const int64_t p = ch + gl;
            int32_t len = 0;
            int64_t bs = 0;
            val_t av = val_t(0);
            if (p < a1) {
                const int32_t j = a.A.col[p];
                bs = a.B.rp[j];
                len = (int32_t)(a.B.rp[j + 1] - bs);
                if (!COUNT) av = a.A.val[p];
            }
            const int32_t inc = group_inclusive_scan<G>(gm, gl, len);
            const int total = __shfl_sync(gm, inc, G - 1, G);
            const unsigned nz = __ballot_sync(gm, len > 0) >> (lane_id() & ~(G - 1));
            const int np = __popc(G == 32 ? nz : nz & ((1u << (G & 31)) - 1u));
            if (len > 0) {
                const int q = __popc(nz & (le >> 1));
                S.start[q] = inc - len;
                S.base[q] = bs - (inc - len);
                if (!COUNT) S.av[q] = av;
            }
            if (gl >= np) S.start[gl] = INT_MAX;
            S.start[G + gl] = INT_MAX;
            __syncwarp(gm);
            int part = 0;
            for (int q0 = 0; q0 < total; q0 += U * G) {
                int64_t pos[U];
                int pt[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int q = q0 + u * G;
                    const unsigned d = (unsigned)(S.start[part + 1 + gl] - q);
                    const unsigned m = group_or<G>(gm, (q < total && d < (unsigned)G) ? 1u << d : 0u);
                    pt[u] = part + __popc(m & le);
                    part += __popc(m);
                    pos[u] = S.base[pt[u]] + (q + gl);
                }
                int32_t c[U];
                val_t v[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (q0 + u * G + gl < total) c[u] = __ldg(a.B.col + pos[u]);
                if (!COUNT) {
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (q0 + u * G + gl < total) v[u] = __ldg(a.B.val + pos[u]);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int dst = filled + q0 + u * G + gl;
                    if (q0 + u * G + gl < total && dst < N) {
                        S.key[dst] = COUNT ? (K)(uint32_t)c[u] : ((K)(uint32_t)c[u] << (LB & (8 * sizeof(K) - 1))) | (K)dst;
                        if (!COUNT) S.val[dst] = S.av[pt[u]] * v[u];
                    }
                }
            }
            filled += total;
            __syncwarp(gm);  // the part table is free again, and the products are visible
        }
        K key[E];
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] = e * G + gl < filled ? S.key[e * G + gl] : PAD;

        // ---- bitonic sort, ascending on i = gl*E + e ----
#pragma unroll
        for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                if (j >= E) {
                    const bool lower = (gl & (j / E)) == 0;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const K pk = __shfl_xor_sync(gm, key[e], j / E, G);
                        const bool up = ((gl * E + e) & k) == 0;
                        key[e] = (lower == up) ? (pk < key[e] ? pk : key[e]) : (pk > key[e] ? pk : key[e]);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if ((e & j) == 0) {
                            const bool up = ((gl * E + e) & k) == 0;
                            const K x = key[e], y = key[e | j];
                            const K mn = x < y ? x : y, mx = x < y ? y : x;
                            key[e] = up ? mn : mx;
                            key[e | j] = up ? mx : mn;
                        }
                    }
                }
            }
        }

        if constexpr (COUNT) {
            // distinct columns: entries that differ from their predecessor (the pad excluded)
            const K before = __shfl_up_sync(gm, key[E - 1], 1, G);
            int cnt = 0;
#pragma unroll
            for (int e = 0; e < E; ++e)
                cnt += (key[e] != PAD && (e > 0 ? key[e] != key[e > 0 ? e - 1 : 0] : (gl == 0 || key[e] != before))) ? 1 : 0;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) cnt += __shfl_xor_sync(gm, cnt, d, G);
            if (gl == 0) a.nnzc[row] = cnt;
            __syncwarp(gm);  // the next row's expansion reuses the keys
        } else {
            // ---- compress: segmented sums over runs of equal columns ----
            uint32_t col[E];
            val_t val[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                // the pad's column (all ones) is beyond every real one
                col[e] = key[e] == PAD ? ~0u : (uint32_t)(key[e] >> (LB & (8 * sizeof(K) - 1)));
                val[e] = key[e] == PAD ? val_t(0) : S.val[(int)(key[e] & (K)(N - 1))];
            }
#pragma unroll
            for (int e = 1; e < E; ++e)
                if (col[e] == col[e - 1]) val[e] += val[e - 1];
            const uint32_t first = col[0], last = col[E - 1];
            const uint32_t prev_last = __shfl_up_sync(gm, last, 1, G);
            const bool cont = gl > 0 && prev_last == first && first != ~0u;
            if (__any_sync(gm, cont)) {
                // R = running sum of the run that ends this lane; f = a run starts in this lane
                val_t Rs = val[E - 1];
                bool f = !((first == last) && cont);
#pragma unroll
                for (int d = 1; d < G; d <<= 1) {
                    const val_t Rn = __shfl_up_sync(gm, Rs, d, G);
                    const bool fn = __shfl_up_sync(gm, (int)f, d, G) != 0;
                    if (gl >= d && !f) {
                        Rs += Rn;
                        f = fn;
                    }
                }
                const val_t carry = __shfl_up_sync(gm, Rs, 1, G);
                if (cont) {
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (col[e] == first) val[e] += carry;
                }
            }
            uint32_t next_first = __shfl_down_sync(gm, first, 1, G);
            if (gl == G - 1) next_first = ~0u;  // nothing follows; the pad never ends a run
            int cnt = 0;
            unsigned tails = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t nk = (e + 1 < E) ? col[e + 1 < E ? e + 1 : 0] : next_first;
                if (col[e] != ~0u && col[e] != nk) {
                    tails |= 1u << e;
                    ++cnt;
                }
            }
            const int inc = group_inclusive_scan<G>(gm, gl, cnt);
            const int total = __shfl_sync(gm, inc, G - 1, G);
            const int64_t o = a.ctil_rp[row];
            const bool fits = SPG_IN(o + total <= a.ctil_rp[row + 1], 102);  // the row's space in C~ (or C)
            // through shared memory, so that the row leaves in one contiguous run
            __syncwarp(gm);
            int q = inc - cnt;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (tails & (1u << e)) {
                    S.key[q] = (K)col[e];
                    S.val[q] = val[e];
                    ++q;
                }
            }
            __syncwarp(gm);
            if (fits) {
                for (int r = gl; r < total; r += G) {
                    a.ctil_col[o + r] = (int32_t)S.key[r];
                    a.ctil_val[o + r] = S.val[r];
                }
            }
            if (gl == 0) a.nnzc[row] = total;
            __syncwarp(gm);  // the next row's expansion reuses the arrays
        }
    }
}

template <int G, int E, typename K, bool COUNT>
static cudaError_t esc_go(const StageArgs &a, const RowSet &R, cudaStream_t st) {
    constexpr int GROUPS = ESC_NT / G;
    const int64_t need = (R.n + GROUPS - 1) / GROUPS;
    const int64_t grid = R.dev_lo ? persistent_blocks((const void *)k_esc<G, E, K, COUNT>, ESC_NT, 0, need) : need;
    if (grid <= 0) return cudaErrorInvalidValue;
    k_esc<G, E, K, COUNT><<<(unsigned)grid, ESC_NT, 0, st>>>(a, R);
    return cudaGetLastError();
}

// The counting pass sorts plain columns; else the packed key must hold column and number, and
// stay below the pad.
template <int G, int E>
static cudaError_t esc_pick(const StageArgs &a, const RowSet &R, bool count_only, cudaStream_t st) {
    if (count_only) return esc_go<G, E, uint32_t, true>(a, R, st);
    if (a.B.ncols * (G * E) < (int64_t(1) << 32)) return esc_go<G, E, uint32_t, false>(a, R, st);
    return esc_go<G, E, uint64_t, false>(a, R, st);
}

cudaError_t launch_esc_set(const StageArgs &a, const RowSet &R, int max_u, bool count_only, cudaStream_t st) {
    if (R.n <= 0) return cudaSuccess;
    if (max_u <= 32 && R.n >= ESC_NET_ROWS && a.A.nnz <= ESC_NET_ENTRIES * a.A.nrows) return launch_net_set(a, R, max_u, count_only, st);
    if (max_u <= 8) return esc_pick<8, 1>(a, R, count_only, st);
    if (max_u <= 16) return esc_pick<8, 2>(a, R, count_only, st);
    if (max_u <= 32) return esc_pick<16, 2>(a, R, count_only, st);
    if (max_u <= 64) return esc_pick<32, 2>(a, R, count_only, st);
    if (max_u <= 128) return esc_pick<32, 4>(a, R, count_only, st);
    if (max_u <= 256) return esc_pick<32, 8>(a, R, count_only, st);
    if (max_u <= 512) return esc_pick<32, 16>(a, R, count_only, st);
    return cudaErrorInvalidValue;
}

}  // namespace spg
