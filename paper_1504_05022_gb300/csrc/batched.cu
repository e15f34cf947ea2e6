// Batched products: many independent C_i = A_i * B_i computed as one product of
// block-diagonal matrices, diag(A_1..A_n) * diag(B_1..B_n) = diag(A_1 B_1 .. A_n B_n).
// The concatenation gives A_i's columns an offset of sum_{j<i} k_j, so they
// select B_i's rows; B_i's columns keep their own numbering (0 .. n_i - 1): a
// row of C_i only ever combines rows of B_i, so no row mixes columns of two
// pairs, and the concatenated C holds every C_i with its own column numbers.
// Every stage of the framework runs once over the rows of all pairs (one launch
// per bin for the whole batch).  The split step only rebases each C_i's row
// pointers; its columns and values are views into the concatenated C.
#include "internal.h"
#include "common.cuh"

namespace spg {

SPG_DEV int find_pair(const int64_t *off, int64_t npairs, int64_t x) {
    // largest i with off[i] <= x
    int64_t lo = 0, hi = npairs - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid - 1;
    }
    return (int)lo;
}

SPG_DEV int64_t rp_at(const void *rp, int bits, int64_t i) {
    return bits == 64 ? static_cast<const int64_t *>(rp)[i] : (int64_t) static_cast<const int32_t *>(rp)[i];
}

// Row pointers of the concatenated A (rows of all pairs) and B.
__global__ void k_concat_rp(const PairDesc *d, int64_t npairs, const int64_t *moff, const int64_t *koff, int64_t M,
                            int64_t K, int64_t annz, int64_t bnnz, int64_t *a_rp, int64_t *b_rp) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < M) {
        const int i = find_pair(moff, npairs, r);
        a_rp[r] = d[i].annz_off + rp_at(d[i].a_rp, d[i].a_bits, r - d[i].moff);
    } else if (r == M) {
        a_rp[M] = annz;
    }
    if (r < K) {
        const int i = find_pair(koff, npairs, r);
        b_rp[r] = d[i].bnnz_off + rp_at(d[i].b_rp, d[i].b_bits, r - d[i].koff);
    } else if (r == K) {
        b_rp[K] = bnnz;
    }
}

// Entries of the concatenated A (columns shifted into the pair's block) and B.
__global__ void k_concat_entries(const PairDesc *d, int64_t npairs, const int64_t *annz_off, const int64_t *bnnz_off,
                                 int64_t annz, int64_t bnnz, int32_t *a_col, val_t *a_val, int32_t *b_col,
                                 val_t *b_val, int values_only) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < annz) {
        const int i = find_pair(annz_off, npairs, t);
        const int64_t l = t - d[i].annz_off;
        if (!values_only) a_col[t] = d[i].a_col[l] + (int32_t)d[i].koff;
        a_val[t] = d[i].a_val[l];
    }
    if (t < bnnz) {
        const int i = find_pair(bnnz_off, npairs, t);
        const int64_t l = t - d[i].bnnz_off;
        if (!values_only) b_col[t] = d[i].b_col[l];
        b_val[t] = d[i].b_val[l];
    }
}

cudaError_t launch_concat(const PairDesc *d, int64_t npairs, const int64_t *moff, const int64_t *koff,
                          const int64_t *annz_off, const int64_t *bnnz_off, int64_t M, int64_t K, int64_t annz,
                          int64_t bnnz, int64_t *a_rp, int32_t *a_col, val_t *a_val, int64_t *b_rp, int32_t *b_col,
                          val_t *b_val, bool values_only, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    if (!values_only) {
        const int64_t rmax = (M > K ? M : K) + 1;
        k_concat_rp<<<(unsigned)((rmax + 255) / 256), 256, 0, st>>>(d, npairs, moff, koff, M, K, annz, bnnz, a_rp,
                                                                   b_rp);
    }
    const int64_t emax = annz > bnnz ? annz : bnnz;
    if (emax > 0)
        k_concat_entries<<<(unsigned)((emax + 255) / 256), 256, 0, st>>>(d, npairs, annz_off, bnnz_off, annz, bnnz,
                                                                        a_col, a_val, b_col, b_val,
                                                                        values_only ? 1 : 0);
    return cudaGetLastError();
}

// C_i's row pointers, rebased to 0; pair i occupies rp_out[moff_i + i .. moff_i + i + m_i].
__global__ void k_split_out(const PairDesc *d, int64_t npairs, const int64_t *c_rp, int64_t M, int64_t *rp_out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < M + npairs) {
        // entry t of the rebased row-pointer array: pair i holds m_i + 1 entries starting at moff_i + i
        int64_t lo = 0, hi = npairs - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (d[mid].moff + mid <= t) lo = mid; else hi = mid - 1;
        }
        const int i = (int)lo;
        const int64_t r = t - (d[i].moff + i);
        rp_out[t] = c_rp[d[i].moff + r] - c_rp[d[i].moff];
    }
}

cudaError_t launch_split_out(const PairDesc *d, int64_t npairs, const int64_t *c_rp, int64_t M, int64_t *rp_out,
                             cudaStream_t st) {
    const int64_t n = M + npairs;
    if (n <= 0) return cudaSuccess;
    k_split_out<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d, npairs, c_rp, M, rp_out);
    return cudaGetLastError();
}

// Per pair i: prod[i] = sum over the entries a_ik of A_i of nnz(b_k*), the
// products of the pair (Algorithm 2 summed over its rows), and clow[i] = sum
// over the rows of A_i of max_k nnz(b_k*), a lower bound of nnz(C_i) (a row of
// C contains every column of each B row it merges).  A block takes R consecutive rows of
// the concatenation, eight lanes per row, and a warp each long row; columns outside [0, k_i) are
// skipped (they are rejected later when inputs are checked).  prod and clow must be zeroed.
// Latency-bound: about eight blocks per SM over all rows (64 blocks per pair, whatever its size,
// took 0.79 ms for 20 pairs of 252 k rows together).
constexpr int PAIR_NT = 256, PAIR_G = 8, PAIR_ROWS_MAX = 2048;
constexpr int PAIR_LONG = 16 * PAIR_G;

__global__ void __launch_bounds__(PAIR_NT)
k_pair_products(const PairDesc *d, int64_t npairs, const int64_t *moff, int64_t M, int R, unsigned long long *prod,
                unsigned long long *clow) {
    __shared__ int64_t sh[2][PAIR_NT / 32];
    __shared__ int32_t nlong, longs[PAIR_ROWS_MAX];
    const int64_t r0 = (int64_t)blockIdx.x * R, r1 = min(M, r0 + R);
    const int first = find_pair(moff, npairs, r0);
    const bool one = find_pair(moff, npairs, r1 - 1) == first;  // all rows of one pair: summed in the block
    if (threadIdx.x == 0) nlong = 0;
    __syncthreads();
    const int lane = lane_id(), wid = warp_id(), gl = threadIdx.x & (PAIR_G - 1);
    const unsigned gm = ((1u << PAIR_G) - 1u) << (lane & ~(PAIR_G - 1));
    int64_t s = 0, lo = 0;
    // the entries e0, e0 + step, ... of a row of pair i
    auto row_of = [&](const PairDesc &q, int64_t e0, int64_t a1, int step, int64_t &rs, int64_t &rm) {
        rs = rm = 0;
#pragma unroll 4
        for (int64_t e = e0; e < a1; e += step) {
            const int32_t k = q.a_col[e];
            if (k >= 0 && k < q.k) {
                const int64_t len = rp_at(q.b_rp, q.b_bits, k + 1) - rp_at(q.b_rp, q.b_bits, k);
                rs += len;
                rm = len > rm ? len : rm;
            }
        }
    };
    auto add = [&](int i, int64_t rs, int64_t rm) {  // by one thread per row
        if (one) {
            s += rs;
            lo += rm;
        } else if (rs > 0) {
            atomicAdd(prod + i, (unsigned long long)rs);
            atomicAdd(clow + i, (unsigned long long)rm);
        }
    };
    for (int64_t r = r0 + threadIdx.x / PAIR_G; r < r1; r += PAIR_NT / PAIR_G) {
        const int i = one ? first : find_pair(moff, npairs, r);
        const PairDesc &q = d[i];
        const int64_t l = r - moff[i];
        const int64_t a0 = rp_at(q.a_rp, q.a_bits, l), a1 = rp_at(q.a_rp, q.a_bits, l + 1);
        if (a1 - a0 > PAIR_LONG) {
            if (gl == 0) longs[atomicAdd(&nlong, 1)] = (int)(r - r0);
            continue;
        }
        int64_t rs, rm;
        row_of(q, a0 + gl, a1, PAIR_G, rs, rm);
#pragma unroll
        for (int o = PAIR_G / 2; o > 0; o >>= 1) {
            rs += __shfl_xor_sync(gm, rs, o, PAIR_G);
            const int64_t x = __shfl_xor_sync(gm, rm, o, PAIR_G);
            rm = x > rm ? x : rm;
        }
        if (gl == 0) add(i, rs, rm);
    }
    __syncthreads();
    for (int t = wid; t < nlong; t += PAIR_NT / 32) {
        const int64_t r = r0 + longs[t];
        const int i = one ? first : find_pair(moff, npairs, r);
        const PairDesc &q = d[i];
        const int64_t l = r - moff[i];
        int64_t rs, rm;
        row_of(q, rp_at(q.a_rp, q.a_bits, l) + lane, rp_at(q.a_rp, q.a_bits, l + 1), 32, rs, rm);
        rs = warp_reduce_sum(rs);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t x = __shfl_xor_sync(SPG_FULL, rm, o);
            rm = x > rm ? x : rm;
        }
        if (lane == 0) add(i, rs, rm);
    }
    if (!one) return;
    s = warp_reduce_sum(s);
    lo = warp_reduce_sum(lo);
    if (lane == 0) {
        sh[0][wid] = s;
        sh[1][wid] = lo;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        int64_t t = 0;
        for (int w = 0; w < PAIR_NT / 32; ++w) t += sh[threadIdx.x][w];
        if (t) atomicAdd((threadIdx.x == 0 ? prod : clow) + first, (unsigned long long)t);
    }
}

cudaError_t launch_pair_products(const PairDesc *d, int64_t npairs, const int64_t *moff, int64_t M, int64_t *prod,
                                 int64_t *clow, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(prod, 0, sizeof(int64_t) * npairs, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(clow, 0, sizeof(int64_t) * npairs, st);
    if (e != cudaSuccess || M <= 0) return e;
    int64_t R = PAIR_NT / PAIR_G;  // whole passes of the block
    while (R < PAIR_ROWS_MAX && (M + R - 1) / R > 8 * 152) R *= 2;
    k_pair_products<<<(unsigned)((M + R - 1) / R), PAIR_NT, 0, st>>>(
        d, npairs, moff, M, (int)R, reinterpret_cast<unsigned long long *>(prod),
        reinterpret_cast<unsigned long long *>(clow));
    return cudaGetLastError();
}

// out[i] = c_rp[moff_i] (first entry of C_i in the concatenation), out[np] = c_rp[M].
__global__ void k_gather_first(const PairDesc *d, int64_t npairs, const int64_t *c_rp, int64_t M, int64_t *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < npairs) out[i] = c_rp[d[i].moff];
    else if (i == npairs) out[npairs] = c_rp[M];
}

cudaError_t launch_gather_first(const PairDesc *d, int64_t npairs, const int64_t *c_rp, int64_t M, int64_t *out,
                                cudaStream_t st) {
    k_gather_first<<<(unsigned)((npairs + 256) / 256), 256, 0, st>>>(d, npairs, c_rp, M, out);
    return cudaGetLastError();
}

}  // namespace spg
