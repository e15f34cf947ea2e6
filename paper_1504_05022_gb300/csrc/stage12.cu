// Stage 1 (upper bound, Algorithm 2) and stage 2 (binning and C~ sizing,
// Algorithm 3) of the SpGEMM framework, plus input widening and validation.
//
// Stage 1 gives a group of lanes to each row of A (as many as the rows' average length
// asks for), a warp to each long row and a whole block to a hub row, so that none unbalances the
// kernel the way one-thread-per-row (the paper's launch shape) would.  The same kernel bins the row,
// counts the bins of its block of rows and finds the column range of the bin-37 rows: u_i
// never goes through a prefix sum over A's nonzeros, which took 16 bytes of traffic per
// nonzero and three launches.
//
// Stage 2 runs on the GPU instead of a CPU core (the paper's choice, Section 4.1)
// and without device-wide atomics: per-block 38-bin histograms, one block that scans the
// (bin, block) counts with a warp per bin, and a stable scatter that keeps rows
// in ascending order inside every bin.
#include "internal.h"
#include "scan.cuh"

#include <mutex>
#include <vector>

namespace spg {

int persistent_blocks(const void *kern, int nt, size_t smem, int64_t cap) {
    static std::mutex mu;
    static std::vector<int> sms;  // SM count per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    int nsm = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        if ((int)sms.size() <= dev) sms.resize(dev + 1, 0);
        if (sms[dev] == 0 && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 0;
        nsm = sms[dev];
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int64_t g = (int64_t)nsm * per_sm;
    return (int)(cap > 0 && cap < g ? cap : g);
}

__global__ void k_widen_rowptr(const int32_t *in, int64_t *out, int64_t n, const int32_t *in2, int64_t *out2,
                               int64_t n2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (int64_t)in[i];
    if (i < n2) out2[i] = (int64_t)in2[i];
}

cudaError_t launch_widen_rowptr(const int32_t *in, int64_t *out, int64_t n, cudaStream_t st, const int32_t *in2,
                                int64_t *out2, int64_t n2) {
    const int64_t most = n > n2 ? n : n2;
    if (most <= 0) return cudaSuccess;
    k_widen_rowptr<<<(unsigned)((most + 255) / 256), 256, 0, st>>>(in, out, n, in2, out2, n2);
    return cudaGetLastError();
}

// One warp per row: row_ptr monotone and within [0, nnz], columns in range and
// strictly ascending.  Writes 1 into *status on the first violation found.
__global__ void k_validate(DevCSR M, int64_t *status) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w > M.nrows) return;
    if (w == M.nrows) {
        if (lane == 0 && (M.rp[0] != 0 || M.rp[M.nrows] != M.nnz)) *status = 1;
        return;
    }
    const int64_t s = M.rp[w], e = M.rp[w + 1];
    bool bad = (s > e) || (s < 0) || (e > M.nnz);
    if (!bad) {
        for (int64_t p = s + lane; p < e; p += 32) {
            int32_t c = M.col[p];
            if (c < 0 || c >= M.ncols) bad = true;
            if (p + 1 < e && M.col[p + 1] <= c) bad = true;
        }
    }
    if (__any_sync(SPG_FULL, bad) && lane == 0) *status = 1;
}

cudaError_t launch_validate(const DevCSR &M, int64_t *status, cudaStream_t st) {
    int64_t warps = M.nrows + 1;
    int64_t threads = warps * 32;
    k_validate<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(M, status);
    return cudaGetLastError();
}

// ---------------- stages 1 and 2 ----------------

struct StoreI64 {
    int64_t *out;
    SPG_DEV void operator()(int64_t i, int64_t v) const { out[i] = v; }
};

constexpr int BOUND_NT = 512;
constexpr int BIN_NT = 256;  // of the scatter
constexpr int BIN_NW = BIN_NT / 32;
constexpr int LONG_STEPS = 16;      // a row longer than this many times its group is taken by a warp,
constexpr int HUB_ENTRIES = 1024;   // one of more entries than this by the block

// Lanes per row: a quarter of the average length of A's rows or more, so that a lane has about
// four entries' gathers in flight; more lanes while that leaves SMs without a block.
static int bound_group(int64_t m, int64_t nnz) {
    const int64_t avg = m > 0 ? nnz / m : 0;
    int g = avg <= 16 ? 4 : avg <= 32 ? 8 : avg <= 64 ? 16 : 32;
    while (g < 32 && g < avg && m * g < (int64_t)152 * BOUND_NT) g *= 2;
    return g;
}

// Stage 1 runs a block per BOUND_NT / group rows, or twice as many where that leaves blocks
// enough (more would let a run of hub rows, the low rows of an R-MAT matrix, hold up an SM: 13
// times as many took 1.7 ms at 2^20 rows, once 0.42); stage 2 bins blocks of that many rows
// times a factor that leaves about four per SM (of 152), since one block scans the counts.
static int64_t bound_rows(int64_t m, int64_t nnz) {
    const int64_t rows = BOUND_NT / bound_group(m, nnz);
    const int64_t fold = m / (rows * 608);
    return rows * (fold < 1 ? 1 : fold > 2 ? 2 : fold);
}
static int64_t bin_rows_per_block(int64_t m, int64_t nnz) {
    const int64_t rows = bound_rows(m, nnz);
    const int64_t factor = (m + rows * 608 - 1) / (rows * 608);
    return rows * (factor < 1 ? 1 : factor);
}

int64_t bin_blocks(int64_t m, int64_t nnz) {
    const int64_t r = bin_rows_per_block(m, nnz);
    return (m + r - 1) / r;
}

// Algorithm 3: bin 0 (u = 0), bin 1 (u = 1), bins 2..32 (u = 2..32, one bin per
// size), bins 33..36 (33-64, 65-128, 129-256, 257-512), bin 37 (u > 512).
SPG_DEV int bin_of(int64_t u) {
    if (u <= 32) return (int)u;
    if (u <= 64) return 33;
    if (u <= 128) return 34;
    if (u <= 256) return 35;
    if (u <= 512) return 36;
    return 37;
}

// Size of row i in C~.  Hybrid (Algorithm 3): u_i for bins 0..36, a fixed
// initial size (256) for bin 37.  Upper bound: u_i.  Learned: u_i for bins
// 0..36, the predicted size (never above u_i) for bin 37.  Bin-37 rows computed
// by the dense-slice kernels take none in every policy, and the precise method
// has no C~ at all.
SPG_DEV int64_t cap_of(int64_t u, int b, int64_t i, const CapPolicy &P, bool dense) {
    if (P.policy == POLICY_PRECISE) return 0;  // counted first, then computed straight into C
    if (dense) return 0;  // written straight into C
    if (P.policy == POLICY_UPPER_BOUND) return u;
    if (P.policy == POLICY_LEARNED && P.pred_cap != nullptr && b == BIN_MERGE) {
        int64_t c = P.pred_cap[i];
        if (c > P.cap_max) c = P.cap_max;  // longer rows are split into column slices anyway
        return c < u ? (c < 1 ? 1 : c) : u;
    }
    if (b == BIN_MERGE) return P.initial_cap < u ? P.initial_cap : u;
    return u;
}

SPG_DEV bool dense_row(int b, int64_t i, const CapPolicy &P) {
    return b == BIN_MERGE && P.dense != nullptr && P.dense[i] != 0;
}

// u_i, bin and row size of every row, and per `factor` blocks the histogram of the rows and the
// sums of C~ entries and of u_i and the rows that only the batched merge kernel can take
// (part[0..nblk), part[nblk..2 nblk), part[2 nblk..3 nblk)), zeroed before when factor > 1.  Bin-37 rows also get their column
// range [lo, hi) (first and last column of every B row they select) and the flag that sends them
// to the dense-slice kernels: u_i >= dmin (dmin > 0), else div u_i >= hi - lo -- their products
// cover at least a div-th of the columns they can reach, so the accumulator's O(hi - lo) clearing
// and write-out are small beside them.  By default div = 32 up to DENSE_LONG_U products, where
// the register merge kernel is the other way, and 512 above, where it is the batched one.  The
// product by hybrid / learned plans, ms, at div 8, 32 and 64: R-MAT 2^16 x 16 4.70, 3.64, 3.53 /
// 3.84, 3.52, 3.55, 2^17 x 8 9.23, 4.38, 3.95 / 5.09, 3.74, 3.73, 2^18 x 8 37.9, 14.6, 10.7 / 27.0,
// 10.7, 9.78 (at 64 the learned plan, at its peak there, no longer needs less memory than the
// bound's).  Rows of uniformly random columns are the slices' worst case, merge against slices:
// u = 2,500 of 200,000 columns (div 80) 18.7, 16.0, u = 1,600 (125) 11.7, 13.8, u = 4,096 of
// 500,000 (122) 3.86, 5.28; above the line u = 9,216 of 4,000,000 (434) 46.7, 34.3.
// Rows of fewer than 1,024 products stay with the register merge, where hubs leave it little to
// gain (R-MAT 2^16 x 16: 3.54 / 3.56), and ranges of at most DENSE_SHORT_RANGE columns at an
// eighth, the line that small products were always given (R-MAT 2^13 x 16: 0.57 against 0.47).
// Latency-bound (two dependent gathers per nonzero): the 27-point
// operator on 64^3 (6.9 M nonzeros) takes 45 us here (cold caches) and took 113 us as a prefix
// sum, a marking pass and a histogram pass.
template <int G>
__global__ void __launch_bounds__(BOUND_NT, 3)
k_bound(DevCSR A, DevCSR B, CapPolicy P, BoundOut O, int R, int factor, int64_t nblk) {
    __shared__ int32_t hist[NUM_BINS];
    constexpr int ROWS = BOUND_NT / G;
    __shared__ int32_t nlong, longs[2 * ROWS];
    __shared__ int64_t scratch[BOUND_NT / 32 + 1];
    __shared__ int32_t range[2];
    const int gl = threadIdx.x & (G - 1), grp = threadIdx.x / G;
    const unsigned gm = G == 32 ? SPG_FULL : ((1u << (G & 31)) - 1u) << (lane_id() & ~(G - 1));
    if (threadIdx.x < NUM_BINS) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        nlong = 0;
        if (blockIdx.x == 0) *O.err = 0;
    }
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * R;
    int64_t capsum = 0, usum = 0, batched = 0;
    auto sum_of = [&](int64_t p0, int64_t p1, int step) {
        int64_t u = 0;
#pragma unroll 4
        for (int64_t p = p0; p < p1; p += step) {
            const int32_t k = A.col[p];
            u += B.rp[k + 1] - B.rp[k];
        }
        return u;
    };
    auto range_of = [&](int64_t p0, int64_t p1, int step, int32_t &cmin, int32_t &cmax) {
        cmin = INT32_MAX;
        cmax = -1;
        int64_t sum = 0;
        constexpr int UN = 4;  // entries whose dependent gathers are in flight together
        for (int64_t p = p0; p < p1; p += UN * step) {
            int64_t rs[UN], re[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                rs[u] = re[u] = 0;
                if (p + u * step < p1) {
                    const int32_t k = A.col[p + u * step];
                    rs[u] = B.rp[k];
                    re[u] = B.rp[k + 1];
                }
            }
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                if (re[u] > rs[u]) {
                    cmin = min(cmin, B.col[rs[u]]);
                    cmax = max(cmax, B.col[re[u] - 1]);
                }
                sum += re[u] - rs[u];
            }
        }
        return sum;
    };
    // by one thread per row; the range is that of a bin-37 row where flags are wanted
    auto finish = [&](int64_t i, int64_t u, int b, int64_t nA, int32_t cmin, int32_t cmax) {
        bool dense = false;
        if (P.dense != nullptr) {
            if (b == BIN_MERGE) {
                const int64_t span = (int64_t)cmax - cmin + 1;  // u > 0, so some B row is not empty
                const int div = u > DENSE_LONG_U ? O.div_long : span > DENSE_SHORT_RANGE ? O.div : O.div_short;
                dense = O.dmin > 0 ? u >= O.dmin
                                   : (int64_t)div * u >= span && (span <= DENSE_SHORT_RANGE || u >= O.floor);
                O.lo[i] = cmin;
                O.hi[i] = cmax + 1;
            }
            O.flag[i] = (uint8_t)dense;
        }
        O.u[i] = u;
        O.bin[i] = (uint8_t)b;
        O.nnzc[i] = (b <= 1) ? (int32_t)u : 0;
        atomicAdd(&hist[b], 1);
        capsum += cap_of(u, b, i, P, dense);
        usum += u;
        if (b == BIN_MERGE && !dense && merge_small_threads(u, (int)min(nA, (int64_t)INT32_MAX), O.small_u) == 0) ++batched;
    };
    for (int r0 = 0; r0 < R; r0 += ROWS) {
        const int64_t i = base + r0 + grp;
        if (i >= A.nrows) break;  // the whole group
        const int64_t a0 = A.rp[i], a1 = A.rp[i + 1];
        if (a1 - a0 > LONG_STEPS * G) {
            if (gl == 0) longs[atomicAdd(&nlong, 1)] = r0 + grp;
            continue;
        }
        int64_t u = sum_of(a0 + gl, a1, G);
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) u += __shfl_xor_sync(gm, u, d, G);
        const int b = bin_of(u);
        int32_t cmin = 0, cmax = 0;
        if (b == BIN_MERGE && P.dense != nullptr) {
            range_of(a0 + gl, a1, G, cmin, cmax);
#pragma unroll
            for (int d = G / 2; d > 0; d >>= 1) {
                cmin = min(cmin, __shfl_xor_sync(gm, cmin, d, G));
                cmax = max(cmax, __shfl_xor_sync(gm, cmax, d, G));
            }
        }
        if (gl == 0) finish(i, u, b, a1 - a0, cmin, cmax);
    }
    __syncthreads();
    const int nl = nlong;
    for (int l = warp_id(); l < nl; l += BOUND_NT / 32) {
        const int64_t i = base + longs[l];
        const int64_t a0 = A.rp[i], a1 = A.rp[i + 1];
        if (a1 - a0 > HUB_ENTRIES) continue;
        int32_t cmin = 0, cmax = 0;
        int64_t u;
        if (P.dense != nullptr) {  // most long rows are in bin 37: one pass for both
            u = warp_reduce_sum(range_of(a0 + lane_id(), a1, 32, cmin, cmax));
            cmin = __reduce_min_sync(SPG_FULL, cmin);
            cmax = __reduce_max_sync(SPG_FULL, cmax);
        } else {
            u = warp_reduce_sum(sum_of(a0 + lane_id(), a1, 32));
        }
        const int b = bin_of(u);
        if (lane_id() == 0) finish(i, u, b, a1 - a0, cmin, cmax);
    }
    for (int l = 0; l < nl; ++l) {
        const int64_t i = base + longs[l];
        const int64_t a0 = A.rp[i], a1 = A.rp[i + 1];
        if (a1 - a0 <= HUB_ENTRIES) continue;
        __syncthreads();
        if (threadIdx.x < 2) range[threadIdx.x] = threadIdx.x == 0 ? INT32_MAX : -1;
        const int64_t u = block_reduce_sum<BOUND_NT>(sum_of(a0 + threadIdx.x, a1, BOUND_NT), scratch);
        const int b = bin_of(u);
        if (b == BIN_MERGE && P.dense != nullptr) {
            int32_t cmin, cmax;
            range_of(a0 + threadIdx.x, a1, BOUND_NT, cmin, cmax);
            cmin = __reduce_min_sync(SPG_FULL, cmin);
            cmax = __reduce_max_sync(SPG_FULL, cmax);
            if (lane_id() == 0) {
                atomicMin(&range[0], cmin);
                atomicMax(&range[1], cmax);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) finish(i, u, b, a1 - a0, range[0], range[1]);
    }
    __syncthreads();
    // the block's three sums, a warp's at a time
    __shared__ int64_t sums[3][BOUND_NT / 32];
    capsum = warp_reduce_sum(capsum);
    usum = warp_reduce_sum(usum);
    batched = warp_reduce_sum(batched);
    if (lane_id() == 0) {
        sums[0][warp_id()] = capsum;
        sums[1][warp_id()] = usum;
        sums[2][warp_id()] = batched;
    }
    __syncthreads();
    const int64_t blk = blockIdx.x / factor;
    if (threadIdx.x < NUM_BINS) {
        int32_t *h = &O.hist[(int64_t)threadIdx.x * nblk + blk];
        if (factor == 1) *h = hist[threadIdx.x];
        else if (hist[threadIdx.x] != 0) atomicAdd(h, hist[threadIdx.x]);
    } else if (threadIdx.x >= 64 && threadIdx.x < 67) {
        const int k = threadIdx.x - 64;
        int64_t t = 0;
        for (int w = 0; w < BOUND_NT / 32; ++w) t += sums[k][w];
        int64_t *o = &O.part[k * nblk + blk];
        if (factor == 1) *o = t;
        else if (t != 0) atomicAdd((unsigned long long *)o, (unsigned long long)t);
    }
}

// Exclusive scan of v[0..n) in place by one warp; returns the total.
template <typename T>
SPG_DEV T warp_scan_array(T *v, int64_t n) {
    T carry = 0;
    const int lane = lane_id();
    constexpr int UN = 8;
    for (int64_t i0 = 0; i0 < n; i0 += 32 * UN) {
        T x[UN];
#pragma unroll
        for (int q = 0; q < UN; ++q) x[q] = i0 + 32 * q + lane < n ? v[i0 + 32 * q + lane] : T(0);
#pragma unroll
        for (int q = 0; q < UN; ++q) {
            const T inc = warp_inclusive_scan(x[q]);
            if (i0 + 32 * q + lane < n) v[i0 + 32 * q + lane] = carry + inc - x[q];
            carry += __shfl_sync(SPG_FULL, inc, 31);
        }
    }
    return carry;
}

// One block: exclusive scans of every bin's block counts (a warp per bin, offsets inside the
// bin) and of the per-block C~ sizes; writes the summary, also into host memory the device can
// write (`host`, when given), and C~.rp[m].
__global__ void __launch_bounds__(1024)
k_bin_scan(int64_t m, int32_t *hist, int64_t nblk, int64_t *part, int64_t *ctil_rp, BinSummary *summary,
           BinSummary *host) {
    __shared__ int64_t total[NUM_BINS + 3], bstart[NUM_BINS + 1];
    const int lane = lane_id();
    for (int b = warp_id(); b < NUM_BINS + 3; b += 32) {
        const int64_t t = b < NUM_BINS ? (int64_t)warp_scan_array(hist + b * nblk, nblk)
                                       : warp_scan_array(part + (b - NUM_BINS) * nblk, nblk);
        if (lane == 0) total[b] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t s = 0;
        for (int b = 0; b < NUM_BINS; ++b) {
            bstart[b] = s;
            s += total[b];
        }
        bstart[NUM_BINS] = s;
        ctil_rp[m] = total[NUM_BINS];
    }
    __syncthreads();
    BinSummary *dst[2] = {summary, host};
    for (int k = 0; k < (host != nullptr ? 2 : 1); ++k) {
        BinSummary *S = dst[k];
        if (threadIdx.x < NUM_BINS) S->bin_count[threadIdx.x] = total[threadIdx.x];
        if (threadIdx.x <= NUM_BINS) S->bin_start[threadIdx.x] = bstart[threadIdx.x];
        if (threadIdx.x < NUM_LAUNCH_CLASSES) S->class_count[threadIdx.x] = 0;
        if (threadIdx.x == 0) {
            S->sum_cap = total[NUM_BINS];
            S->sum_u = total[NUM_BINS + 1];
            S->merge_batched = total[NUM_BINS + 2];
            S->dense_count = S->dense_entries = 0;
            S->dense_end[0] = S->dense_end[1] = 0;
        }
    }
}

__global__ void __launch_bounds__(BIN_NT)
k_bin_scatter(int64_t m, int R, const int64_t *u_in, const uint8_t *bin_in, CapPolicy P,
              const int32_t *hist_off, const int64_t *cap_off, int64_t nblk, const BinSummary *summary,
              int32_t *bin_rows, int64_t *ctil_rp) {
    __shared__ int32_t wcnt[BIN_NW][NUM_BINS];
    __shared__ int32_t run[NUM_BINS];
    __shared__ int64_t scratch[BIN_NW + 1];
    const int lane = lane_id(), wid = warp_id();
    // the next place of each bin's rows
    if (threadIdx.x < NUM_BINS)
        run[threadIdx.x] = (int32_t)summary->bin_start[threadIdx.x] + hist_off[(int64_t)threadIdx.x * nblk + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * R;
    const int64_t end = min(m, base + R);
    int64_t capcarry = cap_off[blockIdx.x];
    const unsigned lt_mask = (1u << lane) - 1u;
    for (int64_t i0 = base; i0 < end; i0 += BIN_NT) {
        for (int t = threadIdx.x; t < BIN_NW * NUM_BINS; t += BIN_NT) (&wcnt[0][0])[t] = 0;
        __syncthreads();
        const int64_t i = i0 + threadIdx.x;
        const bool valid = i < end;
        int b = valid ? (int)bin_in[i] : 255;
        unsigned peers = __match_any_sync(SPG_FULL, b);
        int rank = __popc(peers & lt_mask);
        if (valid && lane == __ffs(peers) - 1) wcnt[wid][b] = __popc(peers);
        __syncthreads();
        int64_t cap = 0;
        if (valid) {
            int pos = run[b] + rank;
            for (int w = 0; w < wid; ++w) pos += wcnt[w][b];
            bin_rows[pos] = (int32_t)i;
            cap = cap_of(u_in[i], b, i, P, dense_row(b, i, P));
        }
        int64_t tot;
        int64_t ex = block_exclusive_scan<BIN_NT>(cap, scratch, tot);
        if (valid) ctil_rp[i] = capcarry + ex;
        capcarry += tot;
        if (threadIdx.x < NUM_BINS) {
            int32_t s = 0;
#pragma unroll
            for (int w = 0; w < BIN_NW; ++w) s += wcnt[w][threadIdx.x];
            run[threadIdx.x] += s;
        }
        __syncthreads();
    }
}

// The rows of C~ laid out again from the stored u_i and bins under policy P (the learned
// sizes are known only after the binning): ctil_rp[0..m] and the total into *total.
struct LoadCap {
    const int64_t *u;
    const uint8_t *bin;
    CapPolicy P;
    SPG_DEV int64_t operator()(int64_t i) const { return cap_of(u[i], (int)bin[i], i, P, dense_row((int)bin[i], i, P)); }
};

cudaError_t launch_cap_rescan(int64_t m, const int64_t *u, const uint8_t *bin, CapPolicy P, int64_t *ctil_rp,
                              int64_t *partial, int64_t *total, cudaStream_t st) {
    cudaError_t e = device_exclusive_scan(m, LoadCap{u, bin, P}, StoreI64{ctil_rp}, partial, total, st);
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(ctil_rp + m, total, sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
}

cudaError_t launch_bound(const DevCSR &A, const DevCSR &B, const CapPolicy &P, const BoundOut &O, cudaStream_t st) {
    const int64_t nblk = bin_blocks(A.nrows, A.nnz);
    if (P.dense != nullptr && (O.div < 1 || O.div_short < 1 || O.div_long < 1)) return cudaErrorInvalidValue;
    if (nblk <= 0) return cudaMemsetAsync(O.err, 0, sizeof(int64_t), st);
    const int64_t rows = bound_rows(A.nrows, A.nnz);
    const int factor = (int)(bin_rows_per_block(A.nrows, A.nnz) / rows);
    if (factor > 1) {
        cudaError_t e = cudaMemsetAsync(O.hist, 0, sizeof(int32_t) * NUM_BINS * nblk, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(O.part, 0, sizeof(int64_t) * 3 * nblk, st);
        if (e != cudaSuccess) return e;
    }
    auto go = [&](auto kern) {
        kern<<<(unsigned)((A.nrows + rows - 1) / rows), BOUND_NT, 0, st>>>(A, B, P, O, (int)rows, factor, nblk);
        return cudaGetLastError();
    };
    switch (bound_group(A.nrows, A.nnz)) {
        case 4: return go(k_bound<4>);
        case 8: return go(k_bound<8>);
        case 16: return go(k_bound<16>);
        default: return go(k_bound<32>);
    }
}

cudaError_t launch_binning(int64_t m, int64_t nnzA, const CapPolicy &P, const BoundOut &O, int32_t *bin_rows,
                           int64_t *ctil_rp, BinSummary *summary, BinSummary *host, cudaStream_t st) {
    const int64_t nblk = bin_blocks(m, nnzA);
    k_bin_scan<<<1, 1024, 0, st>>>(m, O.hist, nblk, O.part, ctil_rp, summary, host);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (nblk > 0)
        k_bin_scatter<<<(unsigned)nblk, BIN_NT, 0, st>>>(m, (int)bin_rows_per_block(m, nnzA), O.u, O.bin, P, O.hist,
                                                          O.part, nblk, summary, bin_rows, ctil_rp);
    return cudaGetLastError();
}

}  // namespace spg
