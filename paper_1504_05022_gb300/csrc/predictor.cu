// Learned preallocation: per-row features, a small MLP (forward, gradient,
// Adam), and the prediction of each bin-37 row's temporary size and launch
// class.  Not in the paper: it replaces the fixed 256-entry start of the
// progressive allocation (Section 4.1) by a predicted size, while the exact
// progressive path stays the fallback for any row predicted too small.
//
// Parameter vector (float32): W1[32x8] b1[32] W2[32x32] b2[32] W3[17x32] b3[17]
// then mu[8] sigma[8].  out = W3 relu(W2 relu(W1 (x-mu)/sigma + b1) + b2) + b3;
// out[0..15] are size-class logits, out[16] regresses log2(1 + nnz(c_i)).
#include "spgemm.h"
#include "internal.h"
#include "common.cuh"
#include "dynamic_smem.h"

#include <new>

namespace spg {

constexpr int MLP_IN = SPGEMM_MLP_FEATURES;
constexpr int MLP_HID = SPGEMM_MLP_HIDDEN;
constexpr int MLP_CLS = SPGEMM_MLP_CLASSES;
constexpr int MLP_OUT = MLP_CLS + 1;
constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + MLP_HID * MLP_IN;
constexpr int OFF_W2 = OFF_B1 + MLP_HID;
constexpr int OFF_B2 = OFF_W2 + MLP_HID * MLP_HID;
constexpr int OFF_W3 = OFF_B2 + MLP_HID;
constexpr int OFF_B3 = OFF_W3 + MLP_OUT * MLP_HID;
constexpr int OFF_MU = OFF_B3 + MLP_OUT;
constexpr int OFF_SG = OFF_MU + MLP_IN;
static_assert(OFF_MU == SPGEMM_MLP_NUM_PARAMS, "parameter layout");
static_assert(OFF_SG + MLP_IN == SPGEMM_MLP_NUM_TOTAL, "parameter layout");
constexpr int MLP_WORK = 153;  // floats of scratch per sample (spgemm_mlp_work_floats)

// ---------------- features ----------------

// One warp per row: the 8 features (log2(1+.) of nnz(a_i*), u_i, min/max/mean/std
// of the selected B-row lengths, the column span of the selected B rows, ncols(B)).
__global__ void k_row_features(DevCSR A, DevCSR B, const int64_t *__restrict__ u, int64_t u_min,
                               const uint8_t *__restrict__ skip, float *__restrict__ X) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= A.nrows) return;
    // with the bounds u given, only rows with u_i > u_min (bin 37) need features, and
    // not the dense-slice rows
    if (u != nullptr && u[row] <= u_min) return;
    if (skip != nullptr && skip[row]) return;
    const int64_t a0 = A.rp[row], a1 = A.rp[row + 1];
    double sum_len = 0.0, sg = 0.0, sg2 = 0.0;
    float gmin = 3.4e38f, gmax = -3.4e38f;
    int32_t cmin = INT_MAX, cmax = -1;
    for (int64_t p = a0 + lane; p < a1; p += 32) {
        const int32_t k = A.col[p];
        const int64_t b0 = B.rp[k], b1 = B.rp[k + 1];
        const int64_t len = b1 - b0;
        const float g = log2f(1.f + (float)len);
        sum_len += (double)len;
        sg += (double)g;
        sg2 += (double)g * (double)g;
        gmin = fminf(gmin, g);
        gmax = fmaxf(gmax, g);
        if (len > 0) {
            cmin = min(cmin, B.col[b0]);
            cmax = max(cmax, B.col[b1 - 1]);
        }
    }
    for (int d = 16; d > 0; d >>= 1) {
        sum_len += __shfl_xor_sync(SPG_FULL, sum_len, d);
        sg += __shfl_xor_sync(SPG_FULL, sg, d);
        sg2 += __shfl_xor_sync(SPG_FULL, sg2, d);
        gmin = fminf(gmin, __shfl_xor_sync(SPG_FULL, gmin, d));
        gmax = fmaxf(gmax, __shfl_xor_sync(SPG_FULL, gmax, d));
        cmin = min(cmin, __shfl_xor_sync(SPG_FULL, cmin, d));
        cmax = max(cmax, __shfl_xor_sync(SPG_FULL, cmax, d));
    }
    if (lane == 0) {
        const double n = (double)(a1 - a0);
        float *x = X + row * MLP_IN;
        x[0] = log2f(1.f + (float)n);
        x[1] = log2f(1.f + (float)sum_len);
        if (n > 0) {
            const double mean = sg / n;
            const double var = sg2 / n - mean * mean;
            x[2] = gmin;
            x[3] = gmax;
            x[4] = (float)mean;
            x[5] = (float)sqrt(var > 0.0 ? var : 0.0);
            x[6] = cmax >= 0 ? log2f(1.f + (float)(cmax - cmin + 1)) : 0.f;
        } else {
            x[2] = x[3] = x[4] = x[5] = x[6] = 0.f;
        }
        x[7] = log2f(1.f + (float)B.ncols);
    }
}

cudaError_t launch_row_features(const DevCSR &A, const DevCSR &B, float *X, cudaStream_t st, const int64_t *u,
                                int64_t u_min, const uint8_t *skip) {
    if (A.nrows <= 0) return cudaSuccess;
    const int64_t threads = A.nrows * 32;
    k_row_features<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(A, B, u, u_min, skip, X);
    return cudaGetLastError();
}

// ---------------- MLP ----------------

SPG_DEV void mlp_forward_one(const float *P, const float *x, float *xh, float *h1, float *h2, float *out) {
#pragma unroll
    for (int i = 0; i < MLP_IN; ++i) xh[i] = (x[i] - P[OFF_MU + i]) / P[OFF_SG + i];
#pragma unroll 4
    for (int o = 0; o < MLP_HID; ++o) {
        float z = P[OFF_B1 + o];
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i) z = fmaf(P[OFF_W1 + o * MLP_IN + i], xh[i], z);
        h1[o] = z > 0.f ? z : 0.f;
    }
#pragma unroll 4
    for (int o = 0; o < MLP_HID; ++o) {
        float z = P[OFF_B2 + o];
#pragma unroll 8
        for (int i = 0; i < MLP_HID; ++i) z = fmaf(P[OFF_W2 + o * MLP_HID + i], h1[i], z);
        h2[o] = z > 0.f ? z : 0.f;
    }
#pragma unroll 1
    for (int o = 0; o < MLP_OUT; ++o) {
        float z = P[OFF_B3 + o];
#pragma unroll 8
        for (int i = 0; i < MLP_HID; ++i) z = fmaf(P[OFF_W3 + o * MLP_HID + i], h2[i], z);
        out[o] = z;
    }
}

__global__ void k_mlp_forward(const float *__restrict__ params, const float *__restrict__ X, int64_t n,
                              float *__restrict__ out) {
    __shared__ float P[SPGEMM_MLP_NUM_TOTAL];
    for (int t = threadIdx.x; t < SPGEMM_MLP_NUM_TOTAL; t += blockDim.x) P[t] = params[t];
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float xh[MLP_IN], h1[MLP_HID], h2[MLP_HID], o[MLP_OUT];
    mlp_forward_one(P, X + s * MLP_IN, xh, h1, h2, o);
#pragma unroll
    for (int k = 0; k < MLP_OUT; ++k) out[s * MLP_OUT + k] = o[k];
}

// Loss and gradients of a batch in two launches.
//
// k_mlp_loss_grad: a CTA takes tiles of MLP_TILE samples.  Four threads share a sample, each with
// a quarter of every layer's neurons; activations and deltas lie in shared memory, a row per
// neuron, so that the weight gradients are products of those rows over the tile's samples,
// accumulated in registers over the CTA's tiles.  Every CTA leaves one partial gradient (and
// loss), which k_mlp_grad_sum adds in a fixed order: the result does not depend on timing.
// Each neuron's sum runs over its inputs in ascending order from the bias, as in
// mlp_forward_one.  Bound by shared-memory reads and latency (two CTAs per SM at 8,192 samples).
// A step of 8,192 samples with its Adam update takes 26 us; it took 118 us when one thread ran a
// whole sample and wrote a 612-byte record of it, which the reduction read with a stride.
constexpr int MLP_TILE = 64;
constexpr int MLP_NT = 4 * MLP_TILE;
constexpr int MLP_LD = MLP_TILE + 4;   // floats per row: 16-byte aligned, rows 4 banks apart
constexpr int MLP_MAX_CTAS = 304;      // partial gradients (two CTAs on each of 152 SMs)
constexpr int MLP_Q = MLP_HID / 4;     // a thread's neurons of a hidden layer
constexpr int MLP_PART = SPGEMM_MLP_NUM_PARAMS + 3;  // floats of a partial, with its loss as a double
static_assert(MLP_PART % 2 == 0 && MLP_Q == 8, "");

struct MlpShared {
    float w1t[MLP_IN][MLP_HID], w2t[MLP_HID][MLP_HID], w2[MLP_HID][MLP_HID];
    float w3t[MLP_HID][20], w3[MLP_OUT][MLP_HID];  // *t: by input, then neuron
    float b1[MLP_HID], b2[MLP_HID], b3[20], mu[MLP_IN], sg[MLP_IN];
    float xh[MLP_IN][MLP_LD], h1[MLP_HID][MLP_LD], h2[MLP_HID][MLP_LD];
    float dz1[MLP_HID][MLP_LD], dz2[MLP_HID][MLP_LD], out[MLP_OUT][MLP_LD], dout[MLP_OUT][MLP_LD];
    double loss[MLP_TILE];
};

// z[0..8) += w[0..8) * x (w 16-byte aligned, the same for the whole warp)
SPG_DEV void mlp_fma8(float (&z)[MLP_Q], const float *w, float x) {
    const float4 a = *reinterpret_cast<const float4 *>(w), b = *reinterpret_cast<const float4 *>(w + 4);
    z[0] = fmaf(a.x, x, z[0]);
    z[1] = fmaf(a.y, x, z[1]);
    z[2] = fmaf(a.z, x, z[2]);
    z[3] = fmaf(a.w, x, z[3]);
    z[4] = fmaf(b.x, x, z[4]);
    z[5] = fmaf(b.y, x, z[5]);
    z[6] = fmaf(b.z, x, z[6]);
    z[7] = fmaf(b.w, x, z[7]);
}

// acc += the product of rows x and y over four samples, in pairs (a quarter of the roundings
// that reach the long sum)
SPG_DEV float mlp_dot4(float acc, const float4 &x, const float4 &y) {
    return acc + (fmaf(x.w, y.w, x.z * y.z) + fmaf(x.y, y.y, x.x * y.x));
}

__global__ void __launch_bounds__(MLP_NT)
k_mlp_loss_grad(const float *__restrict__ params, const float *__restrict__ X, const int32_t *__restrict__ cls,
                const float *__restrict__ y, int64_t n, float *__restrict__ part, float *__restrict__ grad,
                double *__restrict__ loss) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpShared &S = *reinterpret_cast<MlpShared *>(mlp_smem);
    const int tid = threadIdx.x;
    for (int t = tid; t < MLP_HID * MLP_IN; t += MLP_NT) S.w1t[t % MLP_IN][t / MLP_IN] = params[OFF_W1 + t];
    for (int t = tid; t < MLP_HID * MLP_HID; t += MLP_NT) {
        const float w = params[OFF_W2 + t];
        S.w2t[t % MLP_HID][t / MLP_HID] = w;
        S.w2[t / MLP_HID][t % MLP_HID] = w;
    }
    for (int t = tid; t < MLP_OUT * MLP_HID; t += MLP_NT) {
        const float w = params[OFF_W3 + t];
        S.w3t[t % MLP_HID][t / MLP_HID] = w;
        S.w3[t / MLP_HID][t % MLP_HID] = w;
    }
    if (tid < MLP_HID) {
        S.b1[tid] = params[OFF_B1 + tid];
        S.b2[tid] = params[OFF_B2 + tid];
    }
    if (tid < MLP_OUT) S.b3[tid] = params[OFF_B3 + tid];
    if (tid < MLP_IN) {
        S.mu[tid] = params[OFF_MU + tid];
        S.sg[tid] = params[OFF_SG + tid];
    }
    const int s = tid & (MLP_TILE - 1), q = tid / MLP_TILE;  // sample of the tile, quarter (the same for a warp)
    const int o0 = q * MLP_Q;                                // the thread's hidden neurons
    // the thread's gradients: W2 rows {ta, ta + 16} x columns {tb, tb + 16}; W1 (tid / 8, tid % 8);
    // W3 rows {tid / 32, tid / 32 + 8} and, in the first warp, row 16, column tid % 32; a bias
    const int ta = tid >> 4, tb = tid & 15, ra = tid >> 5, rb = tid & 31;
    float g2[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, g1 = 0.f, g3[3] = {0.f, 0.f, 0.f}, gb = 0.f;
    double lsum = 0.0;
    for (int64_t base = (int64_t)blockIdx.x * MLP_TILE; base < n; base += (int64_t)gridDim.x * MLP_TILE) {
        const int64_t i = base + s;
        const bool ok = i < n;  // past the end: zero deltas
        __syncthreads();  // the weights are in place; the last tile's rows are free
        // a quarter's two inputs
#pragma unroll
        for (int k = 0; k < MLP_IN / 4; ++k) {
            const int f = q * (MLP_IN / 4) + k;
            S.xh[f][s] = ok ? (X[i * MLP_IN + f] - S.mu[f]) / S.sg[f] : 0.f;
        }
        __syncthreads();
        float h[MLP_Q];
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) h[k] = S.b1[o0 + k];
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) mlp_fma8(h, &S.w1t[k][o0], S.xh[k][s]);
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) S.h1[o0 + k][s] = h[k] > 0.f ? h[k] : 0.f;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) h[k] = S.b2[o0 + k];
#pragma unroll 8
        for (int k = 0; k < MLP_HID; ++k) mlp_fma8(h, &S.w2t[k][o0], S.h1[k][s]);
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) {
            h[k] = h[k] > 0.f ? h[k] : 0.f;
            S.h2[o0 + k][s] = h[k];
        }
        __syncthreads();
        // outputs 4q..4q+3, and 16 by the first quarter
        {
            float o[4] = {S.b3[4 * q], S.b3[4 * q + 1], S.b3[4 * q + 2], S.b3[4 * q + 3]}, o16 = S.b3[16];
#pragma unroll 8
            for (int k = 0; k < MLP_HID; ++k) {
                const float x = S.h2[k][s];
                const float4 w = *reinterpret_cast<const float4 *>(&S.w3t[k][4 * q]);
                o[0] = fmaf(w.x, x, o[0]);
                o[1] = fmaf(w.y, x, o[1]);
                o[2] = fmaf(w.z, x, o[2]);
                o[3] = fmaf(w.w, x, o[3]);
                if (q == 0) o16 = fmaf(S.w3t[k][16], x, o16);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) S.out[4 * q + k][s] = o[k];
            if (q == 0) S.out[16][s] = o16;
        }
        __syncthreads();
        {
            float o[MLP_CLS];
#pragma unroll
            for (int k = 0; k < MLP_CLS; ++k) o[k] = S.out[k][s];
            float mx = o[0];
#pragma unroll
            for (int k = 1; k < MLP_CLS; ++k) mx = fmaxf(mx, o[k]);
            float ex[MLP_CLS], se = 0.f;
#pragma unroll
            for (int k = 0; k < MLP_CLS; ++k) {
                ex[k] = expf(o[k] - mx);
                se += ex[k];
            }
            const int c = ok ? cls[i] : 0;
#pragma unroll
            for (int k = 0; k < MLP_CLS; ++k)
                if (k / 4 == q) S.dout[k][s] = ok ? ex[k] / se - (k == c ? 1.f : 0.f) : 0.f;
            if (q == 0) {
                const float r = ok ? S.out[MLP_CLS][s] - y[i] : 0.f;
                S.dout[MLP_CLS][s] = r;
                if (ok) lsum += (double)(logf(se) + mx - S.out[c][s]) + 0.5 * (double)r * (double)r;
            }
        }
        __syncthreads();
        float dz[MLP_Q];
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) dz[k] = 0.f;
#pragma unroll
        for (int k = 0; k < MLP_OUT; ++k) mlp_fma8(dz, &S.w3[k][o0], S.dout[k][s]);
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) S.dz2[o0 + k][s] = h[k] > 0.f ? dz[k] : 0.f;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) dz[k] = 0.f;
#pragma unroll 8
        for (int k = 0; k < MLP_HID; ++k) mlp_fma8(dz, &S.w2[k][o0], S.dz2[k][s]);
#pragma unroll
        for (int k = 0; k < MLP_Q; ++k) S.dz1[o0 + k][s] = S.h1[o0 + k][s] > 0.f ? dz[k] : 0.f;
        __syncthreads();
        // the gradients, four samples at a time
#pragma unroll 4
        for (int t = 0; t < MLP_TILE; t += 4) {
            auto row = [&](const float (*m)[MLP_LD], int r) { return *reinterpret_cast<const float4 *>(&m[r][t]); };
            const float4 a0 = row(S.dz2, ta), a1 = row(S.dz2, ta + 16), c0 = row(S.h1, tb), c1 = row(S.h1, tb + 16);
            g2[0][0] = mlp_dot4(g2[0][0], a0, c0);
            g2[0][1] = mlp_dot4(g2[0][1], a0, c1);
            g2[1][0] = mlp_dot4(g2[1][0], a1, c0);
            g2[1][1] = mlp_dot4(g2[1][1], a1, c1);
            g1 = mlp_dot4(g1, row(S.dz1, tid >> 3), row(S.xh, tid & 7));
            const float4 d = row(S.h2, rb);
            g3[0] = mlp_dot4(g3[0], row(S.dout, ra), d);
            g3[1] = mlp_dot4(g3[1], row(S.dout, ra + 8), d);
            if (ra == 0) g3[2] = mlp_dot4(g3[2], row(S.dout, 16), d);
            if (tid < 2 * MLP_HID + MLP_OUT) {
                const float4 v = tid < MLP_HID ? row(S.dz1, tid)
                                 : tid < 2 * MLP_HID ? row(S.dz2, tid - MLP_HID) : row(S.dout, tid - 2 * MLP_HID);
                gb += (v.x + v.y) + (v.z + v.w);
            }
        }
    }
    // the loss of the CTA's samples, in the order of the tile's slots
    __syncthreads();
    if (q == 0) S.loss[s] = lsum;
    __syncthreads();
    // one CTA: the result itself; else a partial of MLP_PART floats, the loss first
    float *g = gridDim.x == 1 ? grad : part + (int64_t)blockIdx.x * MLP_PART + 2;
    if (tid == 0) {
        double t = 0.0;
        for (int k = 0; k < MLP_TILE; ++k) t += S.loss[k];
        *(gridDim.x == 1 ? loss : reinterpret_cast<double *>(part + (int64_t)blockIdx.x * MLP_PART)) = t;
    }
    g[OFF_W1 + tid] = g1;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) g[OFF_W2 + (ta + 16 * a) * MLP_HID + tb + 16 * b] = g2[a][b];
    g[OFF_W3 + ra * MLP_HID + rb] = g3[0];
    g[OFF_W3 + (ra + 8) * MLP_HID + rb] = g3[1];
    if (ra == 0) g[OFF_W3 + 16 * MLP_HID + rb] = g3[2];
    if (tid < MLP_HID) g[OFF_B1 + tid] = gb;
    else if (tid < 2 * MLP_HID) g[OFF_B2 + tid - MLP_HID] = gb;
    else if (tid < 2 * MLP_HID + MLP_OUT) g[OFF_B3 + tid - 2 * MLP_HID] = gb;
}

// Sums the partial gradients: 64 parameters per CTA, eight threads a parameter, each over every
// eighth partial in ascending order, in four interleaved sums added pairwise.  The last CTA sums
// the losses.
__global__ void __launch_bounds__(512)
k_mlp_grad_sum(const float *__restrict__ part, int np, float *__restrict__ grad, double *__restrict__ loss) {
    __shared__ float acc[8][64];
    const int c = threadIdx.x & 63, r = threadIdx.x >> 6;
    const int k = blockIdx.x * 64 + c;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (k < SPGEMM_MLP_NUM_PARAMS) {
        for (int p0 = r; p0 < np; p0 += 32) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (p0 + 8 * j < np) v[j] += part[(int64_t)(p0 + 8 * j) * MLP_PART + 2 + k];
        }
    }
    acc[r][c] = (v[0] + v[1]) + (v[2] + v[3]);
    __syncthreads();
    if (r == 0 && k < SPGEMM_MLP_NUM_PARAMS)
        grad[k] = ((acc[0][c] + acc[1][c]) + (acc[2][c] + acc[3][c])) + ((acc[4][c] + acc[5][c]) + (acc[6][c] + acc[7][c]));
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 32) {
        double t = 0.0;
        for (int p = threadIdx.x; p < np; p += 32) t += *reinterpret_cast<const double *>(part + (int64_t)p * MLP_PART);
        t = warp_reduce_sum(t);
        if (threadIdx.x == 0) *loss = t;
    }
}

__global__ void k_mlp_adam(float *__restrict__ params, const float *__restrict__ grad, float *__restrict__ m,
                           float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float scale,
                           float bc1, float bc2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = grad[i] * scale;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

// Plan-side prediction for every row: predicted home size (>= min_cap, <= u_i)
// from the regression head, times `margin`, rounded up to 32; u_i itself when it is
// within a factor `margin` of that size.
__global__ void k_mlp_predict_caps(const float *__restrict__ params, const float *__restrict__ X, int64_t m,
                                   const int64_t *__restrict__ u, int64_t u_min, uint8_t *__restrict__ skip,
                                   float margin, int32_t min_cap, int32_t *__restrict__ pred_cap,
                                   int64_t promote_min) {
    __shared__ float P[SPGEMM_MLP_NUM_TOTAL];
    for (int t = threadIdx.x; t < SPGEMM_MLP_NUM_TOTAL; t += blockDim.x) P[t] = params[t];
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= m) return;
    // the row's bound u_i (Algorithm 2)
    const int64_t uu = u[s];
    // outside bin 37, or a dense-slice row: no prediction needed
    if (uu <= u_min || (skip != nullptr && skip[s])) {
        pred_cap[s] = 0;
        return;
    }
    float xh[MLP_IN], h1[MLP_HID], h2[MLP_HID], o[MLP_OUT];
    mlp_forward_one(P, X + s * MLP_IN, xh, h1, h2, o);
    float reg = fminf(fmaxf(o[MLP_CLS], 0.f), 30.f);
    double nnz = exp2((double)reg) - 1.0;
    if (promote_min > 0 && skip != nullptr && nnz >= (double)promote_min) {
        // the network's choice of kernel: a row this long goes to the dense-slice kernels
        skip[s] = 1;
        pred_cap[s] = 0;
        return;
    }
    double c = ceil(nnz * (double)margin / 32.0) * 32.0;
    int64_t cap = (int64_t)c;
    if (cap < min_cap) cap = min_cap;
    // a bound within a factor `margin` of the sized prediction is taken instead: the row
    // can then never outgrow its slot, for at most `margin` times the prediction's space
    if ((double)uu <= (double)cap * (double)margin) cap = uu;
    if (cap > uu) cap = uu;
    if (cap > INT32_MAX) cap = INT32_MAX;
    pred_cap[s] = (int32_t)cap;
}

cudaError_t launch_predict_caps(const float *params, const float *X, int64_t m, const int64_t *u, float margin,
                                int32_t min_cap, int32_t *pred_cap, cudaStream_t st, int64_t u_min, uint8_t *skip,
                                int64_t promote_min) {
    if (m <= 0) return cudaSuccess;
    k_mlp_predict_caps<<<(unsigned)((m + 127) / 128), 128, 0, st>>>(params, X, m, u, u_min, skip, margin,
                                                                     min_cap, pred_cap, promote_min);
    return cudaGetLastError();
}

// Launch-class partition of the bin-37 rows by predicted size: class g holds
// the rows whose predicted size is at most class_cap[g] (the smallest such g).
// The dense-slice rows go to slot ncls, after the classes.
// Bin 37 is the last segment of bin_rows; its size is read from the stage-2
// summary on the device, so no host round trip is needed.  The order inside a
// class is not fixed (atomics); it only affects scheduling, not C.
__global__ void k_class_count(const int32_t *bin_rows, int64_t m, const BinSummary *summary,
                              const int32_t *pred_cap, const int32_t *class_cap, int ncls, const uint8_t *dense,
                              int32_t *cls_of, int32_t *count) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n37 = summary->bin_count[BIN_MERGE];
    if (j >= n37) return;
    const int32_t row = bin_rows[m - n37 + j];
    const int32_t c = pred_cap[row];
    int g = ncls - 1;
    for (int k = 0; k < ncls; ++k)
        if (c <= class_cap[k]) {
            g = k;
            break;
        }
    if (dense != nullptr && dense[row]) g = ncls;
    cls_of[j] = g;
    atomicAdd(&count[g], 1);
}

__global__ void k_class_starts(const int32_t *count, int ncls, int32_t *start, int32_t *cursor,
                               BinSummary *summary) {
    if (threadIdx.x == 0) {
        int32_t s = 0;
        for (int g = 0; g <= ncls; ++g) {
            start[g] = s;
            cursor[g] = 0;
            if (g < ncls) summary->class_count[g] = count[g];
            s += count[g];
        }
    }
}

__global__ void k_class_scatter(int64_t m, const BinSummary *summary, const int32_t *cls_of, const int32_t *start,
                                int32_t *cursor, int32_t *order) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= summary->bin_count[BIN_MERGE]) return;
    const int g = cls_of[j];
    order[start[g] + atomicAdd(&cursor[g], 1)] = (int32_t)j;
}

cudaError_t launch_class_partition_tail(const int32_t *bin_rows, int64_t m, BinSummary *summary,
                                        const int32_t *pred_cap, const int32_t *class_cap, int ncls,
                                        const uint8_t *dense, int32_t *scratch, int32_t *order, cudaStream_t st) {
    if (m <= 0 || ncls > 31) return m <= 0 ? cudaSuccess : cudaErrorInvalidValue;
    int32_t *count = scratch, *start = scratch + 32, *cursor = scratch + 64, *cls_of = scratch + 96;
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int32_t) * 32, st);
    if (e != cudaSuccess) return e;
    const unsigned g = (unsigned)((m + 255) / 256);
    k_class_count<<<g, 256, 0, st>>>(bin_rows, m, summary, pred_cap, class_cap, ncls, dense, cls_of, count);
    k_class_starts<<<1, 32, 0, st>>>(count, ncls, start, cursor, summary);
    k_class_scatter<<<g, 256, 0, st>>>(m, summary, cls_of, start, cursor, order);
    return cudaGetLastError();
}

}  // namespace spg

// ---------------- C ABI of the predictor ----------------

using namespace spg;

struct spgemm_predictor {
    int device;
    float *params;  // device copy of the SPGEMM_MLP_NUM_TOTAL values
};

extern "C" spgemm_status spgemm_predictor_create(const float *host_params, int64_t n, spgemm_predictor **out) {
    if (!out || !host_params || n != SPGEMM_MLP_NUM_TOTAL) return SPGEMM_ERR_INVALID_ARG;
    *out = nullptr;
    spgemm_predictor *p = new (std::nothrow) spgemm_predictor();
    if (!p) return SPGEMM_ERR_OOM;
    if (cudaGetDevice(&p->device) != cudaSuccess) {
        delete p;
        return SPGEMM_ERR_CUDA;
    }
    cudaError_t e = cudaMalloc(&p->params, sizeof(float) * SPGEMM_MLP_NUM_TOTAL);
    if (e != cudaSuccess) {
        delete p;
        return e == cudaErrorMemoryAllocation ? SPGEMM_ERR_OOM : SPGEMM_ERR_CUDA;
    }
    e = cudaMemcpy(p->params, host_params, sizeof(float) * SPGEMM_MLP_NUM_TOTAL, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(p->params);
        delete p;
        return SPGEMM_ERR_CUDA;
    }
    *out = p;
    return SPGEMM_OK;
}

extern "C" spgemm_status spgemm_predictor_free(spgemm_predictor *p) {
    if (!p) return SPGEMM_OK;
    cudaFree(p->params);
    delete p;
    return SPGEMM_OK;
}

namespace spg {
const float *predictor_params(const void *pred) {
    return pred ? static_cast<const spgemm_predictor *>(pred)->params : nullptr;
}
}  // namespace spg

static spgemm_status widen_in(const spgemm_csr_in *M, DevCSR &D, int64_t **tmp, cudaStream_t st) {
    D.nrows = M->nrows;
    D.ncols = M->ncols;
    D.nnz = M->nnz;
    D.col = M->col_idx;
    D.val = M->val;
    *tmp = nullptr;
    if (M->rowptr_bits == 64) {
        D.rp = static_cast<const int64_t *>(M->row_ptr);
        return SPGEMM_OK;
    }
    if (cudaMallocAsync(reinterpret_cast<void **>(tmp), sizeof(int64_t) * (M->nrows + 1), st) != cudaSuccess)
        return SPGEMM_ERR_OOM;
    if (launch_widen_rowptr(static_cast<const int32_t *>(M->row_ptr), *tmp, M->nrows + 1, st) != cudaSuccess)
        return SPGEMM_ERR_CUDA;
    D.rp = *tmp;
    return SPGEMM_OK;
}

extern "C" spgemm_status spgemm_row_features(const spgemm_csr_in *A, const spgemm_csr_in *B, float *X,
                                             spgemm_stream_t stream) {
    if (!A || !B || (!X && A->nrows > 0)) return SPGEMM_ERR_INVALID_ARG;
    if (A->ncols != B->nrows) return SPGEMM_ERR_SHAPE;
    if ((A->rowptr_bits != 32 && A->rowptr_bits != 64) || (B->rowptr_bits != 32 && B->rowptr_bits != 64))
        return SPGEMM_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    DevCSR a, b;
    int64_t *ta = nullptr, *tb = nullptr;
    spgemm_status s = widen_in(A, a, &ta, st);
    if (s == SPGEMM_OK) s = widen_in(B, b, &tb, st);
    if (s == SPGEMM_OK && launch_row_features(a, b, X, st) != cudaSuccess) s = SPGEMM_ERR_CUDA;
    if (ta) cudaFreeAsync(ta, st);
    if (tb) cudaFreeAsync(tb, st);
    return s;
}

extern "C" spgemm_status spgemm_mlp_forward(const float *params, const float *X, int64_t n, float *out,
                                            spgemm_stream_t stream) {
    if (n < 0 || !params || (n > 0 && (!X || !out))) return SPGEMM_ERR_INVALID_ARG;
    if (n == 0) return SPGEMM_OK;
    k_mlp_forward<<<(unsigned)((n + 127) / 128), 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(params, X, n,
                                                                                                 out);
    return cudaGetLastError() == cudaSuccess ? SPGEMM_OK : SPGEMM_ERR_CUDA;
}

extern "C" spgemm_status spgemm_mlp_loss_grad(const float *params, const float *X, const int32_t *cls,
                                              const float *y, int64_t n, float *work, float *grad, double *loss,
                                              spgemm_stream_t stream) {
    if (n < 0 || !params || !grad || !loss || (n > 0 && (!X || !cls || !y || !work)))
        return SPGEMM_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (n == 0) {
        if (cudaMemsetAsync(loss, 0, sizeof(double), st) != cudaSuccess) return SPGEMM_ERR_CUDA;
        if (cudaMemsetAsync(grad, 0, sizeof(float) * SPGEMM_MLP_NUM_PARAMS, st) != cudaSuccess)
            return SPGEMM_ERR_CUDA;
        return SPGEMM_OK;
    }
    // at most n / MLP_TILE + 1 partials (none for one CTA), which n * MLP_WORK floats hold; their
    // losses are doubles
    const int64_t tiles = (n + MLP_TILE - 1) / MLP_TILE;
    const int ctas = (int)(tiles < MLP_MAX_CTAS ? tiles : MLP_MAX_CTAS);
    static_assert((int64_t)MLP_TILE * MLP_WORK >= 2 * MLP_PART, "the partials of n > MLP_TILE samples fit");
    if (ctas > 1 && reinterpret_cast<uintptr_t>(work) % 8 != 0) work += 1;  // 4-byte aligned: one float is spare
    if (allow_dynamic_smem((const void *)k_mlp_loss_grad, (int)sizeof(MlpShared)) != cudaSuccess)
        return SPGEMM_ERR_CUDA;
    k_mlp_loss_grad<<<ctas, MLP_NT, sizeof(MlpShared), st>>>(params, X, cls, y, n, work, grad, loss);
    if (ctas > 1) k_mlp_grad_sum<<<(SPGEMM_MLP_NUM_PARAMS + 63) / 64, 512, 0, st>>>(work, ctas, grad, loss);
    return cudaGetLastError() == cudaSuccess ? SPGEMM_OK : SPGEMM_ERR_CUDA;
}

extern "C" int64_t spgemm_mlp_work_floats(int64_t n) { return n * (int64_t)MLP_WORK; }

extern "C" spgemm_status spgemm_mlp_adam(float *params, const float *grad, float *m, float *v, int64_t step,
                                         float lr, float grad_scale, spgemm_stream_t stream) {
    if (!params || !grad || !m || !v || step < 1) return SPGEMM_ERR_INVALID_ARG;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    k_mlp_adam<<<(SPGEMM_MLP_NUM_PARAMS + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        params, grad, m, v, SPGEMM_MLP_NUM_PARAMS, lr, b1, b2, eps, grad_scale, bc1, bc2);
    return cudaGetLastError() == cudaSuccess ? SPGEMM_OK : SPGEMM_ERR_CUDA;
}
