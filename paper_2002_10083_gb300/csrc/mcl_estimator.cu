// Learned output-size estimator: per-column features, a 16 -> 64 -> 64 -> 2
// MLP (BF16 weights, FP32 accumulation) predicting y0 = log(1 + nnz_j) and
// y1 = log cf_j for every column of A*A, and its training kernels
// (backward pass, Adam).  The prediction replaces the exact symbolic
// SpGEMM (Sections II and V: memory estimation before every iteration)
// for sizing the accumulators; the numeric pass stays exact whatever the
// estimate (an under-estimate only narrows row ranges).
//
// Parameter layout (5378 values): W1 [64 x 16] (row = output unit), b1 [64],
// W2 [64 x 64], b2 [64], W3 [2 x 64], b3 [2].  Inputs are standardised with
// (x - mu) / sigma (norm = mu[16] then sigma[16]).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "mcl.h"
#include "mcl_device.cuh"
#include "mcl_internal.h"

namespace mcl {

constexpr int NIN = 16, NH = 64, NOUT = 2;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH,
              OFF_B2 = OFF_W2 + NH * NH, OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH,
              NPARAM = OFF_B3 + NOUT;
static_assert(NPARAM == MCL_MLP_NPARAM, "parameter count");
constexpr int HUGE_DEG = 1024;

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) {
    return __uint_as_float(((uint32_t)b) << 16);
}

// ---------------------------------------------------------------------------
// features
// ---------------------------------------------------------------------------

__global__ void k_colmax(CscView A, float* colmax) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = gw; j < A.n; j += nw) {
        float m = 0.0f;
        for (int64_t p = A.colptr[j] + lane; p < A.colptr[j + 1]; p += 32) m = fmaxf(m, A.val[p]);
        m = warp_max(m);
        if (lane == 0) colmax[j] = m;
    }
}

// The 16 features (see oracle/mlp.py FEATURES for the list).  A warp sums the
// entries of `group` columns one after the other, lane l keeping the totals of
// the group's column l, and then each lane finishes its own column: the FP64
// divisions and logarithms (2 lanes per clock and SM) of a whole warp cost what
// those of one column did, 3.8 ms of 300k columns.
__global__ void k_features(CscView A, int32_t iteration, const int32_t* iter_dev,
                           const float* prev_logcf, const float* colmax, float* feats, int group) {
    if (iter_dev) iteration = *iter_dev;  // graph replays keep the index on the device
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float logn = logf((float)(A.n > 0 ? A.n : 1));
    const float logit = log1pf((float)iteration);
    for (int64_t j0 = gw * group; j0 < A.n; j0 += nw * group) {
        const int m = (int)min((int64_t)group, A.n - j0);
        long long t_sd = 0, t_sd2 = 0;
        int t_md = 0, t_huge = 0, t_fmin = INT_MAX, t_lmax = -1, t_first = 0, t_last = 0, t_d = 0;
        double t_sa = 0.0, t_sa2 = 0.0, t_scm = 0.0;
        float t_ma = 0.0f;
        for (int c = 0; c < m; ++c) {
            const int64_t cb = A.colptr[j0 + c], ce = A.colptr[j0 + c + 1];
            long long sd = 0, sd2 = 0;
            int md = 0, huge = 0, fmin = INT_MAX, lmax = -1;
            double sa = 0.0, sa2 = 0.0, scm = 0.0;
            float ma = 0.0f;
            for (int64_t p = cb + lane; p < ce; p += 32) {
                const int k = A.rowidx[p];
                const float a = A.val[p];
                const int64_t ks = A.colptr[k], ke = A.colptr[k + 1];
                const int dk = (int)(ke - ks);
                sd += dk;
                sd2 += (long long)dk * dk;
                md = max(md, dk);
                huge += dk > HUGE_DEG;
                sa += a;
                sa2 += (double)a * a;
                ma = fmaxf(ma, a);
                scm += colmax[k];
                if (dk > 0) {
                    fmin = min(fmin, A.rowidx[ks]);
                    lmax = max(lmax, A.rowidx[ke - 1]);
                }
            }
            sd = warp_sum(sd);
            sd2 = warp_sum(sd2);
            md = warp_max(md);
            huge = warp_sum(huge);
            sa = warp_sum(sa);
            sa2 = warp_sum(sa2);
            ma = warp_max(ma);
            scm = warp_sum(scm);
            fmin = warp_min(fmin);
            lmax = warp_max(lmax);
            if (lane == c) {
                t_sd = sd;
                t_sd2 = sd2;
                t_md = md;
                t_huge = huge;
                t_sa = sa;
                t_sa2 = sa2;
                t_ma = ma;
                t_scm = scm;
                t_fmin = fmin;
                t_lmax = lmax;
                t_d = (int)(ce - cb);
                if (ce > cb) {
                    t_first = A.rowidx[cb];
                    t_last = A.rowidx[ce - 1];
                }
            }
        }
        if (lane < m) {
            const int64_t j = j0 + lane;
            const double dd = (double)t_d;
            float f[NIN];
            f[0] = log1pf((float)t_d);
            f[1] = (float)log1p((double)t_sd);
            f[2] = t_d ? log1pf((float)t_md) : 0.0f;
            f[3] = f[4] = f[8] = f[9] = f[13] = 0.0f;
            if (t_d) {
                const double mean = (double)t_sd / dd;
                const double var = (double)t_sd2 / dd - mean * mean;
                f[3] = (float)log1p(mean);
                f[4] = (float)log1p(var > 0.0 ? var : 0.0);
                f[8] = log1pf((float)(t_last - t_first + 1));
                f[9] = (float)((double)t_huge / dd);
                f[13] = (float)(t_scm / dd);
            }
            f[5] = t_ma;
            f[6] = (float)t_sa;
            f[7] = (float)t_sa2;
            f[10] = logn;
            f[11] = logit;
            f[12] = prev_logcf ? prev_logcf[j] : 0.0f;
            f[14] = t_lmax >= 0 ? (float)log1p((double)(t_lmax - t_fmin) + 1.0) : 0.0f;
            f[15] = 1.0f;
            if (((uintptr_t)feats & 15) == 0) {
#pragma unroll
                for (int q = 0; q < NIN; q += 4)
                    *reinterpret_cast<float4*>(feats + j * NIN + q) = make_float4(f[q], f[q + 1], f[q + 2], f[q + 3]);
            } else {
#pragma unroll
                for (int q = 0; q < NIN; ++q) feats[j * NIN + q] = f[q];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------

// Weights in shared memory as FP32, W2's rows padded by four words: the lanes
// of a warp read four (or eight) rows at once, 16 bytes each, from different
// banks.
constexpr int W2P = NH + 4;

struct __align__(16) MlpWeights {
    float w1[NH * NIN];
    float w2[NH * W2P];
    float w3[NOUT * NH];
    float b1[NH], b2[NH], b3[4];
    float mu[NIN], isg[NIN];
};

__device__ __forceinline__ void load_weights(MlpWeights& M, const uint16_t* wbits, const float* norm) {
    // Eight weights at once where the pointer allows it (every section starts at a multiple of
    // eight): the weights are read once per CTA, and one by one that took half of a small batch.
    static_assert(OFF_B1 % 8 == 0 && OFF_W2 % 8 == 0 && OFF_B2 % 8 == 0 && OFF_W3 % 8 == 0 && OFF_B3 % 8 == 0,
                  "eight weights lie in one section");
    auto place = [&](int p) -> float* {
        return p < OFF_B1 ? M.w1 + p
             : p < OFF_W2 ? M.b1 + (p - OFF_B1)
             : p < OFF_B2 ? M.w2 + (p - OFF_W2) / NH * W2P + (p - OFF_W2) % NH
             : p < OFF_W3 ? M.b2 + (p - OFF_B2)
             : p < OFF_B3 ? M.w3 + (p - OFF_W3) : M.b3 + (p - OFF_B3);
    };
    int done = 0;
    if (((uintptr_t)wbits & 15) == 0) {
        done = NPARAM & ~7;
#pragma unroll 4
        for (int p = threadIdx.x * 8; p < done; p += blockDim.x * 8) {
            const uint4 x = *reinterpret_cast<const uint4*>(wbits + p);
            float4* d = reinterpret_cast<float4*>(place(p));
            d[0] = make_float4(__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xFFFF0000u),
                               __uint_as_float(x.y << 16), __uint_as_float(x.y & 0xFFFF0000u));
            d[1] = make_float4(__uint_as_float(x.z << 16), __uint_as_float(x.z & 0xFFFF0000u),
                               __uint_as_float(x.w << 16), __uint_as_float(x.w & 0xFFFF0000u));
        }
    }
    for (int p = done + threadIdx.x; p < NPARAM; p += blockDim.x) *place(p) = bf16_bits_to_float(wbits[p]);
    if (threadIdx.x < NIN) {
        M.mu[threadIdx.x] = norm[threadIdx.x];
        M.isg[threadIdx.x] = 1.0f / norm[NIN + threadIdx.x];
    }
}

// Units e, e + TPS, ... of a layer for one sample: acc[t] = b[o] + sum_i w[o][i] x[i], i
// ascending in one chain per unit, so that the result does not depend on TPS.
template <int TPS, int K, int STRIDE>
__device__ __forceinline__ void mlp_layer(const float* w, const float* b, const float* x, int e,
                                          float (&acc)[NH / TPS]) {
#pragma unroll
    for (int t = 0; t < NH / TPS; ++t) acc[t] = b[t * TPS + e];
#pragma unroll 2
    for (int i = 0; i < K; i += 4) {
        const float4 xv = *reinterpret_cast<const float4*>(x + i);
#pragma unroll
        for (int t = 0; t < NH / TPS; ++t) {
            const float4 wv = *reinterpret_cast<const float4*>(w + (t * TPS + e) * STRIDE + i);
            acc[t] = fmaf(wv.x, xv.x, acc[t]);
            acc[t] = fmaf(wv.y, xv.y, acc[t]);
            acc[t] = fmaf(wv.z, xv.z, acc[t]);
            acc[t] = fmaf(wv.w, xv.w, acc[t]);
        }
    }
}

// Four threads per sample (16 units each), activations through shared memory.
// With one thread per sample every multiply-add read its weight alone: bound
// by shared-memory reads on large inputs, and on a training batch by the one
// chain of 5,248 multiply-adds per thread on a third of the SMs.
constexpr int FWD_T = 128, FWD_TPS = 4, FWD_S = FWD_T / FWD_TPS;
constexpr int HP4 = NH + 4;  // row stride of activations: 16-byte rows, four words apart in the banks

struct FwdShared {
    MlpWeights m;
    float z[FWD_S][NIN + 4];
    float h[FWD_S][HP4];
    float h2[FWD_S][HP4];
};

// Writes y (out, n x 2) and/or, when est != NULL, the size estimate
// est_j = clamp(ceil(expm1(y0) * safety), 1, min(flops, span)).
__global__ void __launch_bounds__(FWD_T) k_mlp_forward(const float* feats, int64_t n,
                                                       const uint16_t* wbits, const float* norm,
                                                       float* out, int64_t* est, float safety,
                                                       const int64_t* flops, const int32_t* rlo,
                                                       const int32_t* rhi) {
    __shared__ __align__(16) FwdShared S;
    load_weights(S.m, wbits, norm);
    __syncthreads();
    const int q = threadIdx.x / FWD_TPS, e = threadIdx.x % FWD_TPS;
    // a sample's threads are neighbours in one warp, the only one that touches its rows
    for (int64_t base = (int64_t)blockIdx.x * FWD_S; base < n; base += (int64_t)gridDim.x * FWD_S) {
        const int64_t s = base + q;
        const bool v = s < n;
#pragma unroll
        for (int i = 0; i < NIN; i += FWD_TPS)
            S.z[q][i + e] = v ? (feats[s * NIN + i + e] - S.m.mu[i + e]) * S.m.isg[i + e] : 0.0f;
        __syncwarp();
        float acc[NH / FWD_TPS];
        mlp_layer<FWD_TPS, NIN, NIN>(S.m.w1, S.m.b1, S.z[q], e, acc);
#pragma unroll
        for (int t = 0; t < NH / FWD_TPS; ++t) S.h[q][t * FWD_TPS + e] = fmaxf(acc[t], 0.0f);
        __syncwarp();
        mlp_layer<FWD_TPS, NH, W2P>(S.m.w2, S.m.b2, S.h[q], e, acc);
#pragma unroll
        for (int t = 0; t < NH / FWD_TPS; ++t) S.h2[q][t * FWD_TPS + e] = fmaxf(acc[t], 0.0f);
        __syncwarp();
        if (e < NOUT && v) {
            float y = S.m.b3[e];
#pragma unroll 4
            for (int o = 0; o < NH; o += 4) {
                const float4 wv = *reinterpret_cast<const float4*>(S.m.w3 + e * NH + o);
                const float4 hv = *reinterpret_cast<const float4*>(&S.h2[q][o]);
                y = fmaf(wv.x, hv.x, y);
                y = fmaf(wv.y, hv.y, y);
                y = fmaf(wv.z, hv.z, y);
                y = fmaf(wv.w, hv.w, y);
            }
            if (out) out[s * 2 + e] = y;
            if (est && e == 0) {
                int64_t hi = flops[s];
                const int64_t span = (int64_t)rhi[s] - rlo[s] + 1;
                if (span < hi) hi = span;
                if (hi < 1) hi = 1;
                const double x = ceil(expm1((double)fminf(y, 40.0f)) * (double)safety);
                est[s] = x < 1.0 ? 1 : (x > (double)hi ? hi : (int64_t)x);
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// backward (training)
// ---------------------------------------------------------------------------

constexpr int BWD_B = 64;            // samples per CTA
constexpr int BWD_TPS = 8;           // threads per pair of samples (8 units each)
constexpr int BWD_T = BWD_B / 2 * BWD_TPS;

struct BwdShared {
    MlpWeights m;
    float Z[BWD_B][NIN + 4];
    float H1[BWD_B][HP4];
    float H2[BWD_B][HP4];
    float D2[BWD_B][HP4];
    float D1[BWD_B][HP4];
    float DY[BWD_B][NOUT];
    double red[BWD_T / 32];
};

// mlp_layer for two samples: every weight read serves both
template <int TPS, int K, int STRIDE>
__device__ __forceinline__ void mlp_layer2(const float* w, const float* b, const float* x0, const float* x1,
                                           int e, float (&a0)[NH / TPS], float (&a1)[NH / TPS]) {
#pragma unroll
    for (int t = 0; t < NH / TPS; ++t) a0[t] = a1[t] = b[t * TPS + e];
#pragma unroll 2
    for (int i = 0; i < K; i += 4) {
        const float4 u = *reinterpret_cast<const float4*>(x0 + i), v = *reinterpret_cast<const float4*>(x1 + i);
#pragma unroll
        for (int t = 0; t < NH / TPS; ++t) {
            const float4 wv = *reinterpret_cast<const float4*>(w + (t * TPS + e) * STRIDE + i);
            a0[t] = fmaf(wv.x, u.x, a0[t]);
            a1[t] = fmaf(wv.x, v.x, a1[t]);
            a0[t] = fmaf(wv.y, u.y, a0[t]);
            a1[t] = fmaf(wv.y, v.y, a1[t]);
            a0[t] = fmaf(wv.z, u.z, a0[t]);
            a1[t] = fmaf(wv.z, v.z, a1[t]);
            a0[t] = fmaf(wv.w, u.w, a0[t]);
            a1[t] = fmaf(wv.w, v.w, a1[t]);
        }
    }
}

// Gradient of (scale * sum over samples and outputs of (y - t)^2) with
// respect to the (BF16-valued) weights, added into grad; the loss sum
// (unscaled) is added into *loss.
//
// Eight threads per pair of samples for the two passes over the layers (bound
// by the shared-memory reads of the weights: one read serves both samples),
// then the CTA's weight gradients as register tiles (16 of W2 per thread:
// eight words read per sample for 16 multiply-adds).  A thread per sample with
// its activations in shared memory left two warps on an SM: latency-bound,
// 74 us at 8,192 samples; eight threads per sample took 29.
__global__ void __launch_bounds__(BWD_T) k_mlp_backward(const float* feats, const float* targets,
                                                        int64_t n, const uint16_t* wbits,
                                                        const float* norm, float scale,
                                                        float* grad, double* loss) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdShared& S = *reinterpret_cast<BwdShared*>(smem_raw);
    const int tid = threadIdx.x, q = tid / BWD_TPS * 2, e = tid % BWD_TPS;
    load_weights(S.m, wbits, norm);
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * BWD_B + q;
    constexpr int U = NH / BWD_TPS;
    bool v[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        v[p] = s + p < n;
#pragma unroll
        for (int i = 0; i < NIN; i += BWD_TPS)
            S.Z[q + p][i + e] =
                v[p] ? (feats[(s + p) * NIN + i + e] - S.m.mu[i + e]) * S.m.isg[i + e] : 0.0f;
    }
    __syncwarp();
    float acc[2][U];
    mlp_layer2<BWD_TPS, NIN, NIN>(S.m.w1, S.m.b1, S.Z[q], S.Z[q + 1], e, acc[0], acc[1]);
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int t = 0; t < U; ++t) S.H1[q + p][t * BWD_TPS + e] = v[p] ? fmaxf(acc[p][t], 0.0f) : 0.0f;
    __syncwarp();
    mlp_layer2<BWD_TPS, NH, W2P>(S.m.w2, S.m.b2, S.H1[q], S.H1[q + 1], e, acc[0], acc[1]);
    double lsum = 0.0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int o = t * BWD_TPS + e;
            const float h2 = fmaxf(acc[p][t], 0.0f);
            S.H2[q + p][o] = v[p] ? h2 : 0.0f;
            y0 = fmaf(S.m.w3[o], h2, y0);
            y1 = fmaf(S.m.w3[NH + o], h2, y1);
        }
#pragma unroll
        for (int o = BWD_TPS / 2; o > 0; o >>= 1) {
            y0 += __shfl_xor_sync(FULL, y0, o);
            y1 += __shfl_xor_sync(FULL, y1, o);
        }
        y0 += S.m.b3[0];
        y1 += S.m.b3[1];
        const float e0 = v[p] ? y0 - targets[(s + p) * 2] : 0.0f, e1 = v[p] ? y1 - targets[(s + p) * 2 + 1] : 0.0f;
        if (e == 0) lsum += (double)e0 * e0 + (double)e1 * e1;
        const float d0 = 2.0f * e0 * scale, d1 = 2.0f * e1 * scale;
        if (e == 0) {
            S.DY[q + p][0] = d0;
            S.DY[q + p][1] = d1;
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int o = t * BWD_TPS + e;
            S.D2[q + p][o] = acc[p][t] > 0.0f ? d0 * S.m.w3[o] + d1 * S.m.w3[NH + o] : 0.0f;
        }
    }
    __syncwarp();
    {  // D1 of units 8 e .. 8 e + 7
        float g[2][U];
#pragma unroll
        for (int t = 0; t < U; ++t) g[0][t] = g[1][t] = 0.0f;
#pragma unroll 4
        for (int o = 0; o < NH; ++o) {
            const float da = S.D2[q][o], db = S.D2[q + 1][o];
#pragma unroll
            for (int t = 0; t < U; t += 4) {
                const float4 wv = *reinterpret_cast<const float4*>(S.m.w2 + o * W2P + e * U + t);
                g[0][t] = fmaf(da, wv.x, g[0][t]);
                g[0][t + 1] = fmaf(da, wv.y, g[0][t + 1]);
                g[0][t + 2] = fmaf(da, wv.z, g[0][t + 2]);
                g[0][t + 3] = fmaf(da, wv.w, g[0][t + 3]);
                g[1][t] = fmaf(db, wv.x, g[1][t]);
                g[1][t + 1] = fmaf(db, wv.y, g[1][t + 1]);
                g[1][t + 2] = fmaf(db, wv.z, g[1][t + 2]);
                g[1][t + 3] = fmaf(db, wv.w, g[1][t + 3]);
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int t = 0; t < U; ++t)
                S.D1[q + p][e * U + t] = S.H1[q + p][e * U + t] > 0.0f ? g[p][t] : 0.0f;
    }
    lsum = warp_sum(lsum);
    if ((tid & 31) == 0) S.red[tid >> 5] = lsum;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < BWD_T / 32; ++w) t += S.red[w];
        atomicAdd(loss, t);
    }
    // weight gradients: sums over the CTA's samples
    {
        const int o = tid / 16 * 4, i = tid % 16 * 4;  // W2: units o .. o + 3, inputs i .. i + 3
        float g[4][4] = {};
#pragma unroll 4
        for (int b = 0; b < BWD_B; ++b) {
            const float4 dv = *reinterpret_cast<const float4*>(&S.D2[b][o]);
            const float4 hv = *reinterpret_cast<const float4*>(&S.H1[b][i]);
            const float d4[4] = {dv.x, dv.y, dv.z, dv.w}, h4[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) g[r][c] = fmaf(d4[r], h4[c], g[r][c]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicAdd(grad + OFF_W2 + (o + r) * NH + i + c, g[r][c]);
    }
    {
        const int o = tid / 4, i = tid % 4 * 4;  // W1: unit o, inputs i .. i + 3
        float g[4] = {};
#pragma unroll 4
        for (int b = 0; b < BWD_B; ++b) {
            const float dd = S.D1[b][o];
            const float4 zv = *reinterpret_cast<const float4*>(&S.Z[b][i]);
            g[0] = fmaf(dd, zv.x, g[0]);
            g[1] = fmaf(dd, zv.y, g[1]);
            g[2] = fmaf(dd, zv.z, g[2]);
            g[3] = fmaf(dd, zv.w, g[3]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) atomicAdd(grad + OFF_W1 + o * NIN + i + c, g[c]);
    }
    static_assert(BWD_T == NH / 4 * (NH / 4) && BWD_T == NH * NIN / 4, "one tile per thread");
    for (int k = tid; k < 2 * NH + NOUT * NH + NOUT; k += BWD_T) {  // b1, b2, W3, b3
        float g = 0.0f;
        int p;
        if (k < NH) {
            p = OFF_B1 + k;
            for (int b = 0; b < BWD_B; ++b) g += S.D1[b][k];
        } else if (k < 2 * NH) {
            p = OFF_B2 + k - NH;
            for (int b = 0; b < BWD_B; ++b) g += S.D2[b][k - NH];
        } else if (k < 2 * NH + NOUT * NH) {
            const int o = (k - 2 * NH) / NH, i = k % NH;
            p = OFF_W3 + o * NH + i;
            for (int b = 0; b < BWD_B; ++b) g = fmaf(S.DY[b][o], S.H2[b][i], g);
        } else {
            const int o = k - 2 * NH - NOUT * NH;
            p = OFF_B3 + o;
            for (int b = 0; b < BWD_B; ++b) g += S.DY[b][o];
        }
        atomicAdd(grad + p, g);
    }
}

// Adam step on the FP32 master weights; writes their BF16 rounding.
__global__ void k_adam(float* master, float* m, float* v, const float* grad, int64_t step, float lr,
                       float b1, float b2, float eps, uint16_t* wbits) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NPARAM) return;
    const float g = grad[p];
    const float mm = b1 * m[p] + (1.0f - b1) * g;
    const float vv = b2 * v[p] + (1.0f - b2) * g * g;
    m[p] = mm;
    v[p] = vv;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    const float w = master[p] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    master[p] = w;
    wbits[p] = __bfloat16_as_ushort(__float2bfloat16_rn(w));
}

// log cf_j = log(flops_j / max(nnz_j, 1)) from the last numeric pass (input
// to the next iteration's features).
__global__ void k_logcf(int32_t n, const int64_t* flops, const int64_t* bnnz, float* logcf) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int64_t z = bnnz[j] > 0 ? bnnz[j] : 1;
    logcf[j] = flops[j] > 0 ? logf((float)((double)flops[j] / (double)z)) : 0.0f;
}

void launch_colmax_features(const CscView& A, int32_t iteration, const float* prev_logcf,
                            float* colmax, float* feats, cudaStream_t s, const int32_t* iter_dev) {
    if (A.n == 0) return;
    int64_t blocks = ((int64_t)A.n * 32 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_colmax<<<(unsigned)blocks, 256, 0, s>>>(A, colmax);
    count_launches(1);
    // columns per warp: a full warp of them once that still fills the GPU (152 SMs x 32 warps)
    int64_t group = A.n / (152 * 32);
    group = group < 1 ? 1 : (group > 32 ? 32 : group);
    int64_t fb = ((A.n + group - 1) / group * 32 + 255) / 256;
    if (fb > 152 * 16) fb = 152 * 16;
    k_features<<<(unsigned)fb, 256, 0, s>>>(A, iteration, iter_dev, prev_logcf, colmax, feats, (int)group);
    count_launches(1);
}

void launch_mlp_forward(const float* feats, int64_t n, const uint16_t* wbits, const float* norm,
                        float* out, int64_t* est, float safety, const int64_t* flops,
                        const int32_t* rlo, const int32_t* rhi, cudaStream_t s) {
    if (n == 0) return;
    int64_t blocks = (n + FWD_S - 1) / FWD_S;
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_mlp_forward<<<(unsigned)blocks, FWD_T, 0, s>>>(feats, n, wbits, norm, out, est, safety,
                                                      flops, rlo, rhi);
    count_launches(1);
}

void launch_mlp_backward(const float* feats, const float* targets, int64_t n,
                         const uint16_t* wbits, const float* norm, float scale, float* grad,
                         double* loss, cudaStream_t s) {
    if (n == 0) return;
    const size_t smem = sizeof(BwdShared);
    cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t blocks = (n + BWD_B - 1) / BWD_B;
    k_mlp_backward<<<(unsigned)blocks, BWD_T, smem, s>>>(feats, targets, n, wbits, norm, scale,
                                                          grad, loss);
    count_launches(1);
}

void launch_adam(float* master, float* m, float* v, const float* grad, int64_t step, float lr,
                 float b1, float b2, float eps, uint16_t* wbits, cudaStream_t s) {
    k_adam<<<(NPARAM + 255) / 256, 256, 0, s>>>(master, m, v, grad, step, lr, b1, b2, eps, wbits);
    count_launches(1);
}

__global__ void k_iter_bump(int32_t* it) {
    if (threadIdx.x == 0) ++*it;
}

void launch_iter_bump(int32_t* it, cudaStream_t s) {
    k_iter_bump<<<1, 32, 0, s>>>(it);
    count_launches(1);
}

void launch_logcf(int32_t n, const int64_t* flops, const int64_t* bnnz, float* logcf,
                  cudaStream_t s) {
    if (n == 0) return;
    k_logcf<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, flops, bnnz, logcf);
    count_launches(1);
}

}  // namespace mcl
