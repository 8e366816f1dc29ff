// Learned rate controller, network side: the 80 features, input
// normalisation, forward pass, back-propagation with deterministic
// (fixed-order) minibatch sums, and Adam.  The network is tiny (9409
// parameters), so it runs on plain FMA units: one warp per sample for
// inference, one cluster of 16 CTAs for a run of training steps; single
// gradients and the smallest and largest batches use one warp per minibatch
// row for the forward and delta pass and one thread per parameter for the
// gradient sums (in tiles that stage the minibatch in shared memory) and the
// update.
#include <cmath>
#include <cstring>

#include <cuda_bf16.h>

#include "host_common.h"

namespace dctgb {

constexpr int kIn = DCT_MLP_INPUTS, kHid = DCT_MLP_HIDDEN, kParams = DCT_MLP_PARAMS;
constexpr int oW1 = 0, oB1 = kHid * kIn, oW2 = oB1 + kHid, oB2 = oW2 + kHid * kHid, oW3 = oB2 + kHid,
              oB3 = oW3 + kHid;
static_assert(oB3 + 1 == kParams, "parameter layout");
static_assert(oW1 % 4 == 0 && oW2 % 4 == 0 && kIn % 4 == 0 && kHid % 4 == 0, "16-byte weight rows");

// per-sample cache (floats): xn[80] a1[64] h1[64] a2[64] h2[64] da2[64]
// da1[64] y dz, every vector 16-byte aligned (the row is 468 floats)
constexpr int cXn = 0, cA1 = cXn + kIn, cH1 = cA1 + kHid, cA2 = cH1 + kHid, cH2 = cA2 + kHid, cDa2 = cH2 + kHid,
              cDa1 = cDa2 + kHid, cY = cDa1 + kHid, cDz = cY + 1, kCache = ((cDz + 1 + 3) / 4) * 4;
static_assert(cH1 % 4 == 0 && cH2 % 4 == 0 && cDa2 % 4 == 0 && cDa1 % 4 == 0 && kCache % 4 == 0, "cache alignment");

__device__ __forceinline__ float gelu(float a) { return 0.5f * a * (1.0f + erff(a * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float a) {
    return 0.5f * (1.0f + erff(a * 0.70710678118654752f)) + a * expf(-0.5f * a * a) * 0.39894228040143268f;
}
__device__ __forceinline__ float act(float h, int bf16) {
    return bf16 ? __bfloat162float(__float2bfloat16_rn(h)) : h;
}

// Inference, one warp per sample: lane l owns hidden units l and l + 32 of both
// layers, every sum over its inputs in ascending order (the inputs a lane does
// not hold come by shuffle).  W1 and W2 are staged transposed with rows padded
// to 65 floats, as in k_mlp_delta.  One thread per sample took 219 us for the
// 48 frames of a small rate-control call (a serial walk over 9,409 parameters
// in global memory); this takes 10 us.
constexpr int kFwdRows = 8;                    // samples (warps) per CTA
constexpr int kTStride = kHid + 1;             // padded row of a transposed weight matrix

__global__ void __launch_bounds__(kFwdRows * 32)
k_mlp_forward(const float* __restrict__ P, const float* __restrict__ feats, const float* __restrict__ mean,
              const float* __restrict__ stdv, int bf16, int n, float* __restrict__ y_out, int* __restrict__ q_out) {
    __shared__ float w1t[kIn * kTStride];       // w1t[i * 65 + j] = W1[j][i]
    __shared__ float w2t[kHid * kTStride];
#pragma unroll 8
    for (int e = threadIdx.x; e < kHid * kIn; e += kFwdRows * 32) w1t[(e % kIn) * kTStride + e / kIn] = P[oW1 + e];
#pragma unroll 8
    for (int e = threadIdx.x; e < kHid * kHid; e += kFwdRows * 32) w2t[(e % kHid) * kTStride + e / kHid] = P[oW2 + e];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int s = blockIdx.x * kFwdRows + (threadIdx.x >> 5); s < n; s += gridDim.x * kFwdRows) {   // warp-uniform
        const float* x = feats + (size_t)s * kIn;
        float xn[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int i = lane + 32 * k;
            xn[k] = i < kIn ? (x[i] - mean[i]) / stdv[i] : 0.0f;
        }
        float a[2], h[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) a[k] = P[oB1 + lane + 32 * k];
#pragma unroll
        for (int i = 0; i < kIn; ++i) {
            const float v = __shfl_sync(0xffffffffu, xn[i >> 5], i & 31);
#pragma unroll
            for (int k = 0; k < 2; ++k) a[k] = fmaf(w1t[i * kTStride + lane + 32 * k], v, a[k]);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            h[k] = act(gelu(a[k]), bf16);
            a[k] = P[oB2 + lane + 32 * k];
        }
#pragma unroll
        for (int i = 0; i < kHid; ++i) {
            const float v = __shfl_sync(0xffffffffu, h[i >> 5], i & 31);
#pragma unroll
            for (int k = 0; k < 2; ++k) a[k] = fmaf(w2t[i * kTStride + lane + 32 * k], v, a[k]);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) h[k] = act(gelu(a[k]), bf16);
        const float w3[2] = {P[oW3 + lane], P[oW3 + lane + 32]};
        float z = P[oB3];
#pragma unroll
        for (int j = 0; j < kHid; ++j)
            z = fmaf(__shfl_sync(0xffffffffu, w3[j >> 5], j & 31), __shfl_sync(0xffffffffu, h[j >> 5], j & 31), z);
        const float y = 1.0f / (1.0f + expf(-z));
        if (lane == 0) {
            if (y_out) y_out[s] = y;
            if (q_out) {
                const float q = rintf(1.0f + 99.0f * y);
                q_out[s] = (int)fminf(100.0f, fmaxf(1.0f, q));
            }
        }
    }
}

// forward + output delta + hidden deltas of one minibatch row per warp:
// lane l owns hidden units l and l + 32 of both layers; every sum runs over
// its inputs in ascending order as k_mlp_forward's does (the inputs a lane
// does not hold come by shuffle), so the cache holds the same values.  The
// CTA first stages W1 and W2 transposed in shared memory with rows padded
// to 65 floats: the forward sums read W^T[i][lane] and the backward sum
// reads W2[j][lane] = W2^T[lane][j], both free of bank conflicts (reading
// W1 straight from global memory touched 32 cache lines per warp access).
constexpr int kDeltaRows = 8;                  // minibatch rows (warps) per CTA

__global__ void __launch_bounds__(kDeltaRows * 32)
k_mlp_delta(const float* __restrict__ P, const float* __restrict__ feats, const float* __restrict__ labels,
            const int* __restrict__ index, const float* __restrict__ mean, const float* __restrict__ stdv, int bf16,
            int batch, float* __restrict__ cache) {
    __shared__ float w1t[kIn * kTStride];       // w1t[i * 65 + j] = W1[j][i]
    __shared__ float w2t[kHid * kTStride];      // w2t[i * 65 + j] = W2[j][i]
    {
        // 16-byte loads along the rows of W1 and W2 (both start 16-byte
        // aligned), all issued before the first shared-memory store
        constexpr int n1 = kHid * kIn / 4, n2 = kHid * kHid / 4, nv = n1 + n2;
        constexpr int per = (nv + kDeltaRows * 32 - 1) / (kDeltaRows * 32);
        const float4* P4 = reinterpret_cast<const float4*>(P);
        float4 v[per];
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int e = threadIdx.x + u * kDeltaRows * 32;
            if (e < n1) v[u] = P4[oW1 / 4 + e];
            else if (e < nv) v[u] = P4[oW2 / 4 + e - n1];
        }
#pragma unroll
        for (int u = 0; u < per; ++u) {
            const int e = threadIdx.x + u * kDeltaRows * 32;
            if (e < n1) {
                const int j = (4 * e) / kIn, i = 4 * e - j * kIn;
                w1t[(i + 0) * kTStride + j] = v[u].x;
                w1t[(i + 1) * kTStride + j] = v[u].y;
                w1t[(i + 2) * kTStride + j] = v[u].z;
                w1t[(i + 3) * kTStride + j] = v[u].w;
            } else if (e < nv) {
                const int f = 4 * (e - n1), j = f / kHid, i = f - j * kHid;
                w2t[(i + 0) * kTStride + j] = v[u].x;
                w2t[(i + 1) * kTStride + j] = v[u].y;
                w2t[(i + 2) * kTStride + j] = v[u].z;
                w2t[(i + 3) * kTStride + j] = v[u].w;
            }
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= batch) return;                                   // warp-uniform, after the only barrier
    const int s = index[b];
    float* c = cache + (size_t)b * kCache;
    const float* x = feats + (size_t)s * kIn;
    float xn[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = lane + 32 * k;
        xn[k] = i < kIn ? (x[i] - mean[i]) / stdv[i] : 0.0f;
        if (i < kIn) c[cXn + i] = xn[k];
    }
    // layer 1
    float a1[2], h1[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) a1[k] = P[oB1 + lane + 32 * k];
    for (int i = 0; i < kIn; ++i) {
        const float v = __shfl_sync(0xffffffffu, xn[i >> 5], i & 31);
#pragma unroll
        for (int k = 0; k < 2; ++k) a1[k] = fmaf(w1t[i * kTStride + lane + 32 * k], v, a1[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        h1[k] = act(gelu(a1[k]), bf16);
        c[cA1 + lane + 32 * k] = a1[k];
        c[cH1 + lane + 32 * k] = h1[k];
    }
    // layer 2
    float a2[2], h2[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) a2[k] = P[oB2 + lane + 32 * k];
    for (int i = 0; i < kHid; ++i) {
        const float v = __shfl_sync(0xffffffffu, h1[i >> 5], i & 31);
#pragma unroll
        for (int k = 0; k < 2; ++k) a2[k] = fmaf(w2t[i * kTStride + lane + 32 * k], v, a2[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        h2[k] = act(gelu(a2[k]), bf16);
        c[cA2 + lane + 32 * k] = a2[k];
        c[cH2 + lane + 32 * k] = h2[k];
    }
    // output, in the same order on every lane
    float z = P[oB3];
    for (int j = 0; j < kHid; ++j) z = fmaf(P[oW3 + j], __shfl_sync(0xffffffffu, h2[j >> 5], j & 31), z);
    const float y = 1.0f / (1.0f + expf(-z));
    const float dz = 2.0f * (y - labels[s]) / (float)batch * y * (1.0f - y);
    if (lane == 0) {
        c[cY] = y;
        c[cDz] = dz;
    }
    float da2[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        da2[k] = dz * P[oW3 + lane + 32 * k] * gelu_grad(a2[k]);
        c[cDa2 + lane + 32 * k] = da2[k];
    }
    float s2[2] = {0.0f, 0.0f};
    for (int j = 0; j < kHid; ++j) {
        const float d = __shfl_sync(0xffffffffu, da2[j >> 5], j & 31);
#pragma unroll
        for (int k = 0; k < 2; ++k) s2[k] = fmaf(d, w2t[(lane + 32 * k) * kTStride + j], s2[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) c[cDa1 + lane + 32 * k] = s2[k] * gelu_grad(a1[k]);
}

// Per-parameter minibatch sums, one output per thread, each over the rows
// in ascending order (deterministic).  CTAs 0..15 own the W1 gradients of
// four hidden units (320 outputs), CTAs 16..31 the W2 gradients of four
// units (256), CTA 32 the b1 sums, CTA 33 the b2 sums and CTA 34 the W3 and
// b3 sums and the loss.  Each CTA stages the cache columns it needs for
// kGradRows rows at a time in shared memory (contiguous reads), then every
// thread runs its sum over the staged rows.
constexpr int kGradUnits = 4;
constexpr int kGradRows = 128;
constexpr int kW1Tiles = kHid / kGradUnits, kW2Tiles = kHid / kGradUnits;
constexpr int kGradCtas = kW1Tiles + kW2Tiles + 3;
constexpr int kGradThreads = kGradUnits * kIn;               // the widest tile
static_assert(kHid % kGradUnits == 0 && kGradThreads >= kHid + 2, "gradient tiling");

// Adam step for one parameter (k_adam and the fused gradient kernel)
struct AdamArgs {
    float* P;
    float* m;
    float* v;
    float lr, b1, b2, eps, c1, c2;
};

// The fused multiply-adds are written out so that every kernel that inlines
// this rounds alike.
__device__ __forceinline__ void adam_step(const AdamArgs& a, float& P, float& m, float& v, float gi) {
    m = fmaf(1.0f - a.b1, gi, __fmul_rn(a.b1, m));
    v = fmaf(__fmul_rn(1.0f - a.b2, gi), gi, __fmul_rn(a.b2, v));
    P = __fsub_rn(P, __fdiv_rn(__fmul_rn(a.lr, __fmul_rn(m, a.c1)), __fadd_rn(__fsqrt_rn(__fmul_rn(v, a.c2)), a.eps)));
}
__device__ __forceinline__ void adam_update(const AdamArgs& a, int p, float gi) {
    adam_step(a, a.P[p], a.m[p], a.v[p], gi);
}

// ADAM: also apply the Adam step to each parameter as soon as its sum is
// final (each parameter belongs to one thread; nothing in this kernel reads
// the parameters), saving the separate update launch of a training step.
template <bool ADAM>
__global__ void __launch_bounds__(kGradThreads)
k_mlp_grad(const float* __restrict__ cache, const float* __restrict__ labels, const int* __restrict__ index,
           int batch, float* __restrict__ grad, float* __restrict__ loss, AdamArgs adam) {
    __shared__ __align__(16) float sm[kGradRows * (kGradUnits + kIn)];
    const int t = threadIdx.x;
    const int blk = blockIdx.x;
    // the staged row: `ncol` floats (a multiple of 4) = na float4 from cache
    // column ca, then nb float4 from column cb; the last CTA's rows end with
    // (dz, y - label, 0, 0)
    int ncol, ca, na, cb, nb;
    const bool last = blk == kW1Tiles + kW2Tiles + 2;
    if (blk < kW1Tiles) {
        ca = cDa1 + kGradUnits * blk; na = kGradUnits / 4; cb = cXn; nb = kIn / 4;
    } else if (blk < kW1Tiles + kW2Tiles) {
        ca = cDa2 + kGradUnits * (blk - kW1Tiles); na = kGradUnits / 4; cb = cH1; nb = kHid / 4;
    } else if (blk == kW1Tiles + kW2Tiles) {
        ca = cDa1; na = kHid / 4; cb = 0; nb = 0;
    } else if (blk == kW1Tiles + kW2Tiles + 1) {
        ca = cDa2; na = kHid / 4; cb = 0; nb = 0;
    } else {
        ca = cH2; na = kHid / 4; cb = 0; nb = 0;
    }
    const int nv = na + nb + (last ? 1 : 0);
    ncol = 4 * nv;
    float4* sm4 = reinterpret_cast<float4*>(sm);
    const float4* cache4 = reinterpret_cast<const float4*>(cache);
    float g = 0.0f;
    for (int r0 = 0; r0 < batch; r0 += kGradRows) {
        const int rows = min(kGradRows, batch - r0);
        const int total = rows * nv;
        __syncthreads();
        // 16-byte loads, eight in flight per thread before the stores
        for (int e0 = t; e0 < total; e0 += 8 * kGradThreads) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int e = e0 + u * kGradThreads;
                if (e < total) {
                    const int r = e / nv, k = e - r * nv;
                    const size_t row4 = (size_t)(r0 + r) * (kCache / 4);
                    if (k < na) {
                        v[u] = cache4[row4 + ca / 4 + k];
                    } else if (k < na + nb) {
                        v[u] = cache4[row4 + cb / 4 + k - na];
                    } else {
                        const float* row = cache + (size_t)(r0 + r) * kCache;
                        v[u] = make_float4(row[cDz], row[cY] - labels[index[r0 + r]], 0.0f, 0.0f);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int e = e0 + u * kGradThreads;
                if (e < total) sm4[e] = v[u];
            }
        }
        __syncthreads();
        if (blk < kW1Tiles + kW2Tiles) {
            const int nin = blk < kW1Tiles ? kIn : kHid;
            if (t < kGradUnits * nin) {
                const int u = t / nin, i = t - u * nin;
                for (int r = 0; r < rows; ++r) g = fmaf(sm[r * ncol + u], sm[r * ncol + kGradUnits + i], g);
            }
        } else if (blk < kW1Tiles + kW2Tiles + 2) {
            if (t < kHid)
                for (int r = 0; r < rows; ++r) g += sm[r * ncol + t];
        } else if (t < kHid) {                           // W3
            for (int r = 0; r < rows; ++r) g = fmaf(sm[r * ncol + kHid], sm[r * ncol + t], g);
        } else if (t == kHid) {                          // b3
            for (int r = 0; r < rows; ++r) g += sm[r * ncol + kHid];
        } else if (t == kHid + 1) {                      // loss
            for (int r = 0; r < rows; ++r) {
                const float d = sm[r * ncol + kHid + 1];
                g = fmaf(d, d, g);
            }
        }
    }
    int p = -1;
    if (blk < kW1Tiles) {
        if (t < kGradUnits * kIn) p = oW1 + (kGradUnits * blk) * kIn + t;
    } else if (blk < kW1Tiles + kW2Tiles) {
        if (t < kGradUnits * kHid) p = oW2 + (kGradUnits * (blk - kW1Tiles)) * kHid + t;
    } else if (blk == kW1Tiles + kW2Tiles) {
        if (t < kHid) p = oB1 + t;
    } else if (blk == kW1Tiles + kW2Tiles + 1) {
        if (t < kHid) p = oB2 + t;
    } else if (t < kHid) {
        p = oW3 + t;
    } else if (t == kHid) {
        p = oB3;
    } else if (t == kHid + 1) {
        *loss = g / (float)batch;
    }
    if (p >= 0) {
        grad[p] = g;
        if (ADAM) adam_update(adam, p, g);
    }
}

__global__ void k_adam(AdamArgs a, const float* __restrict__ g) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kParams) return;
    adam_update(a, p, g[p]);
}

// ---------------------------------------------------------------------------
// A run of training steps in one launch: one cluster of 16 CTAs
// ---------------------------------------------------------------------------
// A step of k_mlp_delta and k_mlp_grad is bound by latency, not by work (5.8
// million multiply-adds): two dependent launches, the weights staged anew and
// the cache columns fetched by few CTAs cost 24 us.  Here a cluster stays on 16
// SMs for all steps.  Every CTA holds all weights, as 16 records of one owner's
// four hidden units each.  Phase F: CTA c runs rows 16c..16c+15 of a group of
// 256 through forward and deltas (a warp takes 32 units of 4 rows, so a weight
// is loaded once for four rows).  All CTAs need all rows' inputs and first-layer
// outputs: each CTA writes its rows to global memory and has them multicast to
// the cluster while the rest of phase F runs (one copy per receiver instead, or
// every CTA fetching all rows from L2, both moved about 12 bytes per clock and
// SM: 13,000 clocks a step).  The deltas of the units a CTA owns go to it in one
// bulk copy between shared memories.  Phase G: CTA c sums its units' gradients
// over the rows in ascending order, applies Adam to parameters it keeps in
// registers and multicasts its record.  Every copy is counted by the
// receiver's mbarrier; a CTA that holds all 16 new records knows that every CTA
// has finished its sums, so the buffers it sends into next are free, and no
// other barrier is needed.  The inputs of the next rows load while phase G
// runs.  All sums and updates have the operands and order of the two kernels:
// the same bits.  16,000 rows, batch 256 (63 steps): 770 us an epoch against
// 1540 us.
constexpr int kCluster = 16;
constexpr int kEpochThreads = 512;
constexpr int kOwned = kHid / kCluster;                // hidden units a CTA owns per layer
constexpr int kGroupRows = 256;                        // rows in flight
constexpr int kCtaRows = kGroupRows / kCluster;
constexpr int kEpochSteps = 64;                        // steps per launch
// Smaller batches have no room in the workspace for the cluster's exchange
// area, larger ones fill the GPU with the two kernels.
constexpr int kEpochMinBatch = 64, kEpochMaxBatch = 1024;
static_assert(kOwned == 4 && kCtaRows == 16 && kIn % 4 == 0, "phases F and G index by fours");

// One owner's weights: W1 rows (80, padded to 81), W2 rows (64, padded to 65),
// b1, b2, W3 of its four units and (owner 0) b3.  With 604 floats a record,
// lane u reading its unit's W1 or W2 row hits bank (28 (u / 4) + 17 or 1 (u % 4))
// mod 32: all 32 distinct.
constexpr int kW1Row = kIn + 1, kW2Row = kHid + 1;
constexpr int rW2 = kOwned * kW1Row, rB1 = rW2 + kOwned * kW2Row, rB2 = rB1 + 4, rW3 = rB2 + 4, rB3 = rW3 + 4,
              kRecord = 604;
static_assert(rB3 + 1 <= kRecord && rB1 % 4 == 0 && kRecord % 4 == 0, "record layout");

struct EpochArgs {
    float *P, *m, *v;
    const float *feats, *labels;
    const int* order;                 // of the first step's first row
    const float *mean, *stdv;
    float* loss;                      // of the first step
    float* exch;                      // kCluster * kExch floats
    int bf16, n, batch, nsteps;       // n rows left from the first step on
    float lr, b1, b2, eps;
    float c1[kEpochSteps], c2[kEpochSteps];
};

// What one CTA's 16 rows hold for one receiver: da1, da2, h2 of the
// receiver's units and (y, dz, y - label, 0).
struct __align__(16) Deltas {
    float d1[kCtaRows][4], d2[kCtaRows][4], h2[kCtaRows][4], z[kCtaRows][4];
};
// A CTA's part of the exchange area: its rows' inputs and h1, its record.
constexpr int xH1 = kCtaRows * kIn, xRec = xH1 + kCtaRows * kHid, kExch = xRec + kRecord;
static_assert(kCluster * kExch <= kEpochMinBatch * kCache + 2 * kParams, "the exchange area fits the workspace");

struct __align__(16) EpochSmem {
    float w[kCluster * kRecord];               // all weights
    float gx[kGroupRows][kIn], gh[kGroupRows][kHid];   // received: inputs and h1 of 256 rows
    Deltas gd[kCluster];                       // received, by sender
    float x[kCtaRows][kIn], h1[kCtaRows][kHid];        // this CTA's rows
    Deltas sd[kCluster];                       // to send, by receiver
    unsigned long long bar[2];                 // rows, records
    int failed;                                // a wait ran out (the losses become NaN)
};
static_assert(sizeof(EpochSmem) <= 232448, "shared memory of one CTA");
constexpr unsigned kRowBytes = (kCtaRows * (kIn + kHid)) * 4 + sizeof(Deltas);   // one CTA's rows to one receiver

__device__ __forceinline__ unsigned sm_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
}
// Bulk copy of `bytes` from this CTA's shared memory to the same or another
// place (dst: an address in this CTA's window) in CTA `rank`, counted on the
// receiver's copy of mbarrier `bar`.
__device__ __forceinline__ void send(unsigned rank, void* dst, const void* src, unsigned bytes, void* bar) {
    unsigned d, b;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(sm_addr(dst)), "r"(rank));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(sm_addr(bar)), "r"(rank));
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d),
                 "r"(sm_addr(src)), "r"(bytes), "r"(b)
                 : "memory");
}
// Bulk copy from global memory to `dst` in every CTA of the cluster, counted on
// each one's mbarrier `bar`.
__device__ __forceinline__ void multicast(void* dst, const void* src, unsigned bytes, void* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.multicast::cluster [%0], [%1], %2, [%3], %4;" ::"r"(
            sm_addr(dst)),
        "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(sm_addr(bar)), "h"((unsigned short)0xFFFF)
        : "memory");
}
// Waits for the phase of `parity` of a mbarrier, for at most about a second.
__device__ __forceinline__ bool wait_bar(const void* bar, unsigned parity) {
    const long long t0 = clock64();
    unsigned ok;
    do {
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(sm_addr(bar)), "r"(parity)
                     : "memory");
    } while (!ok && clock64() - t0 < 2000000000ll);
    return ok != 0;
}
__device__ __forceinline__ void expect_bytes(void* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(sm_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;" ::: "memory"); }

// acc[r] += w x[r] over N inputs in ascending order for four rows; x(r, i)
// gives four inputs of a row, w(i) one weight.
template <int N, typename X, typename W>
__device__ __forceinline__ void dot4(float (&acc)[4], X in, W w) {
#pragma unroll 5
    for (int i = 0; i < N; i += 4) {
        float4 x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(in(r, i));
        const float w0 = w(i), w1 = w(i + 1), w2 = w(i + 2), w3 = w(i + 3);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fmaf(w0, x[r].x, acc[r]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fmaf(w1, x[r].y, acc[r]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fmaf(w2, x[r].z, acc[r]);
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fmaf(w3, x[r].w, acc[r]);
    }
}

// g[u] += d(r)[u] x[r] over `rows` rows in ascending order, eight loaded ahead;
// d(r) gives the four deltas of row r.
template <int LD, typename D>
__device__ __forceinline__ void grad4(float (&g)[4], const float* x, int rows, D d) {
    int r = 0;
    for (; r + 8 <= rows; r += 8) {
        float xv[8];
        float4 dv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            xv[k] = x[(r + k) * LD];
            dv[k] = *reinterpret_cast<const float4*>(d(r) + 4 * k);      // eight rows of one sender
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            g[0] = fmaf(dv[k].x, xv[k], g[0]);
            g[1] = fmaf(dv[k].y, xv[k], g[1]);
            g[2] = fmaf(dv[k].z, xv[k], g[2]);
            g[3] = fmaf(dv[k].w, xv[k], g[3]);
        }
    }
    for (; r < rows; ++r) {
        const float4 dv = *reinterpret_cast<const float4*>(d(r));
        g[0] = fmaf(dv.x, x[r * LD], g[0]);
        g[1] = fmaf(dv.y, x[r * LD], g[1]);
        g[2] = fmaf(dv.z, x[r * LD], g[2]);
        g[3] = fmaf(dv.w, x[r * LD], g[3]);
    }
}

__global__ void __launch_bounds__(kEpochThreads, 1) k_mlp_epoch(const __grid_constant__ EpochArgs a) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    EpochSmem& S = *reinterpret_cast<EpochSmem*>(smem_raw);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = blockIdx.x;                               // one cluster: CTA rank = block index
    for (int e = t; e < kHid * kIn; e += kEpochThreads) {
        const int u = e / kIn, i = e - u * kIn;
        S.w[(u >> 2) * kRecord + (u & 3) * kW1Row + i] = a.P[oW1 + e];
    }
    for (int e = t; e < kHid * kHid; e += kEpochThreads) {
        const int u = e / kHid, i = e - u * kHid;
        S.w[(u >> 2) * kRecord + rW2 + (u & 3) * kW2Row + i] = a.P[oW2 + e];
    }
    if (t < kHid) {
        float* r = S.w + (t >> 2) * kRecord + (t & 3);
        r[rB1] = a.P[oB1 + t];
        r[rB2] = a.P[oB2 + t];
        r[rW3] = a.P[oW3 + t];
    }
    if (t == 0) {
        S.w[rB3] = a.P[oB3];
        S.failed = 0;
        for (int k = 0; k < 2; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_addr(&S.bar[k])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    float* const exch = a.exch + (size_t)rank * kExch;

    // owned parameters, in registers for the whole run: threads 0..79 column t
    // of W1 (four units), 96..159 column t - 96 of W2, the first lanes of warps
    // 5..8 b1, b2, W3 and (CTA 0) b3, lane 0 of warp 9 the loss (each its own
    // warp: as branches of one warp they would run one after the other)
    int np = 0, p0 = 0, pstep = 0, rpos = 0, rstep = 0;
    if (t < kIn) { np = 4; p0 = oW1 + kOwned * rank * kIn + t; pstep = kIn; rpos = t; rstep = kW1Row; }
    else if (t >= 96 && t < 96 + kHid) {
        np = 4; p0 = oW2 + kOwned * rank * kHid + t - 96; pstep = kHid; rpos = rW2 + t - 96; rstep = kW2Row;
    } else if (warp >= 5 && warp < 8 && lane < 4) {
        np = 1; p0 = (warp == 5 ? oB1 : warp == 6 ? oB2 : oW3) + kOwned * rank + lane; rpos = rB1 + 4 * (warp - 5) + lane;
    } else if (warp == 8 && lane == 0 && rank == 0) { np = 1; p0 = oB3; rpos = rB3; }
    const bool sums_loss = warp == 9 && lane == 0;
    float P[4], M[4], V[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (u < np) {
            P[u] = a.P[p0 + u * pstep];
            M[u] = a.m[p0 + u * pstep];
            V[u] = a.v[p0 + u * pstep];
        }

    // this thread's elements of the CTA's 16 x 80 inputs, loaded ahead
    constexpr int kElems = (kCtaRows * kIn + kEpochThreads - 1) / kEpochThreads;
    float xf[kElems], mu[kElems], sd[kElems], label = 0.0f;
#pragma unroll
    for (int k = 0; k < kElems; ++k) {
        const int e = t + k * kEpochThreads;
        mu[k] = e < kCtaRows * kIn ? a.mean[e % kIn] : 0.0f;
        sd[k] = e < kCtaRows * kIn ? a.stdv[e % kIn] : 1.0f;
    }
    const int unit = 32 * (warp & 1) + lane, rq = 4 * ((warp >> 1) & 3);   // phase F, warps 0..7
    const auto load_rows = [&](int step, int g0) {
        const int cnt = step < a.nsteps ? min(a.batch, a.n - step * a.batch) : 0;
        const int row0 = g0 + kCtaRows * rank;
        const int* const index = a.order + (size_t)step * a.batch;
#pragma unroll
        for (int k = 0; k < kElems; ++k) {
            const int e = t + k * kEpochThreads, r = e / kIn;
            xf[k] = mu[k];
            if (e < kCtaRows * kIn && row0 + r < cnt) xf[k] = __ldg(a.feats + (size_t)__ldg(index + row0 + r) * kIn + e - r * kIn);
        }
        const int row = row0 + rq + (lane & 3);
        label = row < cnt ? __ldg(a.labels + __ldg(index + row)) : 0.0f;
    };
    load_rows(0, 0);
    cluster_sync();                                            // mbarriers are ready everywhere

    unsigned row_phase = 0;
    for (int step = 0; step < a.nsteps; ++step) {
        const int cnt = min(a.batch, a.n - step * a.batch);
        float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int g0 = 0; g0 < cnt; g0 += kGroupRows) {
            if (g0 > 0) cluster_sync();                        // every CTA's sums over the previous rows are done
            if (S.failed) continue;                            // uniform: a barrier since the last wait
            // ---- phase F: rows row0 .. row0 + 15 of this minibatch
            const int row0 = g0 + kCtaRows * rank;
            if (t == 0) expect_bytes(&S.bar[0], kCluster * kRowBytes);
#pragma unroll
            for (int k = 0; k < kElems; ++k) {
                const int e = t + k * kEpochThreads;
                if (e < kCtaRows * kIn) {
                    const float x = (xf[k] - mu[k]) / sd[k];
                    (&S.x[0][0])[e] = x;
                    exch[e] = x;
                }
            }
            fence_async();
            __syncthreads();
            if (t == 0) multicast(S.gx[kCtaRows * rank], exch, sizeof(S.x), &S.bar[0]);
            if (warp < 8) {
                const auto bar = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
                const float* const rec = S.w + (unit >> 2) * kRecord + (unit & 3);
                const float* const w1 = S.w + (unit >> 2) * kRecord + (unit & 3) * kW1Row;
                const float* const w2 = S.w + (unit >> 2) * kRecord + rW2 + (unit & 3) * kW2Row;
                float a1[4], a2[4], s[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) a1[r] = rec[rB1];
                dot4<kIn>(a1, [&](int r, int i) { return &S.x[rq + r][i]; }, [&](int i) { return w1[i]; });
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float h = act(gelu(a1[r]), a.bf16);
                    S.h1[rq + r][unit] = h;
                    exch[xH1 + (rq + r) * kHid + unit] = h;
                    a2[r] = rec[rB2];
                }
                fence_async();
                bar();
                if (t == 0) multicast(S.gh[kCtaRows * rank], exch + xH1, sizeof(S.h1), &S.bar[0]);
                dot4<kHid>(a2, [&](int r, int i) { return &S.h1[rq + r][i]; }, [&](int i) { return w2[i]; });
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    S.sd[unit >> 2].h2[rq + r][unit & 3] = act(gelu(a2[r]), a.bf16);
                }
                bar();
                // output and its delta: lane r < 4 of both warps of a row quad
                float dz;
                {
                    const int r = lane & 3, row = row0 + rq + r;
                    float z = S.w[rB3];
#pragma unroll 8
                    for (int j = 0; j < kHid; j += 4) {
                        const float4 w = *reinterpret_cast<const float4*>(S.w + (j >> 2) * kRecord + rW3);
                        const float4 h = *reinterpret_cast<const float4*>(S.sd[j >> 2].h2[rq + r]);
                        z = fmaf(w.x, h.x, z);
                        z = fmaf(w.y, h.y, z);
                        z = fmaf(w.z, h.z, z);
                        z = fmaf(w.w, h.w, z);
                    }
                    const float y = 1.0f / (1.0f + expf(-z));
                    dz = row < cnt ? 2.0f * (y - label) / (float)cnt * y * (1.0f - y) : 0.0f;
                    // every receiver's copy: 16 receivers over 8 lanes a row of two warps
                    *reinterpret_cast<float4*>(S.sd[(lane >> 2) + 8 * (warp & 1)].z[rq + r]) =
                        make_float4(y, dz, y - label, 0.0f);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float d = __shfl_sync(0xffffffffu, dz, r) * rec[rW3] * gelu_grad(a2[r]);
                    S.sd[unit >> 2].d2[rq + r][unit & 3] = d;
                    s[r] = 0.0f;
                }
                bar();
                dot4<kHid>(s, [&](int r, int j) { return S.sd[j >> 2].d2[rq + r]; },
                             [&](int j) { return S.w[(j >> 2) * kRecord + rW2 + (j & 3) * kW2Row + unit]; });
#pragma unroll
                for (int r = 0; r < 4; ++r) S.sd[unit >> 2].d1[rq + r][unit & 3] = s[r] * gelu_grad(a1[r]);
            }
            fence_async();
            __syncthreads();
            if (t < kCluster) send(t, &S.gd[rank], &S.sd[t], sizeof(Deltas), &S.bar[0]);
            // the next rows' inputs load during phase G
            if (g0 + kGroupRows < cnt) load_rows(step, g0 + kGroupRows);
            else load_rows(step + 1, 0);

            // ---- phase G over these rows
            const int rows = min(kGroupRows, cnt - g0);
            if (!wait_bar(&S.bar[0], row_phase & 1)) S.failed = 1;
            ++row_phase;
            if (t < kIn) {
                grad4<kIn>(g, &S.gx[0][t], rows, [&](int r) { return &S.gd[r >> 4].d1[r & 15][0]; });
            } else if (t >= 96 && t < 96 + kHid) {
                grad4<kHid>(g, &S.gh[0][t - 96], rows, [&](int r) { return &S.gd[r >> 4].d2[r & 15][0]; });
            } else if (warp == 5 && lane < 4) {
#pragma unroll 16
                for (int r = 0; r < rows; ++r) g[0] += S.gd[r >> 4].d1[r & 15][lane];
            } else if (warp == 6 && lane < 4) {
#pragma unroll 16
                for (int r = 0; r < rows; ++r) g[0] += S.gd[r >> 4].d2[r & 15][lane];
            } else if (warp == 7 && lane < 4) {
#pragma unroll 16
                for (int r = 0; r < rows; ++r) g[0] = fmaf(S.gd[r >> 4].z[r & 15][1], S.gd[r >> 4].h2[r & 15][lane], g[0]);
            } else if (warp == 8 && lane == 0) {
#pragma unroll 16
                for (int r = 0; r < rows; ++r) g[0] += S.gd[r >> 4].z[r & 15][1];
            } else if (sums_loss) {
#pragma unroll 16
                for (int r = 0; r < rows; ++r) {
                    const float d = S.gd[r >> 4].z[r & 15][2];
                    g[0] = fmaf(d, d, g[0]);
                }
            }
        }
        if (sums_loss && rank == 0) a.loss[step] = S.failed ? __int_as_float(0x7fc00000) : g[0] / (float)cnt;
        if (t == 0 && !S.failed) expect_bytes(&S.bar[1], kCluster * kRecord * 4);
        const AdamArgs ad{nullptr, nullptr, nullptr, a.lr, a.b1, a.b2, a.eps, a.c1[step], a.c2[step]};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < np) {
                adam_step(ad, P[u], M[u], V[u], g[u]);
                exch[xRec + rpos + u * rstep] = P[u];
            }
        fence_async();
        __syncthreads();
        // a CTA whose wait ran out sends nothing more, so the others' waits run
        // out too; all still meet at every cluster barrier
        if (!S.failed) {
            if (t == 0) multicast(S.w + kRecord * rank, exch + xRec, kRecord * 4, &S.bar[1]);
            if (!wait_bar(&S.bar[1], step & 1)) S.failed = 1;
        }
        __syncthreads();
    }
    if (S.failed) {                                            // copies still on their way, again with a limit
        wait_bar(&S.bar[0], (row_phase - 1) & 1);
        wait_bar(&S.bar[1], (a.nsteps - 1) & 1);
    }
    cluster_sync();                                            // no CTA leaves while another still sends to it
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (u < np) {
            a.P[p0 + u * pstep] = P[u];
            a.m[p0 + u * pstep] = M[u];
            a.v[p0 + u * pstep] = V[u];
        }
}

// training target of a quality label: (Q - 1) / 99 (IEEE division, as the
// host would compute it in float32)
__global__ void k_quality_labels(const int32_t* __restrict__ q, int n, float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)(q[i] - 1) / 99.0f;
}

// mean and standard deviation of every feature (float64): one CTA per
// feature, each thread summing a fixed stride of rows, the partial sums
// combined in a fixed tree (deterministic); a standard deviation below 1e-6
// becomes 1
constexpr int kNormThreads = 256;

__device__ double cta_sum_fixed(double v, double* red) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kNormThreads)
k_feat_norm(const float* __restrict__ feats, int n, float* __restrict__ mean, float* __restrict__ stdv) {
    __shared__ double red[kNormThreads];
    const int i = blockIdx.x;
    double s = 0.0;
    for (int r = threadIdx.x; r < n; r += kNormThreads) s += (double)feats[(size_t)r * kIn + i];
    const double mu = cta_sum_fixed(s, red) / n;
    double v = 0.0;
    for (int r = threadIdx.x; r < n; r += kNormThreads) {
        const double d = (double)feats[(size_t)r * kIn + i] - mu;
        v += d * d;
    }
    const double sd = sqrt(cta_sum_fixed(v, red) / n);
    if (threadIdx.x == 0) {
        mean[i] = (float)mu;
        stdv[i] = sd < 1e-6 ? 1.0f : (float)sd;
    }
}

// Feature k of one frame from its statistics words (float64 arithmetic), one
// thread each: one thread per frame took 104 us for 48 frames, nearly all of
// it the 64 logarithms one after the other.
__global__ void k_features(const unsigned long long* __restrict__ stats, const int* __restrict__ width,
                           const int* __restrict__ height, const float* __restrict__ target, int n,
                           float* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * kIn) return;
    const int f = (int)(e / kIn), k = (int)(e - (long long)f * kIn);
    const unsigned long long* st = stats + (size_t)f * kStatsWords;
    const double nb = (double)st[kStBlocks], ns = (double)st[kStSamples], nd = nb * 56.0;
    float o = 1.0f;
    if (k < 64) {
        o = (float)log1p((double)st[k] / nb);
    } else if (k == 64) {
        o = (float)((double)st[kStSum] / ns / 128.0);
    } else if (k == 65) {
        const double mean = (double)st[kStSum] / ns;
        double var = (double)st[kStSum2] / ns - mean * mean;
        if (var < 0.0) var = 0.0;
        o = (float)(sqrt(var) / 64.0);
    } else if (k == 66 || k == 67) {
        o = (float)((double)st[k == 66 ? kStMin : kStMax] / 255.0);
    } else if (k == 68 || k == 69) {
        o = (float)((double)st[k == 68 ? kStAbsDx : kStAbsDy] / nd / 32.0);
    } else if (k == 70 || k == 71) {
        o = (float)(sqrt((double)st[k == 70 ? kStDx2 : kStDy2] / nd) / 32.0);
    } else if (k < 76) {
        o = (float)((double)st[kStLowAc + k - 72] / nb);
    } else if (k == 76 || k == 77) {
        o = (float)(log2((double)(k == 76 ? width : height)[f]) / 11.0);
    } else if (k == 78) {
        o = (float)(((double)target[f] - 35.0) / 7.0);
    }
    out[e] = o;
}

cudaError_t launch_features(const unsigned long long* stats, const int* w, const int* h, const float* t, int n,
                            float* out, cudaStream_t s) {
    k_features<<<(unsigned)(((long long)n * kIn + 127) / 128), 128, 0, s>>>(stats, w, h, t, n, out);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const dct_mlp* net, const float* feats, int n, float* y, int* q, cudaStream_t s) {
    const int ctas = (n + kFwdRows - 1) / kFwdRows;
    k_mlp_forward<<<ctas < 1024 ? ctas : 1024, kFwdRows * 32, 0, s>>>(net->params, feats, net->feat_mean, net->feat_std, net->act_bf16, n,
                                               y, q);
    return cudaGetLastError();
}

static bool adam_params_ok(float lr, float beta1, float beta2, float eps) {
    return lr > 0.f && beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f && beta2 < 1.f && eps > 0.f;
}

// advances the network's step count and returns the Adam arguments of that
// step (bias corrections computed on the host in float64)
static AdamArgs next_adam_step(dct_mlp* net, float lr, float beta1, float beta2, float eps) {
    net->step += 1;
    const double c1 = 1.0 / (1.0 - std::pow((double)beta1, net->step));
    const double c2 = 1.0 / (1.0 - std::pow((double)beta2, net->step));
    return AdamArgs{net->params, net->adam_m, net->adam_v, lr, beta1, beta2, eps, (float)c1, (float)c2};
}

// one minibatch: forward and deltas (one warp per row, 8 rows per CTA,
// weights staged once per CTA), then one CTA per gradient tile
template <bool ADAM>
static cudaError_t launch_train_step(const dct_mlp* net, const float* feats, const float* labels, const int* index,
                                     int batch, float* grad, float* loss, void* workspace, AdamArgs adam,
                                     cudaStream_t s) {
    float* cache = static_cast<float*>(workspace);
    k_mlp_delta<<<(batch + kDeltaRows - 1) / kDeltaRows, kDeltaRows * 32, 0, s>>>(
        net->params, feats, labels, index, net->feat_mean, net->feat_std, net->act_bf16, batch, cache);
    k_mlp_grad<ADAM><<<kGradCtas, kGradThreads, 0, s>>>(cache, labels, index, batch, grad, loss, adam);
    return cudaGetLastError();
}

// Whether this device can hold the training cluster (16 CTAs of one cluster
// need one GPC with as many SMs free of other limits).
static bool epoch_cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(kCluster);
    cfg.blockDim = dim3(kEpochThreads);
    cfg.dynamicSmemBytes = sizeof(EpochSmem);
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaFuncSetAttribute(k_mlp_epoch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EpochSmem)) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, k_mlp_epoch, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

static dct_status check_net(const dct_mlp* net, bool train) {
    if (!net || !net->params || !net->feat_mean || !net->feat_std)
        return fail(DCT_ERR_INVALID_ARG, "network pointers are null");
    if (train && (!net->adam_m || !net->adam_v)) return fail(DCT_ERR_INVALID_ARG, "Adam state pointers are null");
    if (net->act_bf16 != 0 && net->act_bf16 != 1) return fail(DCT_ERR_INVALID_ARG, "act_bf16 must be 0 or 1");
    if (((uintptr_t)net->params) & 15u) return fail(DCT_ERR_INVALID_ARG, "params must be 16-byte aligned");
    return DCT_OK;
}

}  // namespace dctgb

using namespace dctgb;

extern "C" {

dct_status dct_features(const uint64_t* stats, const int32_t* width, const int32_t* height, const float* target,
                        int n, float* feats_out, dct_stream_t stream) {
    if (!stats || !width || !height || !target || !feats_out) return fail(DCT_ERR_INVALID_ARG, "null pointer");
    if (n < 1) return fail(DCT_ERR_INVALID_ARG, "n must be >= 1");
    cudaError_t e = launch_features(reinterpret_cast<const unsigned long long*>(stats), width, height, target, n,
                                    feats_out, (cudaStream_t)stream);
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "features launch");
}

dct_status dct_mlp_set_norm(dct_mlp* net, const float* feats, int n, dct_stream_t stream) {
    dct_status st = check_net(net, false);
    if (st != DCT_OK) return st;
    if (!feats || n < 1) return fail(DCT_ERR_INVALID_ARG, "feats null or n < 1");
    k_feat_norm<<<kIn, kNormThreads, 0, (cudaStream_t)stream>>>(feats, n, net->feat_mean, net->feat_std);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "norm launch");
}

dct_status dct_mlp_forward(const dct_mlp* net, const float* feats, int n, float* y_out, int32_t* quality_out,
                           dct_stream_t stream) {
    dct_status st = check_net(net, false);
    if (st != DCT_OK) return st;
    if (!feats || n < 1) return fail(DCT_ERR_INVALID_ARG, "feats null or n < 1");
    cudaError_t e = launch_mlp_forward(net, feats, n, y_out, quality_out, (cudaStream_t)stream);
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "forward launch");
}

dct_status dct_mlp_labels(const int32_t* quality, int n, float* labels_out, dct_stream_t stream) {
    if (!quality || !labels_out) return fail(DCT_ERR_INVALID_ARG, "null pointer");
    if (n < 1) return fail(DCT_ERR_INVALID_ARG, "n must be >= 1");
    k_quality_labels<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(quality, n, labels_out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "labels launch");
}

size_t dct_mlp_workspace_bytes(int batch) {
    if (batch < 1) return 0;
    return sizeof(float) * ((size_t)batch * kCache + kParams + 4);
}

dct_status dct_mlp_loss_grad(const dct_mlp* net, const float* feats, const float* labels, const int32_t* index,
                             int batch, float* grad_out, float* loss_out, void* workspace, dct_stream_t stream) {
    dct_status st = check_net(net, false);
    if (st != DCT_OK) return st;
    if (!feats || !labels || !index || !grad_out || !loss_out || !workspace)
        return fail(DCT_ERR_INVALID_ARG, "null pointer");
    if (batch < 1 || batch > (1 << 20)) return fail(DCT_ERR_INVALID_ARG, "batch must be 1..2^20");
    if (((uintptr_t)workspace) & 15u) return fail(DCT_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
    cudaError_t e = launch_train_step<false>(net, feats, labels, index, batch, grad_out, loss_out, workspace,
                                             AdamArgs{}, (cudaStream_t)stream);
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "gradient launch");
}

dct_status dct_mlp_adam(dct_mlp* net, const float* grad, float lr, float beta1, float beta2, float eps,
                        dct_stream_t stream) {
    dct_status st = check_net(net, true);
    if (st != DCT_OK) return st;
    if (!grad) return fail(DCT_ERR_INVALID_ARG, "null grad");
    if (!adam_params_ok(lr, beta1, beta2, eps)) return fail(DCT_ERR_INVALID_ARG, "Adam hyper-parameters out of range");
    k_adam<<<(kParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(next_adam_step(net, lr, beta1, beta2, eps), grad);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "adam launch");
}

dct_status dct_mlp_train_epoch(dct_mlp* net, const float* feats, const float* labels, const int32_t* order, int n,
                               int batch, float lr, float* loss_out, void* workspace, dct_stream_t stream) {
    dct_status st = check_net(net, true);
    if (st != DCT_OK) return st;
    if (!feats || !labels || !order || !loss_out || !workspace) return fail(DCT_ERR_INVALID_ARG, "null pointer");
    if (n < 1 || batch < 1 || batch > (1 << 20)) return fail(DCT_ERR_INVALID_ARG, "n >= 1 and batch in 1..2^20");
    if (!adam_params_ok(lr, 0.9f, 0.999f, 1e-8f)) return fail(DCT_ERR_INVALID_ARG, "learning rate must be > 0");
    if (((uintptr_t)workspace) & 15u) return fail(DCT_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
    // batches that one cluster handles: runs of steps in one launch
    cudaStream_t st_ = (cudaStream_t)stream;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    if (batch >= kEpochMinBatch && batch <= kEpochMaxBatch && epoch_cluster_config(cfg, at, st_)) {
        const int steps = (n + batch - 1) / batch;
        for (int k0 = 0; k0 < steps; k0 += kEpochSteps) {
            EpochArgs a;
            memset(&a, 0, sizeof a);
            a.nsteps = steps - k0 < kEpochSteps ? steps - k0 : kEpochSteps;
            for (int k = 0; k < a.nsteps; ++k) {
                const AdamArgs s = next_adam_step(net, lr, 0.9f, 0.999f, 1e-8f);
                a.c1[k] = s.c1;
                a.c2[k] = s.c2;
                a.b1 = s.b1;
                a.b2 = s.b2;
                a.eps = s.eps;
            }
            a.lr = lr;
            a.P = net->params;
            a.m = net->adam_m;
            a.v = net->adam_v;
            a.feats = feats;
            a.labels = labels;
            a.order = order + (size_t)k0 * batch;
            a.mean = net->feat_mean;
            a.stdv = net->feat_std;
            a.loss = loss_out + k0;
            a.exch = static_cast<float*>(workspace);
            a.bf16 = net->act_bf16;
            a.n = n - k0 * batch;
            a.batch = batch;
            cudaError_t e = cudaLaunchKernelEx(&cfg, k_mlp_epoch, a);
            if (e != cudaSuccess) return cuda_fail(e, "training launch");
        }
        return DCT_OK;
    }
    // per minibatch: the delta kernel, then the gradient sums with the Adam
    // step fused (same arithmetic as dct_mlp_loss_grad + dct_mlp_adam)
    float* grad = reinterpret_cast<float*>(static_cast<char*>(workspace) + dct_mlp_workspace_bytes(batch));
    for (int b0 = 0, k = 0; b0 < n; b0 += batch, ++k) {
        const int cnt = n - b0 < batch ? n - b0 : batch;
        cudaError_t e = launch_train_step<true>(net, feats, labels, order + b0, cnt, grad, loss_out + k, workspace,
                                                next_adam_step(net, lr, 0.9f, 0.999f, 1e-8f), (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e, "training step launch");
    }
    return DCT_OK;
}

}  // extern "C"
