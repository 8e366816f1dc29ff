// Learned rate controller, network side: the 80 features, input
// normalisation, forward pass, back-propagation with deterministic
// (fixed-order) minibatch sums, and Adam.  The network is tiny (9409
// parameters), so it runs on plain FMA units: one warp per sample for
// inference, one cluster of 16 CTAs for a run of training steps; single
// gradients (and epochs where no cluster of 16 fits) use one warp per minibatch
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

// Inference, ROWS samples to a warp: lane l owns hidden units l and l + 32 of
// both layers, every sum over its inputs in ascending order (the inputs a lane
// does not hold come by shuffle).  W1 and W2 are staged transposed with rows
// padded to 65 floats, as in k_mlp_delta.  One thread per sample took 219 us for
// the 48 frames of a small rate-control call (a serial walk over 9,409
// parameters in global memory); one sample a warp takes 13 us.  That is bound
// by the shared-memory pipe, which also moves the shuffles; four samples a warp
// read a weight once for four: 100,000 samples 144 us against 213, 1,000,000
// 1346 against 2000 (1905 with a thread per sample).
constexpr int kFwdWarps = 8;                   // warps per CTA
constexpr int kTStride = kHid + 1;             // padded row of a transposed weight matrix

template <int ROWS>
__global__ void __launch_bounds__(kFwdWarps * 32)
k_mlp_forward(const float* __restrict__ P, const float* __restrict__ feats, const float* __restrict__ mean,
              const float* __restrict__ stdv, int bf16, int n, float* __restrict__ y_out, int* __restrict__ q_out) {
    __shared__ float w1t[kIn * kTStride];       // w1t[i * 65 + j] = W1[j][i]
    __shared__ float w2t[kHid * kTStride];
#pragma unroll 8
    for (int e = threadIdx.x; e < kHid * kIn; e += kFwdWarps * 32) w1t[(e % kIn) * kTStride + e / kIn] = P[oW1 + e];
#pragma unroll 8
    for (int e = threadIdx.x; e < kHid * kHid; e += kFwdWarps * 32) w2t[(e % kHid) * kTStride + e / kHid] = P[oW2 + e];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long step = (long long)gridDim.x * kFwdWarps * ROWS;
    for (long long s = ((long long)blockIdx.x * kFwdWarps + (threadIdx.x >> 5)) * ROWS; s < n; s += step) {   // warp-uniform
        float xn[ROWS][3];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float* x = feats + (size_t)(ROWS == 1 || s + r < n ? s + r : s) * kIn;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int i = lane + 32 * k;
                xn[r][k] = i < kIn ? (x[i] - mean[i]) / stdv[i] : 0.0f;
            }
        }
        float a[ROWS][2], h[ROWS][2], z[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int k = 0; k < 2; ++k) a[r][k] = P[oB1 + lane + 32 * k];
        }
#pragma unroll
        for (int i = 0; i < kIn; ++i) {
            const float w[2] = {w1t[i * kTStride + lane], w1t[i * kTStride + lane + 32]};
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const float v = __shfl_sync(0xffffffffu, xn[r][i >> 5], i & 31);
#pragma unroll
                for (int k = 0; k < 2; ++k) a[r][k] = fmaf(w[k], v, a[r][k]);
            }
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                h[r][k] = act(gelu(a[r][k]), bf16);
                a[r][k] = P[oB2 + lane + 32 * k];
            }
        }
#pragma unroll
        for (int i = 0; i < kHid; ++i) {
            const float w[2] = {w2t[i * kTStride + lane], w2t[i * kTStride + lane + 32]};
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const float v = __shfl_sync(0xffffffffu, h[r][i >> 5], i & 31);
#pragma unroll
                for (int k = 0; k < 2; ++k) a[r][k] = fmaf(w[k], v, a[r][k]);
            }
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int k = 0; k < 2; ++k) h[r][k] = act(gelu(a[r][k]), bf16);
            z[r] = P[oB3];
        }
        const float w3[2] = {P[oW3 + lane], P[oW3 + lane + 32]};
#pragma unroll
        for (int j = 0; j < kHid; ++j) {
            const float w = __shfl_sync(0xffffffffu, w3[j >> 5], j & 31);
#pragma unroll
            for (int r = 0; r < ROWS; ++r) z[r] = fmaf(w, __shfl_sync(0xffffffffu, h[r][j >> 5], j & 31), z[r]);
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float y = 1.0f / (1.0f + expf(-z[r]));
            if (lane == 0 && (ROWS == 1 || s + r < n)) {
                if (y_out) y_out[s + r] = y;
                if (q_out) {
                    const float q = rintf(1.0f + 99.0f * y);
                    q_out[s + r] = (int)fminf(100.0f, fmaxf(1.0f, q));
                }
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

// Adam step for one parameter (k_adam and the training cluster)
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

__global__ void __launch_bounds__(kGradThreads)
k_mlp_grad(const float* __restrict__ cache, const float* __restrict__ labels, const int* __restrict__ index,
           int batch, float* __restrict__ grad, float* __restrict__ loss) {
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
    if (p >= 0) grad[p] = g;
}

__global__ void k_adam(AdamArgs a, const float* __restrict__ g) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kParams) return;
    adam_step(a, a.P[p], a.m[p], a.v[p], g[p]);
}

// ---------------------------------------------------------------------------
// A run of training steps in one launch: one cluster of 16 CTAs
// ---------------------------------------------------------------------------
// A step of k_mlp_delta and k_mlp_grad is bound by latency, not by work (5.8
// million multiply-adds): two dependent launches, the weights staged anew and
// the cache columns fetched by few CTAs cost 24 us.  Here a cluster stays on 16
// SMs for all steps, and every CTA holds all weights.  Phase F: CTA c runs rows
// 16c..16c+15 of a group of 256 through forward and deltas (a warp takes 2 rows
// and all units; what bounds it is the shared-memory reads, and two rows by two
// units a thread read least among the splits that fill eight warps).  Phase G:
// CTA 4p + q sums the gradients of units 16p..16p+15 over inputs 20q..20q+19 of
// W1 and 16q..16q+15 of W2 (and b1, b2, W3 of its four units 4(4p + q)..) over
// the rows in ascending order, then Adam runs on them, two parameters a thread.
// The square tiles keep the exchange small: a CTA needs 16 units' deltas and 16
// first-layer outputs of each row (48 KB a group; tiles of four whole rows of
// W1 and W2 need 72 KB), and it fetches its 20 input columns itself, a step
// ahead.  All exchange is by 16-byte stores into the other CTAs' shared memory
// (about 8 bytes a clock and SM; loads from there ran at a quarter of that),
// the first-layer outputs while layer 2 runs, W2's deltas while they are
// propagated back.  Two cluster barriers a step order it: one between the
// stores of phase F and phase G, one between the new weights and the next phase
// F (a batch of several groups adds one per group).  Nothing polls memory, so
// no wait can run out, and only the caller's own loads touch its pointers, so
// any memory the GPU can read will do.  All sums and updates have the operands
// and order of k_mlp_delta, k_mlp_grad and k_adam: the same bits.  16,000 rows, batch 256 (63
// steps): 752 us an epoch against 1540 us.  It runs every batch size: 24 steps,
// us, this way against two launches a step: batch 1 227 / 315, 32 236 / 363, 64 246 /
// 364, 512 531 / 835, 1024 977 / 1398, 4096 3652 / 4737, 65536 64056 / 101761.
constexpr int kCluster = 16, kSide = 4;                // CTAs: kSide x kSide gradient tiles
constexpr int kEpochThreads = 512;
constexpr int kTileUnits = kHid / kSide;               // hidden units of a tile
constexpr int kTileIn1 = kIn / kSide, kTileIn2 = kHid / kSide;   // inputs of a tile of W1, W2
constexpr int kGroupRows = 256;                        // rows in flight
constexpr int kCtaRows = kGroupRows / kCluster;
constexpr int kEpochSteps = 64;                        // steps per launch
static_assert(kTileUnits == 16 && kTileIn2 == 16 && kTileIn1 == 20 && kCtaRows == 16, "phases F and G index by these");

struct EpochArgs {
    float *P, *m, *v;
    const float *feats, *labels;
    const int* order;                 // of the first step's first row
    const float *mean, *stdv;
    float* loss;                      // of the first step
    int bf16, n, batch, nsteps;       // n rows left from the first step on
    float lr, b1, b2, eps;
    float c1[kEpochSteps], c2[kEpochSteps];
};

// Rows of 84 and 68 floats: a quarter warp's 16-byte reads of eight units' rows
// hit eight different bank groups, and all rows start 16-byte aligned.
constexpr int kW1Row = kIn + 4, kW2Row = kHid + 4;
constexpr int kGRow = 16;                              // phase G's rows: 64 bytes, so that a warp's stores into them meet no bank twice
static_assert(kTileUnits == kGRow && kTileIn2 == kGRow && kTileIn1 == kGRow + 4, "phase G's rows");

// A tile's parameters in order: W1[16][20], W2[16][16], b1[4], b2[4], W3[4], b3
// and three unused.
constexpr int tW2 = kTileUnits * kTileIn1, tB = tW2 + kTileUnits * kTileIn2, kTileParams = tB + 16;
static_assert(kTileParams <= 2 * kEpochThreads, "two parameters a thread");

struct __align__(16) EpochSmem {
    float w1[kHid][kW1Row], w2[kHid][kW2Row], b1[kHid], b2[kHid], w3[kHid], b3[4];   // all weights
    // of all rows of a group: the tile's first 16 inputs; received deltas of
    // layers 1 and 2; the last 4 inputs, received h2 of four units, (y, dz, y -
    // label, 1) and four unused; received h1
    float gx[kGroupRows][kGRow], gd1[kGroupRows][kGRow];
    float pad[16];                    // what one load of a warp reads before and after: the other half of the banks
    float gd2[kGroupRows][kGRow], ge[kGroupRows][kGRow], gh1[kGroupRows][kGRow];
    // this CTA's rows
    float x[kCtaRows][kIn], h1[kCtaRows][kW2Row], h2[kCtaRows][kW2Row], d1[kCtaRows][kW2Row], d2[kCtaRows][kW2Row];
    float z[kCtaRows][4], mean[kIn], stdv[kIn];
    // this tile's gradients and new weights: W1, W2, and b1, b2, W3 of four units, b3
    float g[kTileParams], p[kTileParams];
};
static_assert(sizeof(EpochSmem) <= 232448, "shared memory of one CTA");

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Stores v at dst (an address in this CTA's shared memory) of CTA `rank`.
__device__ __forceinline__ void put(unsigned rank, void* dst, float4 v) {
    unsigned d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((unsigned)__cvta_generic_to_shared(dst)), "r"(rank));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(d), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
template <int ID, int THREADS>
__device__ __forceinline__ void bar_sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory"); }
template <int ID, int THREADS>
__device__ __forceinline__ void bar_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(THREADS) : "memory"); }

// acc[k][r] += w[k] x[r] over N inputs in ascending order for two units and two
// rows; x(r, i) and w(k, i) give four inputs of a row and their four weights.
template <int N, typename X, typename W>
__device__ __forceinline__ void dot4(float (&acc)[2][2], X in, W weights) {
#pragma unroll 4
    for (int i = 0; i < N; i += 4) {
        const float4 x[2] = {*reinterpret_cast<const float4*>(in(0, i)), *reinterpret_cast<const float4*>(in(1, i))};
        const float4 w[2] = {weights(0, i), weights(1, i)};
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k >> 1][k & 1] = fmaf(w[k >> 1].x, x[k & 1].x, acc[k >> 1][k & 1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k >> 1][k & 1] = fmaf(w[k >> 1].y, x[k & 1].y, acc[k >> 1][k & 1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k >> 1][k & 1] = fmaf(w[k >> 1].z, x[k & 1].z, acc[k >> 1][k & 1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k >> 1][k & 1] = fmaf(w[k >> 1].w, x[k & 1].w, acc[k >> 1][k & 1]);
    }
}

// One thread's share of phase G: eight sums g[u][k] += d[r][u] x[r][k], u < 4 and
// k < 2, over the rows r in ascending order.
struct GradRows {
    float2 x[4];
    float4 d[4];
};
__device__ __forceinline__ void grad_load(const float* x, const float* d, GradRows& v) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v.x[k] = *reinterpret_cast<const float2*>(x + k * kGRow);
        v.d[k] = *reinterpret_cast<const float4*>(d + k * kGRow);
    }
}
__device__ __forceinline__ void grad_row(float (&g)[4][2], float2 x, float4 d) {
    const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        g[u][0] = fmaf(dv[u], x.x, g[u][0]);
        g[u][1] = fmaf(dv[u], x.y, g[u][1]);
    }
}
// Four rows load while four others are summed; the last load repeats rows of
// the arrays when there are no more.
__device__ __forceinline__ void grad_sum(float (&g)[4][2], const float* x, const float* d, int rows) {
    GradRows v0, v1;
    grad_load(x, d, v0);
    for (int left = rows; ; left -= 8) {
        if (left < 8) {
            for (int r = 0; r < left; ++r)
                grad_row(g, *reinterpret_cast<const float2*>(x + r * kGRow), *reinterpret_cast<const float4*>(d + r * kGRow));
            break;
        }
        grad_load(x + 4 * kGRow, d + 4 * kGRow, v1);
#pragma unroll
        for (int k = 0; k < 4; ++k) grad_row(g, v0.x[k], v0.d[k]);
        const int next = left >= 12 ? 8 * kGRow : 0;
        grad_load(x + next, d + next, v0);
#pragma unroll
        for (int k = 0; k < 4; ++k) grad_row(g, v1.x[k], v1.d[k]);
        x += 8 * kGRow;
        d += 8 * kGRow;
    }
}

__global__ void __launch_bounds__(kEpochThreads, 1) k_mlp_epoch(const __grid_constant__ EpochArgs a) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    EpochSmem& S = *reinterpret_cast<EpochSmem*>(smem_raw);
    constexpr int kHalf = kEpochThreads / 2;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = blockIdx.x;                               // one cluster: CTA rank = block index
    const int tp = rank / kSide, tq = rank % kSide;            // this CTA's tile
    for (int e = t; e < kHid * kIn; e += kEpochThreads) S.w1[e / kIn][e % kIn] = a.P[oW1 + e];
    for (int e = t; e < kHid * kHid; e += kEpochThreads) S.w2[e / kHid][e % kHid] = a.P[oW2 + e];
    if (t < kHid) {
        S.b1[t] = a.P[oB1 + t];
        S.b2[t] = a.P[oB2 + t];
        S.w3[t] = a.P[oW3 + t];
    }
    if (t < 4) S.b3[t] = t == 0 ? a.P[oB3] : 0.0f;
    if (t < kIn) {
        S.mean[t] = a.mean[t];
        S.stdv[t] = a.stdv[t];
    }

    // this thread's sums in phase G: threads 0..39 four units by two inputs of W1,
    // 40..71 of W2, and four more the same sums with other operands, of which
    // they keep g[u][1]: b1 and b2 (inputs y - label and 1), W3 (h2 as the
    // deltas, inputs y and dz), in CTA 0 b3 (the z record as the deltas, inputs
    // y - label and 1) and the loss beside it (g[2][0])
    constexpr int q1 = kTileIn1 / 2, q2 = kTileIn2 / 2, g2 = kTileUnits / 4 * q1, gb = g2 + kTileUnits / 4 * q2;
    const float *gx = nullptr, *gd = nullptr;
    int gpos = 0;                                              // where g[0][0] goes in the tile's order
    if (t < g2) {
        const int u = 4 * (t / q1), i = 2 * (t % q1);
        gx = i < kGRow ? &S.gx[0][i] : &S.ge[0][i - kGRow];
        gd = &S.gd1[0][u];
        gpos = u * kTileIn1 + i;
    } else if (t < gb) {
        const int u = 4 * ((t - g2) / q2), i = 2 * ((t - g2) % q2);
        gx = &S.gh1[0][i];
        gd = &S.gd2[0][u];
        gpos = tW2 + u * kTileIn2 + i;
    } else if (t < gb + 3) {
        gx = &S.ge[0][t < gb + 2 ? 10 : 8];
        gd = t == gb ? &S.gd1[0][4 * tq] : t == gb + 1 ? &S.gd2[0][4 * tq] : &S.ge[0][4];
        gpos = tB + 4 * (t - gb);
    } else if (t == gb + 3 && rank == 0) {
        gx = &S.ge[0][10];
        gd = &S.ge[0][8];
        gpos = tB + 12;
    }
    // the Adam state of tile parameters t and t + 512, for the whole run
    const auto param = [&](int e) {
        if (e < tW2) return oW1 + (kTileUnits * tp + e / kTileIn1) * kIn + kTileIn1 * tq + e % kTileIn1;
        if (e < tB) return oW2 + (kTileUnits * tp + (e - tW2) / kTileIn2) * kHid + kTileIn2 * tq + (e - tW2) % kTileIn2;
        if (e < tB + 12) return (e < tB + 4 ? oB1 : e < tB + 8 ? oB2 : oW3) + 4 * rank + (e - tB) % 4;
        return e == tB + 12 && rank == 0 ? oB3 : -1;
    };
    int pi[2];
    float P[2], M[2], V[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        pi[k] = param(t + k * kEpochThreads);
        if (pi[k] >= 0) {
            P[k] = a.P[pi[k]];
            M[k] = a.m[pi[k]];
            V[k] = a.v[pi[k]];
        }
    }

    // inputs, loaded ahead: threads 0..255 elements t + 256 k of the CTA's 16
    // rows of 80, the others the tile's 20 columns of row th.  The row indices
    // load a phase earlier, so that no thread waits for one.
    const bool fwd = t < kHalf;
    const int th = t & (kHalf - 1);
    constexpr int kOwn = kCtaRows * kIn / kHalf;
    const bool vec = (((uintptr_t)a.feats) & 15u) == 0;
    float xf[kTileIn1], label = 0.0f;
    int idx[kOwn + 1];                                         // -1: no such row
    const int rq = 2 * (warp & 7);                             // phase F: rows rq and rq + 1, units lane and lane + 32
    const auto load_index = [&](int step, int g0) {
        const int cnt = step < a.nsteps ? min(a.batch, a.n - step * a.batch) : 0;
        const int* const order = a.order + (size_t)step * a.batch;
        const auto at = [&](int row) { return row < cnt ? __ldg(order + row) : -1; };
        if (fwd) {
#pragma unroll
            for (int k = 0; k < kOwn; ++k) idx[k] = at(g0 + kCtaRows * rank + (t + k * kHalf) / kIn);
            idx[kOwn] = at(g0 + kCtaRows * rank + rq + (lane & 1));
        } else {
            idx[0] = at(g0 + th);
        }
    };
    const auto load_rows = [&] {
        if (fwd) {
#pragma unroll
            for (int k = 0; k < kOwn; ++k)
                if (idx[k] >= 0) xf[k] = __ldg(a.feats + (size_t)idx[k] * kIn + (t + k * kHalf) % kIn);
            if (idx[kOwn] >= 0) label = __ldg(a.labels + idx[kOwn]);
        } else if (idx[0] >= 0) {
            const float* const x = a.feats + (size_t)idx[0] * kIn + kTileIn1 * tq;
            if (vec) {
#pragma unroll
                for (int k = 0; k < kTileIn1; k += 4) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(x + k));
                    xf[k] = v.x;
                    xf[k + 1] = v.y;
                    xf[k + 2] = v.z;
                    xf[k + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int k = 0; k < kTileIn1; ++k) xf[k] = __ldg(x + k);
            }
        }
    };
    load_index(0, 0);
    load_rows();
    cluster_arrive();                                          // every CTA of the cluster has started
    cluster_wait();
    __syncthreads();

    for (int step = 0; step < a.nsteps; ++step) {
        const int cnt = min(a.batch, a.n - step * a.batch);
        float g[4][2] = {};
        for (int g0 = 0; g0 < cnt; g0 += kGroupRows) {
            if (g0 > 0) {                                      // every CTA's sums over the previous rows are done
                cluster_arrive();
                cluster_wait();
            }
            if (g0 + kGroupRows < cnt) load_index(step, g0 + kGroupRows);
            else load_index(step + 1, 0);
            // ---- phase F: rows g0 + 16 rank .. + 15 of this minibatch
            const int mine = kCtaRows * rank;
            // 64 threads a receiver: row r, floats 4c..
            const int blk = (t >> 6) & 3, r = (t >> 2) & 15, c = 4 * (t & 3);
            if (fwd) {
#pragma unroll
                for (int k = 0; k < kOwn; ++k) {
                    const int e = t + k * kHalf, r = e / kIn, col = e - r * kIn;
                    S.x[r][col] = g0 + mine + r < cnt ? (xf[k] - S.mean[col]) / S.stdv[col] : 0.0f;
                }
                bar_sync<1, kHalf>();
                float a1[2][2], a2[2][2], s[2][2];             // [unit][row]; from here on a warp reads its own rows
                const auto unit = [&](int k) { return lane + 32 * k; };
#pragma unroll
                for (int k = 0; k < 2; ++k) a1[k][0] = a1[k][1] = S.b1[unit(k)];
                dot4<kIn>(a1, [&](int r, int i) { return &S.x[rq + r][i]; },
                          [&](int k, int i) { return *reinterpret_cast<const float4*>(&S.w1[unit(k)][i]); });
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        S.h1[rq + r][unit(k)] = act(gelu(a1[k][r]), a.bf16);
                        a2[k][r] = S.b2[unit(k)];
                    }
                }
                bar_arrive<2, kEpochThreads>();
                __syncwarp();
                dot4<kHid>(a2, [&](int r, int i) { return &S.h1[rq + r][i]; },
                           [&](int k, int i) { return *reinterpret_cast<const float4*>(&S.w2[unit(k)][i]); });
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) S.h2[rq + r][unit(k)] = act(gelu(a2[k][r]), a.bf16);
                }
                __syncwarp();
                // output and its delta of row lane % 2
                float dz;
                {
                    const int r = lane & 1;
                    float z = S.b3[0];
#pragma unroll 8
                    for (int j = 0; j < kHid; j += 4) {
                        const float4 w = *reinterpret_cast<const float4*>(&S.w3[j]);
                        const float4 h = *reinterpret_cast<const float4*>(&S.h2[rq + r][j]);
                        z = fmaf(w.x, h.x, z);
                        z = fmaf(w.y, h.y, z);
                        z = fmaf(w.z, h.z, z);
                        z = fmaf(w.w, h.w, z);
                    }
                    const float y = 1.0f / (1.0f + expf(-z));
                    dz = g0 + mine + rq + r < cnt ? 2.0f * (y - label) / (float)cnt * y * (1.0f - y) : 0.0f;
                    if (lane < 2) *reinterpret_cast<float4*>(S.z[rq + r]) = make_float4(y, dz, y - label, 1.0f);
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float dzr = __shfl_sync(0xffffffffu, dz, r);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        S.d2[rq + r][unit(k)] = dzr * S.w3[unit(k)] * gelu_grad(a2[k][r]);
                        s[k][r] = 0.0f;
                    }
                }
                bar_arrive<3, kEpochThreads>();
                __syncwarp();
                dot4<kHid>(s, [&](int r, int j) { return &S.d2[rq + r][j]; },
                           [&](int k, int j) {
                               const float* w = &S.w2[j][unit(k)];
                               return make_float4(w[0], w[kW2Row], w[2 * kW2Row], w[3 * kW2Row]);
                           });
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) S.d1[rq + r][unit(k)] = s[k][r] * gelu_grad(a1[k][r]);
                }
            } else {
                if (g0 + th < cnt) {
#pragma unroll
                    for (int k = 0; k < kTileIn1; k += 4) {
                        const float4 m = *reinterpret_cast<const float4*>(&S.mean[kTileIn1 * tq + k]);
                        const float4 d = *reinterpret_cast<const float4*>(&S.stdv[kTileIn1 * tq + k]);
                        *reinterpret_cast<float4*>(k < kGRow ? &S.gx[th][k] : &S.ge[th][0]) = make_float4((xf[k] - m.x) / d.x, (xf[k + 1] - m.y) / d.y,
                                                                               (xf[k + 2] - m.z) / d.z, (xf[k + 3] - m.w) / d.w);
                    }
                }
                bar_sync<2, kEpochThreads>();                  // first-layer outputs: to the tiles of these inputs
                const float4 h1 = *reinterpret_cast<const float4*>(&S.h1[r][kTileIn2 * blk + c]);
#pragma unroll
                for (int k = 0; k < kSide; ++k) put(kSide * ((k + tp) % kSide) + blk, &S.gh1[mine + r][c], h1);
                bar_sync<3, kEpochThreads>();                  // W2's deltas: to the tiles of these units
                const float4 d2 = *reinterpret_cast<const float4*>(&S.d2[r][kTileUnits * blk + c]);
#pragma unroll
                for (int k = 0; k < kSide; ++k) put(kSide * blk + (k + tq) % kSide, &S.gd2[mine + r][c], d2);
                const int to = th >> 4, rr = th & 15;          // every CTA: its units' h2, and z
                put(to, &S.ge[mine + rr][4], *reinterpret_cast<const float4*>(&S.h2[rr][4 * to]));
                put(to, &S.ge[mine + rr][8], *reinterpret_cast<const float4*>(S.z[rr]));
            }
            __syncthreads();
            {
                const float4 d1 = *reinterpret_cast<const float4*>(&S.d1[r][kTileUnits * blk + c]);
#pragma unroll
                for (int k = 0; k < kSide / 2; ++k)
                    put(kSide * blk + (2 * k + (t >> 8) + tq) % kSide, &S.gd1[mine + r][c], d1);
            }
            cluster_arrive();
            load_rows();                                       // the next rows' inputs, during phase G
            cluster_wait();

            // ---- phase G over these rows
            if (gx) grad_sum(g, gx, gd, min(kGroupRows, cnt - g0));
        }
        if (gx && gpos < tB) {
            const int ld = gpos < tW2 ? kTileIn1 : kTileIn2;
#pragma unroll
            for (int u = 0; u < 4; ++u) *reinterpret_cast<float2*>(&S.g[gpos + u * ld]) = make_float2(g[u][0], g[u][1]);
        } else if (gx && gpos < tB + 12) {
#pragma unroll
            for (int u = 0; u < 4; ++u) S.g[gpos + u] = g[u][1];
        } else if (gx) {
            S.g[tB + 12] = g[1][1];
            a.loss[step] = g[2][0] / (float)cnt;
        }
        __syncthreads();
        const AdamArgs ad{nullptr, nullptr, nullptr, a.lr, a.b1, a.b2, a.eps, a.c1[step], a.c2[step]};
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (pi[k] >= 0) {
                adam_step(ad, P[k], M[k], V[k], S.g[t + k * kEpochThreads]);
                S.p[t + k * kEpochThreads] = P[k];
            }
        __syncthreads();
        // the new weights to every CTA: three threads share an item's 16 stores
        constexpr int kItems = kTileParams / 4, kLane = 160;
        static_assert(kItems <= kLane && 3 * kLane <= kEpochThreads, "weight items");
        const int item = t % kLane, part = t / kLane, e = 4 * item;
        float* dst = nullptr;
        if (part >= 3) {
        } else if (e < tW2) {
            dst = &S.w1[kTileUnits * tp + e / kTileIn1][kTileIn1 * tq + e % kTileIn1];
        } else if (e < tB) {
            dst = &S.w2[kTileUnits * tp + (e - tW2) / kTileIn2][kTileIn2 * tq + (e - tW2) % kTileIn2];
        } else if (e < tB + 12) {
            dst = (e == tB ? S.b1 : e == tB + 4 ? S.b2 : S.w3) + 4 * rank;
        } else if (e == tB + 12 && rank == 0) {
            dst = S.b3;
        }
        if (dst) {
            const float4 w = *reinterpret_cast<const float4*>(&S.p[e]);
            for (int k = part; k < kCluster; k += 3) put((k + rank) % kCluster, dst, w);
        }
        cluster_arrive();
        cluster_wait();
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (pi[k] >= 0) {
            a.P[pi[k]] = P[k];
            a.m[pi[k]] = M[k];
            a.v[pi[k]] = V[k];
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

// The features of a frame from its statistics words (float64 arithmetic).  A
// warp takes one feature of 32 frames at a time, so that it computes one kind:
// the 80 features of a frame side by side in a warp ran every kind it met one
// after the other.  Bound by the float64 unit, and for few frames by the latency
// of one logarithm.  us for 48 / 16,000 / 1,000,000 frames: 9 / 140 / 7872 this
// way, 15 / 318 / 18478 side by side, 152 / 171 / 7817 with a thread per frame.
constexpr int kFeatWarps = 4;                  // features a CTA has in hand
static_assert(kIn % kFeatWarps == 0, "feature tiling");

__global__ void __launch_bounds__(32 * kFeatWarps)
k_features(const unsigned long long* __restrict__ stats, const int* __restrict__ width,
           const int* __restrict__ height, const float* __restrict__ target, int n,
           float* __restrict__ out) {
    const long long f = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
    if (f >= n) return;
    const unsigned long long* st = stats + (size_t)f * kStatsWords;
    float* const of = out + (size_t)f * kIn;
    const double nb = (double)st[kStBlocks], ns = (double)st[kStSamples], nd = nb * 56.0;
    for (int k = blockIdx.y * kFeatWarps + (threadIdx.x >> 5); k < kIn; k += gridDim.y * kFeatWarps) {
        float o = 1.0f;
        if (k < 64) {
            o = (float)log1p((double)st[k] / nb);
        } else if (k == 64) {                          // and 65, from the same mean
            const double mean = (double)st[kStSum] / ns;
            double var = (double)st[kStSum2] / ns - mean * mean;
            if (var < 0.0) var = 0.0;
            of[65] = (float)(sqrt(var) / 64.0);
            o = (float)(mean / 128.0);
        } else if (k == 65) {
            continue;
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
        of[k] = o;
    }
}

cudaError_t launch_features(const unsigned long long* stats, const int* w, const int* h, const float* t, int n,
                            float* out, cudaStream_t s) {
    // feature groups: all 20 until the frames alone fill the GPU, then fewer, so
    // that a thread converts a frame's counts once (16,000 frames: 138 to 143 us
    // with 20 to 2 groups; 300,000: 2498 us with 20, 2380 with one)
    int groups = (1 << 18) / n;
    if (groups > kIn / kFeatWarps) groups = kIn / kFeatWarps;
    if (groups < 1) groups = 1;
    k_features<<<dim3((unsigned)(((long long)n + 31) / 32), groups), 32 * kFeatWarps, 0, s>>>(stats, w, h, t, n, out);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const dct_mlp* net, const float* feats, int n, float* y, int* q, cudaStream_t s) {
    // four samples a warp as soon as that leaves every SM a CTA (8,000 samples 23
    // us against 27, 4,000 19 either way, 1,000 19 against 13)
    const bool four = n >= 4 * kFwdWarps * 152;
    const auto kernel = four ? k_mlp_forward<4> : k_mlp_forward<1>;
    const long long rows = (four ? 4 : 1) * kFwdWarps, ctas = (n + rows - 1) / rows;
    kernel<<<ctas < 1024 ? (int)ctas : 1024, kFwdWarps * 32, 0, s>>>(net->params, feats, net->feat_mean, net->feat_std,
                                                                   net->act_bf16, n, y, q);
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
static cudaError_t launch_loss_grad(const dct_mlp* net, const float* feats, const float* labels, const int* index,
                                    int batch, float* grad, float* loss, void* workspace, cudaStream_t s) {
    float* cache = static_cast<float*>(workspace);
    k_mlp_delta<<<(batch + kDeltaRows - 1) / kDeltaRows, kDeltaRows * 32, 0, s>>>(
        net->params, feats, labels, index, net->feat_mean, net->feat_std, net->act_bf16, batch, cache);
    k_mlp_grad<<<kGradCtas, kGradThreads, 0, s>>>(cache, labels, index, batch, grad, loss);
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
    cudaError_t e = launch_loss_grad(net, feats, labels, index, batch, grad_out, loss_out, workspace,
                                     (cudaStream_t)stream);
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
    // runs of steps in one launch, where the device can hold the cluster
    cudaStream_t st_ = (cudaStream_t)stream;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    if (epoch_cluster_config(cfg, at, st_)) {
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
            a.bf16 = net->act_bf16;
            a.n = n - k0 * batch;
            a.batch = batch;
            cudaError_t e = cudaLaunchKernelEx(&cfg, k_mlp_epoch, a);
            if (e != cudaSuccess) return cuda_fail(e, "training launch");
        }
        return DCT_OK;
    }
    // elsewhere step by step, as dct_mlp_loss_grad and dct_mlp_adam
    float* grad = reinterpret_cast<float*>(static_cast<char*>(workspace) + dct_mlp_workspace_bytes(batch));
    for (int b0 = 0, k = 0; b0 < n; b0 += batch, ++k) {
        const int cnt = n - b0 < batch ? n - b0 : batch;
        cudaError_t e = launch_loss_grad(net, feats, labels, order + b0, cnt, grad, loss_out + k, workspace, st_);
        if (e != cudaSuccess) return cuda_fail(e, "training step launch");
        if ((st = dct_mlp_adam(net, grad, lr, 0.9f, 0.999f, 1e-8f, stream)) != DCT_OK) return st;
    }
    return DCT_OK;
}

}  // extern "C"
