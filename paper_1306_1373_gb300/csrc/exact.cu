// Exact-DCT pipeline on the GPU: the "DCT" rows of Tables 3 and 4, i.e. the
// orthonormal 2-D DCT of Eq. 6, quantiser, dequantiser and inverse, in
// float32 with a fixed order of operations (each product and sum rounded on
// its own, no fused multiply-add), so that the quantised codes and the
// rounded pixels are reproducible:
//   rows    Z[i][v] = sum_k C[v][k] x[i][k]     (k ascending), x = p - 128
//   columns X[u][v] = sum_k C[u][k] Z[k][v]
//   q = sgn(X) floor(|X| / Q + 0.5),  D = q Q
//   columns T[i][v] = sum_u C[u][i] D[u][v];  rows y[i][j] = sum_v C[v][j] T[i][v]
//   r = clamp(floor((y + 128) + 0.5), 0, 255)
// Two lanes share a block, with the two-lane tile's transposes
// (kernels_pair.cuh).  The products and sums of a pass run packed (two rows or
// two columns at once, the same roundings).  Bound by the FMA pipes: 47.5
// operations per sample, 12 clocks per 32 samples and SM.  The one-lane form
// with plain operations, IEEE divisions and a byte loop for the SSE took 64 us
// on one 3072 x 3072 plane; this one takes 28.7 us.
#include <cmath>
#include <cstring>

#include "host_common.h"
#include "kernels_pair.cuh"

namespace dctgb {

struct ExactArgs {
    PlaneArg p[kMaxPlanes];
    float Q[2][64];       // quantiser steps (luma, chroma)
    float R[2][64];       // 1 / Q, rounded to float
    int32_t nplanes;
    int32_t ntiles;
};

// Rounded products, as fused multiply-adds with zero: the assembler contracts
// mul.f32x2 with a following add.f32x2, which this pipeline must not (the sign
// of a zero product, the only difference, reaches no code or pixel).
__device__ __forceinline__ f2 f2_mul(f2 a, f2 k) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(k.v), "l"(0ull));
    return r;
}

// C[u][i] = sqrt(2/8) alpha(u) cos(pi u (2i + 1) / 16) is, up to sign, one of
// seven floats kMag[m] = cos(pi m / 16) / 2, m = 1..7 (alpha(0) makes row 0 the
// fourth).  basis_index: m, negative where C[u][i] is.
__host__ __device__ constexpr int basis_index(int u, int i) {
    if (u == 0) return 4;
    int j = (u * (2 * i + 1)) % 32;
    if (j > 16) j = 32 - j;                  // cos is even
    return j > 8 ? -(16 - j) : j;            // and odd about pi / 2
}
__host__ __device__ constexpr float basis_mag(int m) {
    constexpr float mag[8] = {0.0f,          0.490392625f, 0.461939752f, 0.415734798f,
                              0.353553385f,  0.277785122f, 0.191341713f, 0.0975451618f};
    return mag[m];
}

// out[v] = sum_k c(v, k) x[k], k ascending, every product and sum rounded, for
// two vectors; c(v, k) = C[v][k], or its transpose C[k][v] for the inverse.
// Products that differ only in sign are formed once (7 of 8 per input forward,
// 22 of 64 for a whole inverse vector) and subtracted where the sign says so.
template <bool INV, int K, int V, unsigned DONE>
__device__ __forceinline__ void dct8_terms(const f2 (&x)[8], f2 (&p)[8], f2 (&out)[8]) {
    if constexpr (V < 8) {
        constexpr int c = INV ? basis_index(K, V) : basis_index(V, K);
        constexpr int m = c < 0 ? -c : c;
        if constexpr (!((DONE >> m) & 1u)) p[m] = f2_mul(x[K], f2_splat(basis_mag(m)));
        if constexpr (K == 0) out[V] = p[m];          // C[u][0] and C[0][i] are positive
        else if constexpr (c < 0) out[V] = out[V] - p[m];
        else out[V] = out[V] + p[m];
        dct8_terms<INV, K, V + 1, DONE | (1u << m)>(x, p, out);
    }
}
template <bool INV, int K = 0>
__device__ __forceinline__ void dct8(const f2 (&x)[8], f2 (&out)[8]) {
    if constexpr (K < 8) {
        f2 p[8];
        dct8_terms<INV, K, 0, 0u>(x, p, out);
        dct8<INV, K + 1>(x, out);
    }
}

// The same on two float vectors, in place.
template <bool INV>
__device__ __forceinline__ void dct8_two(float (&a)[8], float (&b)[8]) {
    f2 x[8], y[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = f2_pack(a[k], b[k]);
    dct8<INV>(x, y);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float2 t = f2_unpack(y[k]);
        a[k] = t.x;
        b[k] = t.y;
    }
}

// floor(|X| / Q + 0.5) with the quotient and the sum rounded to float, and X's
// sign.  The quotient comes from r = 1 / Q rounded to nearest by Markstein's
// theorem: with q0 = |X| r and its residual |X| - Q q0 (exact in a fused
// multiply-add), q0 + residual r rounds to the correctly rounded quotient.
// Sums below 2^22, so adding 2^23 rounded down leaves the floor.
__device__ __forceinline__ float exact_code(float X, float Q, float r) {
    const float x = fabsf(X);
    const float q0 = __fmul_rn(x, r);
    const float q = __fmaf_rn(__fmaf_rn(-Q, q0, x), r, q0);
    const float t = __fadd_rn(__fadd_rd(__fadd_rn(q, 0.5f), 8388608.0f), -8388608.0f);
    return copysignf(t, X);
}

constexpr int kExactThreads = 128;
constexpr int kExactSmem = (kExactThreads / 32) * (kXBytes + kParkBytes);

template <bool STORE_COEF, bool STORE_RECON>
__global__ void __launch_bounds__(kExactThreads, 6) k_exact(const __grid_constant__ ExactArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ unsigned long long sse_acc[kMaxPlanes];
    __shared__ __align__(16) float tq[2][64], tr[2][64];
    if (threadIdx.x < kMaxPlanes) sse_acc[threadIdx.x] = 0ull;
    for (int i = threadIdx.x; i < 128; i += blockDim.x) {
        tq[i >> 6][i & 63] = a.Q[i >> 6][i & 63];
        tr[i >> 6][i & 63] = a.R[i >> 6][i & 63];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warps = kExactThreads / 32;
    const int k = lane >> 1, h = lane & 1;
    uint8_t* const xb = smem + (threadIdx.x >> 5) * (kXBytes + kParkBytes);
    uint8_t* const xw = xb + k * kXSlot + h * kXRowHalf;   // rows 4h..4h+3, both quads
    uint8_t* const xr = xb + k * kXSlot + h * 16;           // rows 0..7, quad h
    uint8_t* const park = xb + kXBytes + lane * 32;
    const int psw = (lane >> 2) & 1;
    for (int unit = blockIdx.x * warps + (threadIdx.x >> 5); unit < 2 * a.ntiles; unit += gridDim.x * warps) {
        const int tile = unit >> 1;
        int pi = 0;
#pragma unroll
        for (int i = 1; i < kMaxPlanes; ++i)
            if (i < a.nplanes && tile >= a.p[i].tile_begin) pi = i;
        const PlaneArg& P = a.p[pi];
        const int b0 = (tile - P.tile_begin) * kTileBlocks + (unit & 1) * kPairBlocks;
        const int nvalid = min(kPairBlocks, P.nblk - b0);
        if (nvalid <= 0) continue;                           // warp-uniform
        const bool active = k < nvalid;
        const int by = (b0 + k) / P.nbx, bx = (b0 + k) - by * P.nbx;
        const float* const Qt = &tq[P.table][4 * h];
        const float* const Rt = &tr[P.table][4 * h];
        unsigned e = 0;
        uint32_t pix[4][2];
        if (active) {
            load_rows4(P.src, P.src_pitch, P.width, P.height, by, bx, h, (P.flags & kVecSrc) != 0, pix);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) pix[j][0] = pix[j][1] = 0x80808080u;
        }
        park_rows(park, psw, pix);
        float z[4][8];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < 8; ++c)
                z[j][c] = __fadd_rn(__int_as_float((int)__byte_perm(pix[j][c >> 2], 0x4B000000u, 0x7440u | (c & 3))),
                                    -(8388608.0f + 128.0f));
        // rows: Z[i][v] = sum_k C[v][k] x[i][k]
        dct8_two<false>(z[0], z[1]);
        dct8_two<false>(z[2], z[3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            *reinterpret_cast<float4*>(xw + j * 32) = make_float4(z[j][0], z[j][1], z[j][2], z[j][3]);
            *reinterpret_cast<float4*>(xw + j * 32 + 16) = make_float4(z[j][4], z[j][5], z[j][6], z[j][7]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float4 t = *reinterpret_cast<const float4*>(xr + (r >> 2) * kXRowHalf + (r & 3) * 32);
            z[0][r] = t.x;
            z[1][r] = t.y;
            z[2][r] = t.z;
            z[3][r] = t.w;
        }
        // columns: X[u][v] = sum_k C[u][k] Z[k][v]
        dct8_two<false>(z[0], z[1]);
        dct8_two<false>(z[2], z[3]);
        __syncwarp();                                        // transpose reads done
        // quantise (codes as exact small integers in float); stage the codes
        uint8_t* const xc = xb + k * 128 + h * 8;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float4 q4 = *reinterpret_cast<const float4*>(Qt + u * 8);
            const float4 r4 = *reinterpret_cast<const float4*>(Rt + u * 8);
            const float qs[4] = {q4.x, q4.y, q4.z, q4.w}, rs[4] = {r4.x, r4.y, r4.z, r4.w};
            float t[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float q = exact_code(z[i][u], qs[i], rs[i]);
                z[i][u] = __fmul_rn(q, qs[i]);               // dequantised D
                t[i] = __fadd_rn(q, kMagic);
            }
            if (STORE_COEF)
                *reinterpret_cast<uint2*>(xc + ((u ^ (k & 7)) << 4)) = make_uint2(pack_codes(t[0], t[1]), pack_codes(t[2], t[3]));
        }
        if (STORE_COEF) {
            __syncwarp();
            uint4* const g = reinterpret_cast<uint4*>(P.coef + (size_t)b0 * 64) + lane;
            const int q = lane >> 3;
#pragma unroll
            for (int i = 0; i < 4; ++i) {                    // chunk 32 i + lane: block 4 i + q, row lane % 8
                const uint4 w = *reinterpret_cast<const uint4*>(
                    xb + (4 * i + q) * 128 + (((lane & 7) ^ ((4 * i + q) & 7)) << 4));
                if (4 * i + q < nvalid) g[32 * i] = w;
            }
        }
        // columns: T[i][v] = sum_u C[u][i] D[u][v]
        dct8_two<true>(z[0], z[1]);
        dct8_two<true>(z[2], z[3]);
        __syncwarp();                                        // staged codes read
#pragma unroll
        for (int r = 0; r < 8; ++r)
            *reinterpret_cast<float4*>(xr + (r >> 2) * kXRowHalf + (r & 3) * 32) =
                make_float4(z[0][r], z[1][r], z[2][r], z[3][r]);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 t0 = *reinterpret_cast<const float4*>(xw + j * 32);
            const float4 t1 = *reinterpret_cast<const float4*>(xw + j * 32 + 16);
            z[j][0] = t0.x; z[j][1] = t0.y; z[j][2] = t0.z; z[j][3] = t0.w;
            z[j][4] = t1.x; z[j][5] = t1.y; z[j][6] = t1.z; z[j][7] = t1.w;
        }
        // rows: y[i][j] = sum_v C[v][j] T[i][v]; pixels floor((y + 128) + 0.5),
        // clamped before the floor (adding 2^23 rounded down), which commutes
        dct8_two<true>(z[0], z[1]);
        dct8_two<true>(z[2], z[3]);
        uint32_t out[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float y = __fadd_rn(__fadd_rn(z[j][4 * q + i], 128.0f), 0.5f);
                    b[i] = (uint32_t)__float_as_int(__fadd_rd(fminf(fmaxf(y, 0.0f), 255.0f), 8388608.0f));
                }
                out[j][q] = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
            }
        if (STORE_RECON && active)
            store_rows4(P.dst, P.dst_pitch, P.width, P.height, by, bx, h, (P.flags & kVecDst) != 0, out);
        if (active) {
            unpark_rows(park, psw, pix);
            const int nr = min(4, P.height - (by * 8 + 4 * h)), nc = min(8, P.width - bx * 8);
            if (nr == 4 && nc == 8) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const unsigned ad = __vabsdiffu4(out[j][q], pix[j][q]);
                        e = __dp4a(ad, ad, e);
                    }
            } else {
                for (int j = 0; j < nr; ++j)
                    for (int c = 0; c < nc; ++c) {
                        const int d = sample4(out, j, c) - sample4(pix, j, c);
                        e += d * d;
                    }
            }
        }
        const unsigned tot = warp_sum(e);
        if (lane == 0 && tot) atomicAdd(&sse_acc[pi], (unsigned long long)tot);
    }
    __syncthreads();
    if (threadIdx.x < a.nplanes && sse_acc[threadIdx.x]) atomicAdd(a.p[threadIdx.x].sse, sse_acc[threadIdx.x]);
}

template <bool STORE_COEF, bool STORE_RECON>
static cudaError_t launch_exact(const ExactArgs& a, int num_sms, cudaStream_t s) {
    int occ = 0;
    static OccCache cache;
    cudaError_t e = kernel_occupancy(k_exact<STORE_COEF, STORE_RECON>, cache, kExactThreads, kExactSmem, kExactSmem, occ);
    if (e != cudaSuccess) return e;
    k_exact<STORE_COEF, STORE_RECON>
        <<<direct_grid(2 * a.ntiles, kExactThreads, num_sms, occ), kExactThreads, kExactSmem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace dctgb

using namespace dctgb;

extern "C" dct_status dct_exact_fused(dct_plan_t plan, const dct_plane* planes, int nplanes, int quality,
                                      const uint16_t* qtab_host, int qtab_entries, int16_t* coeffs,
                                      const dct_plane* recon_planes, uint64_t* sse_out, dct_stream_t stream) {
    if (!plan) return fail(DCT_ERR_INVALID_ARG, "null plan");
    if (!planes || !sse_out) return fail(DCT_ERR_INVALID_ARG, "null planes or sse_out");
    if (nplanes < 1 || nplanes > kMaxPlanes) return fail(DCT_ERR_INVALID_ARG, "nplanes must be 1..4");
    if (((uintptr_t)sse_out) & 7u) return fail(DCT_ERR_INVALID_ARG, "sse_out must be 8-byte aligned");
    if (coeffs && (((uintptr_t)coeffs) & 15u)) return fail(DCT_ERR_INVALID_ARG, "coeffs must be 16-byte aligned");
    ExactArgs a;
    memset(&a, 0, sizeof a);
    const bool yuv = plan->desc.layout == DCT_LAYOUT_YUV420;
    for (int t = 0; t < 2; ++t) {
        QuantSet qs;
        dct_status st = build_tables(quality, qtab_host, qtab_entries, (t == 1 && yuv) ? 1 : 0, qs);
        if (st != DCT_OK) return st;
        for (int k = 0; k < 64; ++k) {
            a.Q[t][k] = (float)qs.Q[k];
            a.R[t][k] = 1.0f / a.Q[t][k];
        }
    }
    int cursor = 0;
    size_t coef_off = 0;
    for (int i = 0; i < nplanes; ++i) {
        dct_status st = check_plane(plan, planes[i], "plane");
        if (st != DCT_OK) return st;
        PlaneArg& p = a.p[i];
        fill_plane(p, planes[i], cursor);
        p.src = planes[i].data;
        p.src_pitch = planes[i].pitch;
        p.table = (yuv && i > 0) ? 1 : 0;
        int fl = ((((uintptr_t)planes[i].data) & 7u) == 0 && (planes[i].pitch & 7) == 0) ? kVecSrc : 0;
        if (recon_planes) {
            st = check_plane(plan, recon_planes[i], "recon plane");
            if (st != DCT_OK) return st;
            if (recon_planes[i].width != planes[i].width || recon_planes[i].height != planes[i].height)
                return fail(DCT_ERR_INVALID_ARG, "recon plane size differs from input plane");
            p.dst = recon_planes[i].data;
            p.dst_pitch = recon_planes[i].pitch;
            if ((((uintptr_t)recon_planes[i].data) & 7u) == 0 && (recon_planes[i].pitch & 7) == 0) fl |= kVecDst;
        }
        p.flags = fl;
        p.coef = coeffs ? coeffs + coef_off : nullptr;
        coef_off += (size_t)p.nblk * 64;
        p.sse = reinterpret_cast<unsigned long long*>(sse_out) + i;
    }
    a.nplanes = nplanes;
    a.ntiles = cursor;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(sse_out, 0, sizeof(uint64_t) * nplanes, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    const int sms = plan->num_sms;
    e = coeffs ? (recon_planes ? launch_exact<true, true>(a, sms, s) : launch_exact<true, false>(a, sms, s))
               : (recon_planes ? launch_exact<false, true>(a, sms, s) : launch_exact<false, false>(a, sms, s));
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "exact launch");
}
