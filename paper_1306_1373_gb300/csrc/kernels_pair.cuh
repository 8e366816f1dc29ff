// Codec tile with two lanes per 8x8 block: the fused pass and the inverse pass
// alone.
//
// Lanes 2k and 2k+1 share block k of a 16-block half tile: lane h owns rows
// 4h..4h+3 for the row passes and columns 4h..4h+3 for the column passes, 32
// values in registers, and the two transposes go through a padded per-warp
// shared-memory slot (8 stores and 8 loads of 16 bytes per lane each, no bank
// conflicts).  Against the one-lane tile (kernels.cuh) this halves the code of
// a tile and the registers: the fused one-lane kernel is 2700 instructions
// long and waits for instruction fetches (ncu: 1.5 cycles of "no instruction"
// per issued one, 0.1 here).  No pipe is full: issue is busy for 71% of the
// cycles, the integer ALU 60%, the L1 data path 57%, and the rest is latency that
// the resident warps do not hide.  At most 80 registers (24 warps per SM): 138.4
// us on 8192 x 8192 + 4K 4:2:0 against 142.4 us at 64 registers (32 warps,
// spills).  The samples wait for the SSE in a per-lane shared-memory slot, and the codes
// leave through the transpose buffer, free between the two transposes, so that
// a store moves 512 contiguous bytes (8 bytes per lane straight from registers
// touched 16 cache lines per store; the forward pass alone took 83.1 us that
// way, 72.8 us staged).
//
// Transpose slot of block k (kXSlot bytes): row r, column quad q (columns
// 4q..4q+3, four int32) at k*kXSlot + (r>>2)*kXRowHalf + (r&3)*32 + q*16.
// With kXSlot/16 = 2 and kXRowHalf/16 = 1 (mod 8), the 16-byte bank group of
// an access is (lane + const) mod 8 both when lane h writes its rows and when
// it reads its column quad, so each quarter-warp phase hits 8 distinct
// groups.
#pragma once
#include <cstddef>

#include "kernels.cuh"

#ifndef DCTGB_PAIR_MINB
#define DCTGB_PAIR_MINB 3   // resident CTAs of 256 threads per SM (launch bounds: <= 80 registers)
#endif

namespace dctgb {

constexpr int kPairBlocks = kTileBlocks / 2;      // blocks per half tile
constexpr int kXSlot = 288;                       // transpose bytes per block
constexpr int kXRowHalf = 144;                    // offset of rows 4..7 in a slot
constexpr int kXBytes = kPairBlocks * kXSlot;     // per warp
constexpr int kParkBytes = 32 * 32;               // each lane's 32 samples, kept for the SSE

// The part of a QuantSet that a mode reads: [M, Mf, QW, QWc] fused, [M, Mf]
// forward, [QWi] for the inverse of own codes, [Q, W] for the inverse of any.
// Batched warps copy only that part, the two-lane ones keep no room for more (the
// slots of 24 warps take 163 of an SM's 227 KB).
__host__ __device__ constexpr int pair_tab_first(unsigned mode) {
    return (mode & kLoadPix) ? (int)offsetof(QuantSet, M)
                             : (mode & kOwnCodes) ? (int)offsetof(QuantSet, QWi) : (int)offsetof(QuantSet, Q);
}
__host__ __device__ constexpr int pair_tab_bytes(unsigned mode) {
    return (mode & kLoadPix) ? ((mode & kInverse) ? 4 : 2) * 256 : (mode & kOwnCodes) ? 256 : 2 * 256;
}
struct PairTabs {
    const uint32_t* M;
    const float *Mf, *QW, *QWc;
    const int32_t *QWi, *Q, *W;
};
// Views of a table part that starts at byte pair_tab_first(MODE) of its set.
template <unsigned MODE>
__device__ __forceinline__ PairTabs pair_tabs(const uint8_t* part) {
    PairTabs t{};
    if (MODE & kLoadPix) {
        t.M = reinterpret_cast<const uint32_t*>(part);
        t.Mf = reinterpret_cast<const float*>(part + 256);
        t.QW = reinterpret_cast<const float*>(part + 512);
        t.QWc = reinterpret_cast<const float*>(part + 768);
    } else if (MODE & kOwnCodes) {
        t.QWi = reinterpret_cast<const int32_t*>(part);
    } else {
        t.Q = reinterpret_cast<const int32_t*>(part);
        t.W = reinterpret_cast<const int32_t*>(part + 256);
    }
    return t;
}

// Shared memory per warp of the two-lane batched kernel: tables, descriptor,
// transpose buffer, sample slots.
__host__ __device__ constexpr int pair_warp_smem_bytes(unsigned mode) {
    return pair_tab_bytes(mode) + kDescBytes + kXBytes + kParkBytes;
}

// The two-lane tile implements the fused modes (samples in, inverse out) and
// the inverse pass alone (coefficients in, reconstruction and/or SSE out); the
// forward pass alone and the statistics modes keep the one-lane tile.
__host__ __device__ constexpr bool pair_mode_supported(unsigned mode) {
    return !(mode & (kStats | kStatsPrivate)) && (mode & kInverse) && !(mode & kLoadPix) == !!(mode & kLoadCoef) &&
           !((mode & kLoadCoef) && (mode & kStoreCoef));
}

// Loads rows 4h..4h+3 of block (by, bx) as two little-endian words each,
// with edge replication outside the plane.
__device__ __forceinline__ void load_rows4(const uint8_t* __restrict__ src, int pitch, int w, int hgt,
                                           int by, int bx, int h, bool vec, uint32_t (&pix)[4][2]) {
    const int x0 = bx * 8, y0 = by * 8 + 4 * h;
    if (vec && x0 + 8 <= w && by * 8 + 8 <= hgt) {
        const uint8_t* p = src + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(p + (size_t)j * pitch));
            pix[j][0] = v.x;
            pix[j][1] = v.y;
        }
    } else if (x0 + 8 <= w && by * 8 + 8 <= hgt && words_inside(src, pitch, w, hgt, y0, y0 + 3, x0)) {
        const uint8_t* p = src + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int j = 0; j < 4; ++j) load8_unaligned(p + (size_t)j * pitch, pix[j]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int yy = min(y0 + j, hgt - 1);
            const uint8_t* row = src + (size_t)yy * pitch;
            uint32_t wd[2] = {0u, 0u};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int xx = min(x0 + c, w - 1);
                wd[c >> 2] |= (uint32_t)__ldg(row + xx) << (8 * (c & 3));
            }
            pix[j][0] = wd[0];
            pix[j][1] = wd[1];
        }
    }
}

// Stores the in-plane part of rows 4h..4h+3 of block (by, bx).
__device__ __forceinline__ void store_rows4(uint8_t* __restrict__ dst, int pitch, int w, int hgt,
                                            int by, int bx, int h, bool vec, const uint32_t (&pix)[4][2]) {
    const int x0 = bx * 8, y0 = by * 8 + 4 * h;
    if (vec && x0 + 8 <= w && by * 8 + 8 <= hgt) {
        uint8_t* p = dst + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint2*>(p + (size_t)j * pitch) = make_uint2(pix[j][0], pix[j][1]);
    } else if (x0 + 8 <= w && by * 8 + 8 <= hgt) {
        uint8_t* p = dst + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int j = 0; j < 4; ++j) store8_unaligned(p + (size_t)j * pitch, pix[j]);
    } else {
        const int nr = min(4, hgt - y0), nc = min(8, w - x0);
        for (int j = 0; j < nr; ++j) {
            uint8_t* row = dst + (size_t)(y0 + j) * pitch + x0;
            for (int c = 0; c < nc; ++c) row[c] = (uint8_t)(pix[j][c >> 2] >> (8 * (c & 3)));
        }
    }
}

__device__ __forceinline__ int sample4(const uint32_t (&pix)[4][2], int j, int c) {
    return (int)((pix[j][c >> 2] >> (8 * (c & 3))) & 0xFFu);
}

__device__ __forceinline__ void sts128(uint8_t* p, int a, int b, int c, int d) {
    *reinterpret_cast<int4*>(p) = make_int4(a, b, c, d);
}
__device__ __forceinline__ int4 lds128(const uint8_t* p) { return *reinterpret_cast<const int4*>(p); }

// A lane's four sample rows in its 32-byte slot; the halves swap on every
// fourth lane so a quarter warp's 16-byte accesses hit distinct bank groups.
__device__ __forceinline__ void park_rows(uint8_t* slot, int sw, const uint32_t (&pix)[4][2]) {
    *reinterpret_cast<uint4*>(slot + 16 * sw) = make_uint4(pix[0][0], pix[0][1], pix[1][0], pix[1][1]);
    *reinterpret_cast<uint4*>(slot + 16 * (sw ^ 1)) = make_uint4(pix[2][0], pix[2][1], pix[3][0], pix[3][1]);
}
__device__ __forceinline__ void unpark_rows(const uint8_t* slot, int sw, uint32_t (&pix)[4][2]) {
    const uint4 a = *reinterpret_cast<const uint4*>(slot + 16 * sw);
    const uint4 b = *reinterpret_cast<const uint4*>(slot + 16 * (sw ^ 1));
    pix[0][0] = a.x; pix[0][1] = a.y; pix[1][0] = a.z; pix[1][1] = a.w;
    pix[2][0] = b.x; pix[2][1] = b.y; pix[3][0] = b.z; pix[3][1] = b.w;
}

// Rows U.. of a lane's four columns: quantised codes to the stage at xc and,
// for the fused modes, dequantised inputs of the inverse column pass.
template <unsigned MODE, bool FLT, int U = 0>
__device__ __forceinline__ void pair_quant_rows(const PairTabs& T, int h, uint8_t* xc, int sw, const float (&y)[4][8],
                                                int (&c)[4][8]) {
    if constexpr (U < 8) {
        const float4 mf = *reinterpret_cast<const float4*>(&T.Mf[4 * h + U * 8]);
        const float t0 = quant_code<FLT, U, 0>(y[0][U], mf.x, T.M + 4 * h);
        const float t1 = quant_code<FLT, U, 1>(y[1][U], mf.y, T.M + 4 * h);
        const float t2 = quant_code<FLT, U, 2>(y[2][U], mf.z, T.M + 4 * h);
        const float t3 = quant_code<FLT, U, 3>(y[3][U], mf.w, T.M + 4 * h);
        if (MODE & kStoreCoef)
            *reinterpret_cast<uint2*>(xc + ((U ^ sw) << 4)) = make_uint2(pack_codes(t0, t1), pack_codes(t2, t3));
        if (MODE & kInverse) {
            const float4 qw = *reinterpret_cast<const float4*>(&T.QW[4 * h + U * 8]);
            const float4 qc = *reinterpret_cast<const float4*>(&T.QWc[4 * h + U * 8]);
            c[0][U] = dequant_bits(t0, qw.x, qc.x);
            c[1][U] = dequant_bits(t1, qw.y, qc.y);
            c[2][U] = dequant_bits(t2, qw.z, qc.z);
            c[3][U] = dequant_bits(t3, qw.w, qc.w);
        }
        pair_quant_rows<MODE, FLT, U + 1>(T, h, xc, sw, y, c);
    }
}

// Processes halves hf0..hf1 - 1 (16 blocks each) of warp tile `tile_in_plane`
// of plane P.  xb is this warp's kXBytes transpose buffer followed by its
// kParkBytes sample slots.  Returns their SSE (the same in every lane; 0
// without kSse).
template <unsigned MODE>
__device__ __forceinline__ unsigned process_tile_pair(const PlaneArg& P, const PairTabs& T, int tile_in_plane,
                                                      int lane, uint8_t* xb, int hf0 = 0, int hf1 = 2) {
    static_assert(pair_mode_supported(MODE), "no two-lane form of this mode");
    const int k = lane >> 1, h = lane & 1;
    uint8_t* const xw = xb + k * kXSlot + h * kXRowHalf;   // rows 4h..4h+3, both quads
    uint8_t* const xr = xb + k * kXSlot + h * 16;           // rows 0..7, quad h
    // the DC input (column 0) belongs to lane h = 0
    const int dc_bias = h ? 0 : kDcBias;
    uint8_t* const park = xb + kXBytes + lane * 32;
    const int psw = (lane >> 2) & 1;
    unsigned e = 0;
    // block coordinates: one division per tile, then steps of 16 blocks
    const int bt = tile_in_plane * kTileBlocks;
    const int by_t = bt / P.nbx;
    const int bx_t = bt - by_t * P.nbx;

#pragma unroll 1
    for (int hf = hf0; hf < hf1; ++hf) {
        const int b0 = bt + hf * kPairBlocks;
        const int nvalid = min(kPairBlocks, P.nblk - b0);
        if (nvalid <= 0) break;                      // warp-uniform
        const bool active = k < nvalid;
        int by = by_t, bx = bx_t + hf * kPairBlocks + k;
        if (bx >= P.nbx) {
            bx -= P.nbx;
            ++by;
            if (bx >= P.nbx) {                       // planes narrower than 32 blocks
                by += bx / P.nbx;
                bx -= (bx / P.nbx) * P.nbx;
            }
        }

        int v[4][8];
        int c[4][8];
        uint32_t pix[4][2];
        if (MODE & kLoadPix) {
            // row pass on rows 4h..4h+3
            if (active) {
                load_rows4(P.src, P.src_pitch, P.width, P.height, by, bx, h, (P.flags & kVecSrc) != 0, pix);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) pix[j][0] = pix[j][1] = 0x80808080u;
            }
            float z[4][8];
#pragma unroll
            for (int j = 0; j < 4; ++j) pix_row(pix[j], z[j]);
            fwd_vectors<true>(z);

            // the samples wait for the SSE in this lane's slot (the two 16-byte
            // halves swap on every fourth lane: no bank conflicts)
            if (MODE & kSse) park_rows(park, psw, pix);

            // transpose: rows 4h..4h+3 out, columns 4h..4h+3 in
            __syncwarp();
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

            // column pass: z[i][u] = Y[u][4h + i]
            fwd_vectors<false>(z);

            // quantiser and own-code dequantiser; the codes go through the
            // transpose buffer (free between the two transposes) so that the
            // stores to global memory move 512 contiguous bytes each
            if (MODE & kStoreCoef) __syncwarp();             // transpose reads done
            uint8_t* const xc = xb + k * 128 + h * 8;
            if (T.Mf[0] != 0.0f) pair_quant_rows<MODE, true>(T, h, xc, k & 7, z, c);
            else pair_quant_rows<MODE, false>(T, h, xc, k & 7, z, c);
            if (MODE & kStoreCoef) {
                __syncwarp();
                uint4* const g = reinterpret_cast<uint4*>(P.coef + (size_t)b0 * 64) + lane;
                const uint8_t* const xs = xb + (lane >> 3) * 128;
#pragma unroll
                for (int i = 0; i < 4; ++i) {                // chunk 32 i + lane: block 4 i + lane / 8, row lane % 8
                    const uint4 w = *reinterpret_cast<const uint4*>(
                        xs + i * 512 + (((lane & 7) ^ ((4 * i + (lane >> 3)) & 7)) << 4));
                    if (4 * i + (lane >> 3) < nvalid) g[32 * i] = w;
                }
            }
        } else {
            // coefficients in: lane h reads the 8-byte half of each row u; the
            // SSE reference rows wait in its slot
            if (active) {
                const uint2* g = reinterpret_cast<const uint2*>(P.coef + (size_t)(b0 + k) * 64 + 4 * h);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint2 w = __ldg(g + 2 * u);
                    c[0][u] = (int)(int16_t)(w.x & 0xFFFFu);
                    c[1][u] = (int)w.x >> 16;
                    c[2][u] = (int)(int16_t)(w.y & 0xFFFFu);
                    c[3][u] = (int)w.y >> 16;
                }
                if (MODE & kSse) {
                    load_rows4(P.ref, P.ref_pitch, P.width, P.height, by, bx, h, (P.flags & kVecRef) != 0, pix);
                    park_rows(park, psw, pix);
                }
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) c[0][u] = c[1][u] = c[2][u] = c[3][u] = 0;
            }
            if constexpr ((MODE & kOwnCodes) != 0) {
                // this library's own codes (two-pass graph): G = q (Q W), the
                // clamp never acts (|q Q| < 1200)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int4 qw = *reinterpret_cast<const int4*>(T.QWi + 4 * h + u * 8);
                    c[0][u] *= qw.x;
                    c[1][u] *= qw.y;
                    c[2][u] *= qw.z;
                    c[3][u] *= qw.w;
                }
            } else {
                // dequantiser G = clamp(q Q, -4096, 4096) W for arbitrary codes
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int4 q4 = *reinterpret_cast<const int4*>(T.Q + 4 * h + u * 8);
                    const int4 w4 = *reinterpret_cast<const int4*>(T.W + 4 * h + u * 8);
                    c[0][u] = max(-kDequantClamp, min(kDequantClamp, c[0][u] * q4.x)) * w4.x;
                    c[1][u] = max(-kDequantClamp, min(kDequantClamp, c[1][u] * q4.y)) * w4.y;
                    c[2][u] = max(-kDequantClamp, min(kDequantClamp, c[2][u] * q4.z)) * w4.z;
                    c[3][u] = max(-kDequantClamp, min(kDequantClamp, c[3][u] * q4.w)) * w4.w;
                }
            }
        }
        if constexpr ((MODE & kInverse) != 0) {
            // inverse column pass, transpose back, inverse row pass
            constexpr int Z = (MODE & kLoadPix) ? kMagicBits : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) loeffler8_inv<Z>(c[i], i == 0 ? dc_bias : 0);
            __syncwarp();                                // transpose reads done
#pragma unroll
            for (int r = 0; r < 8; ++r)
                sts128(xr + (r >> 2) * kXRowHalf + (r & 3) * 32, c[0][r], c[1][r], c[2][r], c[3][r]);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int4 a = lds128(xw + j * 32);
                const int4 b = lds128(xw + j * 32 + 16);
                v[j][0] = a.x; v[j][1] = a.y; v[j][2] = a.z; v[j][3] = a.w;
                v[j][4] = b.x; v[j][5] = b.y; v[j][6] = b.z; v[j][7] = b.w;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) loeffler8_inv<0>(v[j], 0);

            uint32_t out[4][2];
#pragma unroll
            for (int j = 0; j < 4; ++j) descale_row(v[j], out[j]);
            if ((MODE & kStoreRecon) && active)
                store_rows4(P.dst, P.dst_pitch, P.width, P.height, by, bx, h, (P.flags & kVecDst) != 0, out);

            if ((MODE & kSse) && active) {
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
                        for (int cc = 0; cc < nc; ++cc) {
                            const int d = sample4(out, j, cc) - sample4(pix, j, cc);
                            e += d * d;
                        }
                }
            }
        }
    }
    return (MODE & kSse) ? warp_sum(e) : 0u;
}

// Direct (non-batched) calls with two lanes per block: grid-stride over the
// half tiles of up to kMaxPlanes planes, tables in shared memory, SSE
// summed per CTA and added to each plane's word once (zero on entry).
constexpr int kPairCodecHeader = 2 * (int)sizeof(QuantSet) + kMaxPlanes * 8;
static_assert(kPairCodecHeader % 16 == 0, "per-warp buffers must stay 16-byte aligned");

__host__ __device__ constexpr int pair_codec_smem_bytes(int threads) {
    return kPairCodecHeader + (threads / 32) * (kXBytes + kParkBytes);
}

template <unsigned MODE>
__global__ void __launch_bounds__(256, DCTGB_PAIR_MINB) k_codec_pair(const __grid_constant__ DirectArgs args) {
    extern __shared__ __align__(16) uint8_t smem[];
    QuantSet* tabs = reinterpret_cast<QuantSet*>(smem);
    unsigned long long* csse = reinterpret_cast<unsigned long long*>(smem + 2 * sizeof(QuantSet));
    {
        if (threadIdx.x < kMaxPlanes) csse[threadIdx.x] = 0ull;
        build_tabs(args.tabs, tabs);
    }
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int warps_per_cta = blockDim.x >> 5;
    uint8_t* xb = smem + kPairCodecHeader + warp * (kXBytes + kParkBytes);
    for (int unit = blockIdx.x * warps_per_cta + warp; unit < 2 * args.ntiles; unit += gridDim.x * warps_per_cta) {
        const int tile = unit >> 1, hf = unit & 1;
        int pi = 0;
#pragma unroll
        for (int k = 1; k < kMaxPlanes; ++k)
            if (k < args.nplanes && tile >= args.p[k].tile_begin) pi = k;
        const PlaneArg& P = args.p[pi];
        const uint8_t* part = reinterpret_cast<const uint8_t*>(&tabs[P.table]) + pair_tab_first(MODE);
        const unsigned e = process_tile_pair<MODE>(P, pair_tabs<MODE>(part), tile - P.tile_begin, lane, xb,
                                                       hf, hf + 1);
        if ((MODE & kSse) && lane == 0 && e) atomicAdd(&csse[pi], (unsigned long long)e);
    }
    __syncthreads();
    if (MODE & kSse) init_acc_wait();
    if ((MODE & kSse) && threadIdx.x < args.nplanes && csse[threadIdx.x])
        atomicAdd(args.p[threadIdx.x].sse, csse[threadIdx.x]);
}

// Host launcher of k_codec_pair: one grid of resident CTAs (direct_grid).  A
// call with fewer half tiles than warps in `num_sms` CTAs of `threads` gets
// smaller CTAs (down to two warps), so a small plane spreads over more SMs
// instead of sharing a few SMs' schedulers (a half tile takes one warp
// several microseconds, so that sharing sets the latency of the whole call).
template <unsigned MODE>
inline cudaError_t launch_codec_pair(const DirectArgs& a, int num_sms, int threads, cudaStream_t s) {
    const int units = 2 * a.ntiles;
    while (threads > 64 && (long long)units < (long long)num_sms * (threads / 32)) threads /= 2;
    const size_t smem = pair_codec_smem_bytes(threads);
    static OccCache cache;
    int occ = 0;
    cudaError_t e = kernel_occupancy(k_codec_pair<MODE>, cache, threads, smem, pair_codec_smem_bytes(kDirectThreads), occ);
    if (e != cudaSuccess) return e;
    return launch_behind_init(k_codec_pair<MODE>, direct_grid(units, threads, num_sms, occ), threads, smem, s, a,
                              (MODE & kSse) != 0);
}

}  // namespace dctgb
