// Codec kernels: forward path (Sec. 2.5.2 transform + Sec. 3.2 quantiser),
// inverse path (Sec. 3.2 dequantiser + IDCT) and the SSE of Eq. 24, for
// uint8 planes.  The forward path computes the integers of the flow graph in
// float32 on the FMA pipes (cordic_loeffler.cuh), the inverse path in int32.
//
// Work decomposition: a plane of nbx x nby 8x8 blocks is cut into warp tiles
// of kTileBlocks consecutive blocks in block-major order (b = by * nbx + bx,
// wrapping across block rows).  Lane l of a warp owns block b0 + l and keeps
// its 64 samples in registers, so the row/column transpose between the two
// 1-D passes is free.  Pixel rows move 8 bytes per lane (a warp covers 256
// contiguous bytes of an image row); int16 coefficients go through a
// swizzled per-warp shared-memory stage so the global side moves 16 bytes
// per lane over contiguous 512-byte spans.  The batched kernel prefetches
// the next tile's pixels / coefficients with cp.async while the current
// tile computes.  The path is bound by instruction issue, not by HBM, so the
// code is arranged to minimise instructions per sample.
#pragma once
#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

#include "cordic_loeffler.cuh"
#include "dctgb_spec.h"

#ifndef DCTGB_MINB
#define DCTGB_MINB 2        // minimum resident CTAs per SM (launch bounds: <= 128 registers)
#endif

namespace dctgb {

constexpr int kMaxPlanes = 4;
constexpr int kTileBlocks = 32;                   // blocks per warp tile (one per lane)
constexpr int kStageBytes = kTileBlocks * 128;    // one tile of int16 coefficients
constexpr int kPixBytes = kTileBlocks * 64;       // one tile of uint8 samples

// Per-plane quantiser / dequantiser tables (natural order u*8+v).
// The float entries drive the kernels that quantise on the FMA pipes (see
// quant_code and dequant_bits).
// In the order of the parts that the batched kernels copy: the inverse of own
// codes reads QWi, the forward pass M and Mf, the fused one M to QWc, the inverse
// of any codes Q and W, and a two-pass batch QWi to Mf.
struct QuantSet {
    int32_t QWi[64];  // Q * W
    uint32_t M[64];   // rint(2^32 / (8 * 2^P * g_u g_v Q))
    float Mf[64];     // M * 2^-32, with the tie rule of quant_multiplier;
                      // Mf[0] = 0 when some M does not fit 24 bits
    float QW[64];     // Q * W
    float QWc[64];    // kMagic * (1 - Q * W)
    int32_t Q[64];    // 1..255
    int32_t W[64];    // rint(2^R / (g_u g_v))
};

struct PlaneArg {
    const uint8_t* src;       // samples (forward path, SSE reference in fused mode)
    int16_t* coef;            // block-major coefficients of this plane
    uint8_t* dst;             // reconstruction
    const uint8_t* ref;       // SSE reference for the inverse-only path
    unsigned long long* sse;  // per-plane SSE accumulator (global)
    unsigned long long* stats;// per-plane statistics words (global)
    int32_t src_pitch, dst_pitch, ref_pitch;
    int32_t width, height, nbx, nblk;
    int32_t table;            // index into the launch's QuantSet array
    int32_t tile_begin;       // first global tile index of this plane
    int32_t flags;            // kVecSrc | kVecDst | kVecRef
};
constexpr int kVecSrc = 1, kVecDst = 2, kVecRef = 4;

// What a direct call's kernel needs to build its two table sets (luma,
// chroma) in shared memory: a launch carries 768 bytes instead of 3.5 KB.
struct TabArgs {
    uint32_t M[2][64];
    uint16_t W[64];
    uint8_t Q[2][64];
};

struct DirectArgs {
    PlaneArg p[kMaxPlanes];
    TabArgs tabs;
    int32_t nplanes;
    int32_t ntiles;
};

// Mode bits of the kernel templates.
enum : unsigned {
    kLoadPix = 1u,     // read samples, forward transform, quantise
    kStoreCoef = 2u,   // write the quantised coefficients
    kLoadCoef = 4u,    // read quantised coefficients
    kInverse = 8u,     // dequantise, inverse transform, descale
    kStoreRecon = 16u, // write the reconstruction
    kSse = 32u,        // accumulate the SSE
    kStats = 64u,      // accumulate band-energy and pixel statistics
    kStatsPrivate = 128u, // the statistics sink is this warp's own: plain adds, no atomics
    kOwnCodes = 256u      // the coefficients read back are this library's own codes, written by the
                          // forward kernel of the same graph: the dequantiser clamp never acts
};

// ---- quantiser and own-code dequantiser on the FMA pipes ------------------
//
// Quantiser.  q = sgn(Y) ((|Y| M + 2^31) >> 32) is Y M / 2^32 rounded to the
// nearest integer, halves away from zero.  One fused multiply-add with
// kMagic = 1.5 * 2^23 (where a float32 counts ones) gives kMagic + q: the
// exact product is rounded once, to the nearest integer, halves to even.
// The two differ only at exact halves |Y| M = 2^31 (mod 2^32), which need
// |Y| = 2^(31-k) * odd, k = trailing zero bits of M; the forward graph keeps
// |Y| <= 719380 < 2^20 (interval bound), so k >= 12.  That happens only where
// u and v are both 0 or 4 (g_u g_v = 1, M = rint(2^25 / Q) a high power of two
// for Q = 1, 2, 4, ...); there the multiplier is the next float above
// M * 2^-32, which lifts the exact halves over the half and moves no other
// product across one (tests run every M at kN = 6, and those of 15 steps at kN = 4
// and 5, over every |Y|; that no half occurs elsewhere, at every step and kN).
// M must fit a float's 24 bits: only M > 2^24 (Q = 1, and Q = 2 at the
// smallest gains; quality 93 and up) may not, and tables with such an entry
// take the integer form (Mf[0] = 0).  The integer form costs a 64-bit multiply,
// which issues at 1/8 of the FMA rate (measured: 16 against 128 per clock per
// SM), and the conversions around it; this one costs half an issue slot.  Fused
// graph, 60 M samples: 106.5 us at quality 75, 112.7 at 95 (114.8 with the
// result's conversion in an addition of its own; 111 with integer arithmetic
// throughout, which takes 111 at quality 75 too).
constexpr float kMagic = 12582912.0f;               // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;              // its bits: bits(kMagic + q) = kMagicBits + q
__host__ __device__ constexpr bool tie_entry(int u, int v) { return (u & 3) == 0 && (v & 3) == 0; }
constexpr uint32_t kTieFreeBits = 0xFFFu;   // (M & kTieFreeBits) != 0  <=>  k <= 11

// The float multiplier of M (above): false when M needs more than 24 bits.
__host__ __device__ inline bool quant_multiplier(uint32_t m, float& out) {
    if ((m >> 24) && (m & ((2u << (m >> 25 ? (m >> 26 ? 2 : 1) : 0)) - 1u))) return false;   // M < 2^27
    const float f = (float)m;
    out = f * 2.3283064365386963e-10f;      // 2^-32
    if ((m & kTieFreeBits) == 0) {          // the next float above
        union { float f; uint32_t u; } b;
        b.f = out;
        b.u += 1u;
        out = b.f;
    }
    return true;
}

// Coefficient (u, v) to kMagic + q.
template <bool FLT, int U, int V>
__device__ __forceinline__ float quant_code(float y, float mf, const uint32_t* M) {
    if constexpr (FLT) return __fmaf_rn(y, mf, kMagic);
    // high word of Y M + 2^31, with - [Y < 0] where halves can occur (M < 2^26);
    // kMagicBits comes with the addend (the sum stays below 2^63)
    const int yi = __float_as_int(__fadd_rn(y, kMagic)) - kMagicBits;
    long long p = (long long)yi * (long long)(int)M[U * 8 + V] + (((long long)kMagicBits << 32) + 0x80000000ll);
    if (tie_entry(U, V)) p += (long long)(yi >> 31);
    return __int_as_float((int)(p >> 32));
}

// An own code kMagic + q, dequantised: G = q (Q W) as the integer kMagicBits +
// G, in one fused multiply-add: (kMagic + q) (Q W) + kMagic (1 - Q W) (QWc, an
// exact float: 3 (1 - Q W) 2^22 with Q W < 2^20).  The clamp of the definition
// never acts on this library's own codes: |q Q| <= |X| + Q/2 + 1 < 1200 (the
// Cordic coefficient |X| is within 14 of an orthonormal DCT value at kN = 6,
// itself at most 1024; < 1220 at kN = 4), so |G| < 1220 * 3025 < 2^22 and
// kMagic + G is an exact float32 integer.
__device__ __forceinline__ int dequant_bits(float t, float qw, float qwc) {
    return __float_as_int(__fmaf_rn(t, qw, qwc));
}

// The two table sets of a direct call, from its arguments into shared memory
// (every thread of the CTA; ends with a barrier).
__device__ __forceinline__ void build_tabs(const TabArgs& a, QuantSet* tabs) {
    bool exact = true;
    for (int i = threadIdx.x; i < 128; i += blockDim.x) {
        QuantSet& t = tabs[i >> 6];
        const int k = i & 63;
        const uint32_t m = a.M[i >> 6][k];
        const int q = a.Q[i >> 6][k], w = a.W[k];
        float mf = 0.0f;
        exact = quant_multiplier(m, mf) && exact;
        t.M[k] = m;
        t.Mf[k] = mf;
        t.QWi[k] = q * w;
        t.QW[k] = (float)(q * w);
        t.QWc[k] = kMagic * (1.0f - (float)(q * w));
        t.Q[k] = q;
        t.W[k] = w;
    }
    // a set with an inexact entry would need its own flag; both fall back
    // together, which only costs time
    if (!__syncthreads_and(exact)) {
        if (threadIdx.x < 2) tabs[threadIdx.x].Mf[0] = 0.0f;
        __syncthreads();
    }
}

// int16 pair of two codes kMagic + q: their low halves.
__device__ __forceinline__ uint32_t pack_codes(float t0, float t1) {
    return __byte_perm((uint32_t)__float_as_int(t0), (uint32_t)__float_as_int(t1), 0x5410);
}

// Clamp to 0..255 in one instruction: max(min(v, 255), 0).
__device__ __forceinline__ int clamp_u8(int v) { return __vimin_s32_relu(v, 255); }

// statistics word layout (per plane)
enum : int {
    kStBand = 0,         // 64 words: sum over blocks of (|Y_uv| >> kBandShift)^2
    kStSum = 64, kStSum2 = 65, kStMin = 66, kStMax = 67,
    kStAbsDx = 68, kStAbsDy = 69, kStDx2 = 70, kStDy2 = 71,
    kStLowAc = 72,       // 4 words: blocks whose AC energy < 2^10, 2^14, 2^18, 2^22
    kStBlocks = 76, kStSamples = 77
};

// --------------------------------------------------------------------------
// shared-memory layouts (swizzled, conflict-free for both access patterns)
// --------------------------------------------------------------------------

// Coefficient stage: block `blk` occupies 128 bytes; its row u (8 int16) sits
// in 16-byte slot u ^ (blk & 7).  A lane writing/reading the 8 rows of its own
// block and 8 lanes reading one block's 8 slots both hit 8 distinct
// 16-byte bank groups.
__device__ __forceinline__ int stage_off(int blk, int row) { return blk * 128 + ((row ^ (blk & 7)) << 4); }

// Pixel buffer: lane l's 8 rows of 8 bytes at l * 64; row r in 8-byte slot
// r ^ ((l >> 1) & 7), so 16 lanes reading one row each touch 32 distinct banks.
__device__ __forceinline__ int pix_off(int lane, int r) { return lane * 64 + ((r ^ ((lane >> 1) & 7)) << 3); }

// --------------------------------------------------------------------------
// asynchronous copies (completion via cp.async.wait_group: no spin loops)
// --------------------------------------------------------------------------

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// --------------------------------------------------------------------------
// sample I/O
// --------------------------------------------------------------------------

__device__ __forceinline__ bool interior(const PlaneArg& P, int by, int bx) {
    return bx * 8 + 8 <= P.width && by * 8 + 8 <= P.height;
}

// Eight bytes from any address, as aligned words and funnel shifts: three
// loads instead of eight (a plane with tight odd rows was bound by its byte
// accesses: 64 loads and 64 stores per block).  The words that hold the bytes
// must lie in the plane.
__device__ __forceinline__ void load8_unaligned(const uint8_t* p, uint32_t (&w)[2]) {
    const unsigned o = (unsigned)(uintptr_t)p & 3u;
    const uint32_t* q = reinterpret_cast<const uint32_t*>(p - o);
    const uint32_t a = __ldg(q), b = __ldg(q + 1), c = o ? __ldg(q + 2) : 0u;
    w[0] = __funnelshift_r(a, b, 8 * o);
    w[1] = __funnelshift_r(b, c, 8 * o);
}
// Whether load8_unaligned may read rows y0..y1 at column x0: its words then
// start at or after the plane's first byte and end at or before its last.
__device__ __forceinline__ bool words_inside(const uint8_t* src, int pitch, int w, int h, int y0, int y1, int x0) {
    const uintptr_t first = (uintptr_t)src, last = first + (size_t)(h - 1) * pitch + w;
    return (((uintptr_t)(src + (size_t)y0 * pitch + x0)) & ~(uintptr_t)3) >= first &&
           (((uintptr_t)(src + (size_t)y1 * pitch + x0 + 8) + 3) & ~(uintptr_t)3) <= last;
}

// Eight bytes to any address, as the widest aligned stores that cover them.
__device__ __forceinline__ void store8_unaligned(uint8_t* p, const uint32_t (&w)[2]) {
    const unsigned o = (unsigned)(uintptr_t)p & 3u;
    if (o == 0) {
        reinterpret_cast<uint32_t*>(p)[0] = w[0];
        reinterpret_cast<uint32_t*>(p)[1] = w[1];
    } else if (o == 2) {
        *reinterpret_cast<uint16_t*>(p) = (uint16_t)w[0];
        *reinterpret_cast<uint32_t*>(p + 2) = __funnelshift_r(w[0], w[1], 16);
        *reinterpret_cast<uint16_t*>(p + 6) = (uint16_t)(w[1] >> 16);
    } else {
        // one byte, then 2 + 4 bytes (o = 1) or 4 + 2 bytes (o = 3), one byte
        p[0] = (uint8_t)w[0];
        p[7] = (uint8_t)(w[1] >> 24);
        const uint32_t lo = __funnelshift_r(w[0], w[1], 8);          // bytes 1..4
        if (o == 1) {
            *reinterpret_cast<uint16_t*>(p + 1) = (uint16_t)lo;
            *reinterpret_cast<uint32_t*>(p + 3) = __funnelshift_r(w[0], w[1], 24);
        } else {
            *reinterpret_cast<uint32_t*>(p + 1) = lo;
            *reinterpret_cast<uint16_t*>(p + 5) = (uint16_t)(w[1] >> 8);
        }
    }
}

// Loads block (by, bx) as 8 rows of two little-endian uint32 words.  Samples
// outside the plane repeat the nearest edge sample (edge replication).
__device__ __forceinline__ void load_block(const uint8_t* __restrict__ src, int pitch, int w, int h,
                                           int by, int bx, bool vec, uint32_t (&pix)[8][2]) {
    const int x0 = bx * 8, y0 = by * 8;
    if (vec && x0 + 8 <= w && y0 + 8 <= h) {
        const uint8_t* p = src + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(p + (size_t)r * pitch));
            pix[r][0] = v.x;
            pix[r][1] = v.y;
        }
    } else if (x0 + 8 <= w && y0 + 8 <= h && words_inside(src, pitch, w, h, y0, y0 + 7, x0)) {
        const uint8_t* p = src + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int r = 0; r < 8; ++r) load8_unaligned(p + (size_t)r * pitch, pix[r]);
    } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int yy = min(y0 + r, h - 1);
            const uint8_t* row = src + (size_t)yy * pitch;
            uint32_t wd[2] = {0u, 0u};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int xx = min(x0 + c, w - 1);
                wd[c >> 2] |= (uint32_t)__ldg(row + xx) << (8 * (c & 3));
            }
            pix[r][0] = wd[0];
            pix[r][1] = wd[1];
        }
    }
}

// Issues cp.async copies of this lane's block of tile `tile_in_plane` into
// `buf` (a kPixBytes region) when the block is interior and the plane's rows
// are 8-byte aligned; the consumer re-evaluates the same condition.
__device__ __forceinline__ void prefetch_block(const PlaneArg& P, const uint8_t* base, int pitch, int vec_flag,
                                               int tile_in_plane, int lane, uint8_t* buf) {
    const int b = tile_in_plane * kTileBlocks + lane;
    if (b < P.nblk && (P.flags & vec_flag)) {
        const int by = b / P.nbx, bx = b - by * P.nbx;
        if (interior(P, by, bx)) {
            const uint8_t* p = base + (size_t)(by * 8) * pitch + bx * 8;
#pragma unroll
            for (int r = 0; r < 8; ++r) cp_async8(buf + pix_off(lane, r), p + (size_t)r * pitch);
        }
    }
}

// Issues cp.async copies of tile `tile_in_plane`'s coefficients into `stage`.
__device__ __forceinline__ void prefetch_coef(const PlaneArg& P, int tile_in_plane, int lane, uint8_t* stage) {
    const int b0 = tile_in_plane * kTileBlocks;
    const int nvalid = min(kTileBlocks, P.nblk - b0);
    const uint8_t* g = reinterpret_cast<const uint8_t*>(P.coef + (size_t)b0 * 64);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = k * 32 + lane;
        const int blk = c >> 3;
        if (blk < nvalid) cp_async16(stage + stage_off(blk, c & 7), g + (size_t)c * 16);
    }
}

// Block samples from the prefetch buffer when they were prefetched, else from
// global memory (edge blocks, unaligned planes, first tile of an item).
__device__ __forceinline__ void fetch_block(const PlaneArg& P, const uint8_t* base, int pitch, int vec_flag,
                                            const uint8_t* buf, int lane, int by, int bx, uint32_t (&pix)[8][2]) {
    if (buf && (P.flags & vec_flag) && interior(P, by, bx)) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint2 v = *reinterpret_cast<const uint2*>(buf + pix_off(lane, r));
            pix[r][0] = v.x;
            pix[r][1] = v.y;
        }
    } else {
        load_block(base, pitch, P.width, P.height, by, bx, (P.flags & vec_flag) != 0, pix);
    }
}

// Stores the in-plane part of block (by, bx).
__device__ __forceinline__ void store_block(uint8_t* __restrict__ dst, int pitch, int w, int h,
                                            int by, int bx, bool vec, const uint32_t (&pix)[8][2]) {
    const int x0 = bx * 8, y0 = by * 8;
    if (vec && x0 + 8 <= w && y0 + 8 <= h) {
        uint8_t* p = dst + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int r = 0; r < 8; ++r)
            *reinterpret_cast<uint2*>(p + (size_t)r * pitch) = make_uint2(pix[r][0], pix[r][1]);
    } else if (x0 + 8 <= w && y0 + 8 <= h) {
        uint8_t* p = dst + (size_t)y0 * pitch + x0;
#pragma unroll
        for (int r = 0; r < 8; ++r) store8_unaligned(p + (size_t)r * pitch, pix[r]);
    } else {
        const int nr = min(8, h - y0), nc = min(8, w - x0);
        for (int r = 0; r < nr; ++r) {
            uint8_t* row = dst + (size_t)(y0 + r) * pitch + x0;
            for (int c = 0; c < nc; ++c) row[c] = (uint8_t)(pix[r][c >> 2] >> (8 * (c & 3)));
        }
    }
}

__device__ __forceinline__ int sample(const uint32_t (&pix)[8][2], int r, int c) {
    return (int)((pix[r][c >> 2] >> (8 * (c & 3))) & 0xFFu);
}

__device__ __forceinline__ unsigned warp_sum(unsigned v) { return __reduce_add_sync(0xffffffffu, v); }

// statistics sink updates: atomics when the sink is shared, plain
// read-modify-write when it belongs to the calling warp
template <unsigned MODE>
__device__ __forceinline__ void st_add(unsigned long long* p, unsigned long long v) {
    if (MODE & kStatsPrivate) *p += v;
    else atomicAdd(p, v);
}
template <unsigned MODE>
__device__ __forceinline__ void st_min(unsigned long long* p, unsigned long long v) {
    if (MODE & kStatsPrivate) *p = *p < v ? *p : v;
    else atomicMin(p, v);
}
template <unsigned MODE>
__device__ __forceinline__ void st_max(unsigned long long* p, unsigned long long v) {
    if (MODE & kStatsPrivate) *p = *p > v ? *p : v;
    else atomicMax(p, v);
}

// Shared memory a warp needs in a given mode (batched kernel): its item's
// tables and descriptor, double-buffered samples and coefficient stages.
constexpr int kDescBytes = 128;
static_assert(sizeof(PlaneArg) <= kDescBytes, "descriptor slot too small");
constexpr int kStatBytes = kStatsWords * 8;   // warp-private statistics accumulator
__host__ __device__ constexpr int warp_smem_bytes(unsigned mode) {
    return (int)sizeof(QuantSet) + kDescBytes + ((mode & kStats) ? kStatBytes : 0) +
           (((mode & kLoadPix) || (mode & kSse)) ? 2 * kPixBytes : 0) +
           ((mode & kLoadCoef) ? 2 * kStageBytes : ((mode & kStoreCoef) ? kStageBytes : 0));
}

// --------------------------------------------------------------------------
// one warp tile
// --------------------------------------------------------------------------

// Added once to the DC input, which reaches every output through additions
// only: the descale rounding term 2^(R+2) and the +128 level.
constexpr int kDcBias = (1 << (kR + 2)) + (128 << (kR + 3));

// Eight outputs of the inverse row pass, descaled and clamped, to two words.
__device__ __forceinline__ void descale_row(const int (&v)[8], uint32_t (&out)[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t wd = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) wd |= (uint32_t)clamp_u8(v[4 * h + k] >> (kR + 3)) << (8 * k);
        out[h] = wd;
    }
}

// Columns V and V + 1 of the forward tile: column pass, band statistics,
// quantiser (code pairs to w), and in the fused modes dequantiser and inverse
// column pass (to x).
template <unsigned MODE, bool FLT, int V, int U = 0>
__device__ __forceinline__ void fwd_quant_rows(const QuantSet& T, const float (&y0)[8], const float (&y1)[8],
                                               uint32_t (&w)[8][4], int (&c0)[8], int (&c1)[8]) {
    if constexpr (U < 8) {
        const float2 mf = *reinterpret_cast<const float2*>(&T.Mf[U * 8 + V]);
        const float t0 = quant_code<FLT, U, V>(y0[U], mf.x, T.M), t1 = quant_code<FLT, U, V + 1>(y1[U], mf.y, T.M);
        if (MODE & kStoreCoef) w[U][V / 2] = pack_codes(t0, t1);
        if (MODE & kInverse) {
            const float2 qw = *reinterpret_cast<const float2*>(&T.QW[U * 8 + V]);
            const float2 qc = *reinterpret_cast<const float2*>(&T.QWc[U * 8 + V]);
            c0[U] = dequant_bits(t0, qw.x, qc.x);
            c1[U] = dequant_bits(t1, qw.y, qc.y);
        }
        fwd_quant_rows<MODE, FLT, V, U + 1>(T, y0, y1, w, c0, c1);
    }
}
template <unsigned MODE, bool FLT, int V>
__device__ __forceinline__ void fwd_tile_cols(const QuantSet& T, const float (&f)[8][8], bool active, int lane,
                                              unsigned long long* st, unsigned& ac, uint32_t (&w)[8][4], int (&x)[8][8]) {
    float y[2][8];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int r = 0; r < 8; ++r) y[k][r] = f[r][V + k];
    }
    fwd_vectors<false>(y);
    if (MODE & kStats) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const unsigned a = (unsigned)abs(__float2int_rn(y[k][u])) >> kBandShift;
                const unsigned e = active ? a * a : 0u;
                if (u | (V + k)) ac += e;
                const unsigned tot = warp_sum(e);
                if (lane == 0) st_add<MODE>(&st[kStBand + u * 8 + V + k], tot);
            }
        }
    }
    if (!(MODE & (kStoreCoef | kInverse))) return;
    int c0[8], c1[8];
    fwd_quant_rows<MODE, FLT, V>(T, y[0], y[1], w, c0, c1);
    if (MODE & kInverse) {
        loeffler8_inv<kMagicBits>(c0, V == 0 ? kDcBias : 0);
        loeffler8_inv<kMagicBits>(c1, 0);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            x[r][V] = c0[r];
            x[r][V + 1] = c1[r];
        }
    }
}

// All columns, with the quantiser form of the table: one warp-uniform branch
// per tile (one per coefficient row cost two instructions a sample and cut
// the column pass into small pieces).
template <unsigned MODE>
__device__ __forceinline__ void fwd_columns(const QuantSet& T, const float (&f)[8][8], bool active, int lane,
                                            unsigned long long* st, unsigned& ac, uint32_t (&w)[8][4], int (&x)[8][8]) {
    if (!(MODE & (kStoreCoef | kInverse)) || T.Mf[0] != 0.0f) {
        fwd_tile_cols<MODE, true, 0>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, true, 2>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, true, 4>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, true, 6>(T, f, active, lane, st, ac, w, x);
    } else {
        fwd_tile_cols<MODE, false, 0>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, false, 2>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, false, 4>(T, f, active, lane, st, ac, w, x);
        fwd_tile_cols<MODE, false, 6>(T, f, active, lane, st, ac, w, x);
    }
}

// Processes warp tile `tile_in_plane` of plane P.
//  stage      kStageBytes of this warp's shared memory (coefficients)
//  pixbuf     this tile's prefetched samples (forward) or SSE reference
//             (inverse), or nullptr
//  coef_ready the stage already holds this tile's coefficients
// Statistics go to the 80 words at `st` (shared or global); the return value
// is the tile's SSE (the same in every lane; 0 without kSse).
template <unsigned MODE>
__device__ __forceinline__ unsigned process_tile(const PlaneArg& P, const QuantSet& T, int tile_in_plane, int lane,
                                                 uint8_t* stage, const uint8_t* pixbuf, bool coef_ready,
                                                 unsigned long long* st) {
    const int b0 = tile_in_plane * kTileBlocks;
    const int nvalid = min(kTileBlocks, P.nblk - b0);
    const bool active = lane < nvalid;
    const int b = b0 + lane;
    int by = 0, bx = 0;
    if (active) {
        by = b / P.nbx;
        bx = b - by * P.nbx;
    }

    int x[8][8];
    uint32_t pix[8][2];

    if (MODE & kLoadPix) {
        if (active) {
            fetch_block(P, P.src, P.src_pitch, kVecSrc, pixbuf, lane, by, bx, pix);
        } else {
#pragma unroll
            for (int r = 0; r < 8; ++r) pix[r][0] = pix[r][1] = 0x80808080u;
        }

        if (MODE & kStats) {
            // four samples at a time: byte dot products, absolute
            // differences, minima and maxima (2.8 instructions per sample
            // against 14 one by one)
            unsigned s = 0, s2 = 0, adx = 0, ady = 0, dx2 = 0, dy2 = 0;
            unsigned mn4 = 0xFFFFFFFFu, mx4 = 0u;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                // right neighbours; the last column's is itself
                const uint32_t right[2] = {__funnelshift_r(pix[r][0], pix[r][1], 8), __byte_perm(pix[r][1], 0, 0x3321)};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t p = pix[r][h];
                    s = __dp4a(p, 0x01010101u, s);
                    s2 = __dp4a(p, p, s2);
                    mn4 = __vminu4(mn4, p);
                    mx4 = __vmaxu4(mx4, p);
                    const uint32_t dx = __vabsdiffu4(p, right[h]);
                    adx = __dp4a(dx, 0x01010101u, adx);
                    dx2 = __dp4a(dx, dx, dx2);
                    if (r < 7) {
                        const uint32_t dy = __vabsdiffu4(p, pix[r + 1][h]);
                        ady = __dp4a(dy, 0x01010101u, ady);
                        dy2 = __dp4a(dy, dy, dy2);
                    }
                }
            }
            unsigned mn = 255, mx = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                mn = min(mn, (mn4 >> (8 * k)) & 0xFFu);
                mx = max(mx, (mx4 >> (8 * k)) & 0xFFu);
            }
            if (!active) { s = s2 = adx = ady = dx2 = dy2 = 0; mn = 255; mx = 0; }
            const unsigned vals[8] = {warp_sum(s), warp_sum(s2), __reduce_min_sync(0xffffffffu, mn),
                                      __reduce_max_sync(0xffffffffu, mx), warp_sum(adx), warp_sum(ady),
                                      warp_sum(dx2), warp_sum(dy2)};
            if (lane == 0) {
                st_add<MODE>(&st[kStSum], vals[0]);
                st_add<MODE>(&st[kStSum2], vals[1]);
                st_min<MODE>(&st[kStMin], vals[2]);
                st_max<MODE>(&st[kStMax], vals[3]);
                st_add<MODE>(&st[kStAbsDx], vals[4]);
                st_add<MODE>(&st[kStAbsDy], vals[5]);
                st_add<MODE>(&st[kStDx2], vals[6]);
                st_add<MODE>(&st[kStDy2], vals[7]);
                st_add<MODE>(&st[kStBlocks], (unsigned long long)nvalid);
                st_add<MODE>(&st[kStSamples], (unsigned long long)nvalid * 64ull);
            }
        }

        float f[8][8];
#pragma unroll
        for (int r = 0; r < 8; ++r) pix_row(pix[r], f[r]);
        fwd_vectors<true>(f);

        // column pass, two columns at a time: statistics, quantiser, codes
        // and (fused modes) dequantiser and inverse column pass
        unsigned ac = 0;
        uint32_t w[8][4];
        fwd_columns<MODE>(T, f, active, lane, st, ac, w, x);

        if (MODE & kStats) {
            const unsigned thr[4] = {1u << 10, 1u << 14, 1u << 18, 1u << 22};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned n = warp_sum((active && ac < thr[k]) ? 1u : 0u);
                if (lane == 0) st_add<MODE>(&st[kStLowAc + k], n);
            }
        }

        if (MODE & kStoreCoef) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                *reinterpret_cast<uint4*>(stage + stage_off(lane, u)) = make_uint4(w[u][0], w[u][1], w[u][2], w[u][3]);
            __syncwarp();
            uint4* g = reinterpret_cast<uint4*>(P.coef + (size_t)b0 * 64);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int c = k * 32 + lane;
                const int blk = c >> 3;
                if (blk < nvalid) g[c] = *reinterpret_cast<const uint4*>(stage + stage_off(blk, c & 7));
            }
            __syncwarp();
        }
    }

    if (MODE & kLoadCoef) {
        if (!coef_ready) {
            const uint4* g = reinterpret_cast<const uint4*>(P.coef + (size_t)b0 * 64);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int c = k * 32 + lane;
                const int blk = c >> 3;
                if (blk < nvalid) *reinterpret_cast<uint4*>(stage + stage_off(blk, c & 7)) = __ldg(g + c);
            }
            __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint4 w = *reinterpret_cast<const uint4*>(stage + stage_off(lane, u));
            const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                x[u][2 * k] = (int)(int16_t)(ws[k] & 0xFFFFu);
                x[u][2 * k + 1] = (int)ws[k] >> 16;
            }
        }
        if (!active) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int v = 0; v < 8; ++v) x[u][v] = 0;
        }
    }

    if (MODE & kInverse) {
        // Dequantiser and inverse column pass of stored codes (the fused
        // modes did both above).  Codes written by the forward kernel of
        // the same graph need no clamp (dequant_bits): G = q (Q W).
        if (!(MODE & kLoadPix)) {
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                int c[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (MODE & kOwnCodes) {
                        c[u] = x[u][v] * T.QWi[u * 8 + v];
                    } else {
                        const int t = x[u][v] * T.Q[u * 8 + v];
                        c[u] = max(-kDequantClamp, min(kDequantClamp, t)) * T.W[u * 8 + v];
                    }
                }
                loeffler8_inv<0>(c, v == 0 ? kDcBias : 0);
#pragma unroll
                for (int r = 0; r < 8; ++r) x[r][v] = c[r];
            }
        }
        // inverse row pass, descale and clamp, four samples to a word
        uint32_t out[8][2];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            loeffler8_inv<0>(x[r], 0);
            descale_row(x[r], out[r]);
        }
        if ((MODE & kStoreRecon) && active)
            store_block(P.dst, P.dst_pitch, P.width, P.height, by, bx, (P.flags & kVecDst) != 0, out);

        if (MODE & kSse) {
            if (!(MODE & kLoadPix) && active) fetch_block(P, P.ref, P.ref_pitch, kVecRef, pixbuf, lane, by, bx, pix);
            unsigned e = 0;
            if (active) {
                const int nr = min(8, P.height - by * 8), nc = min(8, P.width - bx * 8);
                if (nr == 8 && nc == 8) {
                    // |r - p| per byte (vabsdiffu4), then the four squares and their
                    // sum in one dp4a
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const unsigned ad = __vabsdiffu4(out[r][h], pix[r][h]);
                            e = __dp4a(ad, ad, e);
                        }
                } else {
                    for (int r = 0; r < nr; ++r)
                        for (int c = 0; c < nc; ++c) {
                            const int d = sample(out, r, c) - sample(pix, r, c);
                            e += d * d;
                        }
                }
            }
            return warp_sum(e);
        }
    }
    return 0u;
}

// --------------------------------------------------------------------------
// persistent kernel over all tiles of up to kMaxPlanes planes (direct calls)
// --------------------------------------------------------------------------

// The kernel behind k_init_acc may start while it still runs (a programmatic
// dependent launch: k_init_acc lets its dependents go at once, so everything
// before it in the stream has finished) and waits for it only where it adds to
// the cleared words, at its end.  The clearing launch takes about 3 us by
// itself; 2731 x 1823 fused with unaligned rows: 18.4 us a call with it hidden
// and rows read as words, 20.5 us before.
__device__ __forceinline__ void init_acc_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct CtaAcc {
    unsigned long long sse[kMaxPlanes];
    unsigned long long st[kMaxPlanes][kStatsWords];
};

template <unsigned MODE>
__global__ void __launch_bounds__(256, DCTGB_MINB) k_codec(const __grid_constant__ DirectArgs args) {
    extern __shared__ __align__(16) uint8_t smem[];
    QuantSet* tabs = reinterpret_cast<QuantSet*>(smem);                       // 2 sets
    CtaAcc* acc = reinterpret_cast<CtaAcc*>(smem + 2 * sizeof(QuantSet));
    uint8_t* stage_all = smem + 2 * sizeof(QuantSet) + sizeof(CtaAcc);

    // tables -> shared memory
    {
        unsigned long long* a = reinterpret_cast<unsigned long long*>(acc);
        for (int i = threadIdx.x; i < (int)(sizeof(CtaAcc) / 8); i += blockDim.x) a[i] = 0ull;
        build_tabs(args.tabs, tabs);
        if (MODE & kStats) {
            if (threadIdx.x < kMaxPlanes) acc->st[threadIdx.x][kStMin] = ~0ull;
            __syncthreads();
        }
    }

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    uint8_t* stage = stage_all + warp * kStageBytes;
    const int warps_per_cta = blockDim.x >> 5;
    const int total_warps = gridDim.x * warps_per_cta;

    for (int tile = blockIdx.x * warps_per_cta + warp; tile < args.ntiles; tile += total_warps) {
        int pi = 0;
#pragma unroll
        for (int k = 1; k < kMaxPlanes; ++k)
            if (k < args.nplanes && tile >= args.p[k].tile_begin) pi = k;
        const PlaneArg& P = args.p[pi];
        const unsigned e = process_tile<MODE>(P, tabs[P.table], tile - P.tile_begin, lane, stage, nullptr, false,
                                              acc->st[pi]);
        if ((MODE & kSse) && lane == 0 && e) atomicAdd(&acc->sse[pi], (unsigned long long)e);
    }

    __syncthreads();
    if (MODE & (kSse | kStats)) init_acc_wait();
    if (MODE & kSse) {
        if (threadIdx.x < args.nplanes && acc->sse[threadIdx.x])
            atomicAdd(args.p[threadIdx.x].sse, acc->sse[threadIdx.x]);
    }
    if (MODE & kStats) {
        for (int i = threadIdx.x; i < args.nplanes * kStatsWords; i += blockDim.x) {
            const int pl = i / kStatsWords, w = i - pl * kStatsWords;
            const unsigned long long v = acc->st[pl][w];
            unsigned long long* g = args.p[pl].stats + w;
            if (w == kStMin) {
                if (v != ~0ull) atomicMin(g, v);
            } else if (w == kStMax) {
                atomicMax(g, v);
            } else if (v) {
                atomicAdd(g, v);
            }
        }
    }
}

// zero the SSE words and the statistics (min words to all ones)
__global__ void k_init_acc(DirectArgs args, int do_sse, int do_stats);

template <typename Args>
inline cudaError_t launch_behind_init(void (*kernel)(Args), int grid, int threads, size_t smem, cudaStream_t s,
                                      const Args& a, bool init) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = init ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

inline size_t codec_smem_bytes(int threads) {
    return 2 * sizeof(QuantSet) + sizeof(CtaAcc) + (size_t)(threads / 32) * kStageBytes;
}

// Grid of a direct call: enough CTAs for every unit of work (one warp each);
// beyond the resident count, a persistent grid of c CTAs per SM, each warp
// taking every (grid size)-th unit.  Every SM then issues c * rounds units
// per warp position, so c (at least two thirds of the resident count, to keep
// the latencies hidden) is the one that wastes the least in the last round: a
// 4K 4:2:0 frame is 40 tiles per SM, 3 rounds of 14 warps instead of 16.
inline int direct_grid(int units, int threads, int num_sms, int occ) {
    const int warps = threads / 32;
    if (occ < 1) occ = 1;
    const long long need = ((long long)units + warps - 1) / warps;
    if (need <= (long long)num_sms * occ) return need < 1 ? 1 : (int)need;
    int best = occ;
    long long best_cost = 0;
    for (int c = occ; c >= 1 && 3 * c >= 2 * occ; --c) {
        const long long per_round = (long long)num_sms * c * warps;
        const long long cost = (((long long)units + per_round - 1) / per_round) * c;
        if (best_cost == 0 || cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return num_sms * best;
}

// Resident CTAs per SM of a direct call's kernel at a CTA size (32 << i
// threads).  It is a property of the loaded kernel on a device, so it is asked
// once per device and size, after raising the kernel's shared-memory limit to
// what its largest CTA needs (the limit belongs to the kernel, not to a size).
// The two calls took 2 us of the 12.5 us of host time of a small direct call;
// with the raw stream query of the Python binding it is down to 7.9 us.
struct OccCache {
    std::atomic<int> occ[64][4] = {};       // [device][log2(threads / 32)], 0: not asked yet
};
template <typename Kernel>
inline cudaError_t kernel_occupancy(Kernel kernel, OccCache& c, int threads, size_t smem, size_t smem_max,
                                    int& occ) {
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) device = -1;
    const int i = threads == 32 ? 0 : threads == 64 ? 1 : threads == 128 ? 2 : 3;
    const bool cached = device >= 0 && device < 64;
    if (cached && (occ = c.occ[device][i].load(std::memory_order_acquire)) > 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
    if (e == cudaSuccess && cached && occ > 0) c.occ[device][i].store(occ, std::memory_order_release);
    return e;
}

// host launchers (one translation unit per family); kDirectThreads per CTA
constexpr int kDirectThreads = 128;
cudaError_t launch_compress(const DirectArgs& a, bool stats, int num_sms, int threads, cudaStream_t s);
cudaError_t launch_reconstruct(const DirectArgs& a, bool sse, int num_sms, int threads, cudaStream_t s);
cudaError_t launch_fused(const DirectArgs& a, bool coef, bool recon, int num_sms, int threads, cudaStream_t s);

}  // namespace dctgb
