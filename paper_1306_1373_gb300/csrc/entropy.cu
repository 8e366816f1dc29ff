// Rate of the quantised coefficients (no counterpart in the paper, which never
// measures the compressed size): counts of the JPEG-style symbols of each
// plane, from which an ideal static code's length follows on the host.
//   DC  category of q00 - q00(previous block in block-major order), 0..15
//   AC  zig-zag run/size symbols; ZRL (0xF0) for every 16 zeros before a
//       non-zero value; EOB (0x00) when trailing zeros remain
//   amplitude bits: the category of every coded value
// One lane owns one block.  Its codes wait in a swizzled shared-memory stage
// (filled by cp.async one tile ahead); the lane turns them into a 64-bit mask of
// the non-zero zig-zag positions and walks the set bits only, so the run of
// zeros before a value is a difference of bit positions.  Symbol counts go to
// per-CTA shared histograms (one per plane) flushed once per CTA.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "host_common.h"

namespace dctgb {

constexpr int kEntWords = DCT_ENTROPY_WORDS;   // 16 DC + 256 AC + amplitude bits + blocks
constexpr int kMaxCodeLen = 16;                 // longest codeword of the prefix codes (as JPEG's Huffman tables)

// Natural index u*8+v of zig-zag position k (T.81 Figure A.6): diagonals
// s = u + v in turn, odd s with u rising, even s with u falling.
__host__ __device__ constexpr int zigzag_index(int k) {
    int n = 0;
    for (int s = 0; s < 15; ++s) {
        const int lo = s > 7 ? s - 7 : 0, hi = s < 7 ? s : 7;
        if (k < n + hi - lo + 1) {
            const int u = (s & 1) ? lo + (k - n) : hi - (k - n);
            return u * 8 + (s - u);
        }
        n += hi - lo + 1;
    }
    return 63;
}
static_assert(zigzag_index(2) == 8 && zigzag_index(3) == 16 && zigzag_index(63) == 63, "zig-zag order");

// Zig-zag position of natural index i, as a constant.
__host__ __device__ constexpr int zigzag_rank(int i) {
    for (int k = 0; k < 64; ++k)
        if (zigzag_index(k) == i) return k;
    return 0;
}

struct EntropyArgs {
    const int16_t* coef[kMaxPlanes];
    unsigned long long* out[kMaxPlanes];
    int32_t nblk[kMaxPlanes];
    int32_t tile_begin[kMaxPlanes + 1];
    int32_t nplanes;
};

__device__ __forceinline__ int category(int v) { return 32 - __clz(abs(v)); }

// Zig-zag mask bits of row U of a block (8 codes in w): bit zigzag_rank set
// where the code is not zero.
template <int U, int K = 0>
__device__ __forceinline__ void mask_row(const uint32_t (&w)[4], uint32_t& lo, uint32_t& hi) {
    if constexpr (K < 4) {
        constexpr int z0 = zigzag_rank(U * 8 + 2 * K), z1 = zigzag_rank(U * 8 + 2 * K + 1);
        if (w[K] & 0xFFFFu) (z0 < 32 ? lo : hi) |= 1u << (z0 & 31);
        if (w[K] >> 16) (z1 < 32 ? lo : hi) |= 1u << (z1 & 31);
        mask_row<U, K + 1>(w, lo, hi);
    }
}
template <int U = 0>
__device__ __forceinline__ void mask_block(const uint8_t* stage, int lane, uint32_t& lo, uint32_t& hi) {
    if constexpr (U < 8) {
        const uint4 v = *reinterpret_cast<const uint4*>(stage + stage_off(lane, U));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        mask_row<U>(w, lo, hi);
        mask_block<U + 1>(stage, lane, lo, hi);
    }
}

constexpr int kEntThreads = 128;
constexpr int kEntWarps = kEntThreads / 32;
constexpr int kEntSmem = kEntWarps * 2 * kStageBytes;   // two tiles of codes per warp

// Bound by instruction issue in the walk over the non-zero codes (a warp
// walks as long as its fullest block) and its two dependent shared-memory
// reads per code.  4K 4:2:0 codes at quality 75 (25 MB): 20.5 us a call; the
// walk over all 63 positions with the codes in registers, behind an upload of
// the block counts that the host waited for, took 35.6 us.
__global__ void __launch_bounds__(kEntThreads) k_entropy(const __grid_constant__ EntropyArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ unsigned int hist[kMaxPlanes][272];
    __shared__ unsigned long long amp[kMaxPlanes];
    __shared__ uint8_t where[64];       // byte offset u * 16 + v * 2 of zig-zag position k in a block
    for (int i = threadIdx.x; i < kMaxPlanes * 272; i += blockDim.x) (&hist[0][0])[i] = 0u;
    if (threadIdx.x < kMaxPlanes) amp[threadIdx.x] = 0ull;
    if (threadIdx.x < 64) where[zigzag_rank(threadIdx.x)] = (uint8_t)(threadIdx.x * 2);
    if (blockIdx.x == 0 && threadIdx.x < a.nplanes) a.out[threadIdx.x][273] = (unsigned long long)a.nblk[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int sw = (lane & 7) << 4;
    uint8_t* const buf = smem + (threadIdx.x >> 5) * 2 * kStageBytes;
    const int ntiles = a.tile_begin[a.nplanes];
    const int step = gridDim.x * kEntWarps;

    const auto plane_of = [&](int tile) {
        int pi = 0;
        while (pi + 1 < a.nplanes && tile >= a.tile_begin[pi + 1]) ++pi;
        return pi;
    };
    const auto fetch = [&](int tile, uint8_t* stage) {
        const int pi = plane_of(tile);
        const int b0 = (tile - a.tile_begin[pi]) * kTileBlocks;
        const int nvalid = min(kTileBlocks, a.nblk[pi] - b0);
        const uint8_t* g = reinterpret_cast<const uint8_t*>(a.coef[pi] + (size_t)b0 * 64);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int c = k * 32 + lane;
            if ((c >> 3) < nvalid) cp_async16(stage + stage_off(c >> 3, c & 7), g + (size_t)c * 16);
        }
    };

    int tile = blockIdx.x * kEntWarps + (threadIdx.x >> 5);
    if (tile < ntiles) fetch(tile, buf);
    cp_async_commit();
    for (int n = 0; tile < ntiles; tile += step, ++n) {
        if (tile + step < ntiles) fetch(tile + step, buf + ((n + 1) & 1) * kStageBytes);
        cp_async_commit();
        cp_async_wait<1>();
        __syncwarp();
        const uint8_t* const stage = buf + (n & 1) * kStageBytes;
        const int pi = plane_of(tile);
        const int b = (tile - a.tile_begin[pi]) * kTileBlocks + lane;
        unsigned* const h = hist[pi];
        unsigned bits = 0;
        if (b < a.nblk[pi]) {
            uint32_t lo = 0, hi = 0;
            mask_block(stage, lane, lo, hi);
            const int16_t* const dcs = reinterpret_cast<const int16_t*>(stage + stage_off(lane, 0));
            int prev = 0;
            if (lane > 0) prev = *reinterpret_cast<const int16_t*>(stage + stage_off(lane - 1, 0));
            else if (b > 0) prev = (int)__ldg(a.coef[pi] + (size_t)b * 64 - 64);
            const int dc = category((int)dcs[0] - prev);
            atomicAdd(&h[dc], 1u);
            bits = dc;
            int last = 0;                       // zig-zag position of the last coded value (DC first)
            const uint8_t* const blk = stage + lane * 128;
            for (unsigned long long m = ((unsigned long long)hi << 32 | lo) & ~1ull; m; m &= m - 1) {
                const int k = __ffsll((long long)m) - 1;
                const int o = where[k];
                const int v = *reinterpret_cast<const int16_t*>(blk + ((o & 0x70) ^ sw) + (o & 15));
                const int run = k - last - 1;
                last = k;
                if (run >= 16) atomicAdd(&h[16 + 0xF0], (unsigned)(run >> 4));
                const int s = category(v);
                atomicAdd(&h[16 + (((run & 15) << 4) | s)], 1u);
                bits += s;
            }
            if (last != 63) atomicAdd(&h[16 + 0x00], 1u);
        }
        const unsigned tot = __reduce_add_sync(0xffffffffu, bits);
        if (lane == 0 && tot) atomicAdd(&amp[pi], (unsigned long long)tot);
        __syncwarp();
    }
    cp_async_wait<0>();
    __syncthreads();
    for (int i = threadIdx.x; i < a.nplanes * 272; i += blockDim.x) {
        const int pl = i / 272, w = i - pl * 272;
        if (hist[pl][w]) atomicAdd(a.out[pl] + w, (unsigned long long)hist[pl][w]);
    }
    if (threadIdx.x < a.nplanes && amp[threadIdx.x]) atomicAdd(a.out[threadIdx.x] + 272, amp[threadIdx.x]);
}

}  // namespace dctgb

using namespace dctgb;

extern "C" dct_status dct_entropy_stats(dct_plan_t plan, const int16_t* coeffs, const dct_plane* planes, int nplanes,
                                        uint64_t* stats_out, dct_stream_t stream) {
    if (!plan || !coeffs || !planes || !stats_out) return fail(DCT_ERR_INVALID_ARG, "null pointer");
    if (nplanes < 1 || nplanes > kMaxPlanes) return fail(DCT_ERR_INVALID_ARG, "nplanes must be 1..4");
    if (((uintptr_t)coeffs) & 15u) return fail(DCT_ERR_INVALID_ARG, "coeffs must be 16-byte aligned");
    if (((uintptr_t)stats_out) & 7u) return fail(DCT_ERR_INVALID_ARG, "stats_out must be 8-byte aligned");
    EntropyArgs a;
    memset(&a, 0, sizeof a);
    size_t off = 0;
    int tiles = 0;
    for (int i = 0; i < nplanes; ++i) {
        const dct_plane& p = planes[i];
        if (p.width < 1 || p.height < 1 || p.width > plan->desc.max_width || p.height > plan->desc.max_height)
            return fail(DCT_ERR_INVALID_ARG, "plane size outside the plan limits");
        const int nblk = ((p.width + 7) / 8) * ((p.height + 7) / 8);
        a.coef[i] = coeffs + off;
        a.out[i] = reinterpret_cast<unsigned long long*>(stats_out) + (size_t)i * kEntWords;
        a.nblk[i] = nblk;
        a.tile_begin[i] = tiles;
        tiles += (nblk + kTileBlocks - 1) / kTileBlocks;
        off += (size_t)nblk * 64;
    }
    a.tile_begin[nplanes] = tiles;
    a.nplanes = nplanes;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(stats_out, 0, sizeof(uint64_t) * kEntWords * nplanes, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    int occ = 0;
    static OccCache cache;
    if ((e = kernel_occupancy(k_entropy, cache, kEntThreads, kEntSmem, kEntSmem, occ)) != cudaSuccess) return cuda_fail(e, "entropy kernel attributes");
    k_entropy<<<direct_grid(tiles, kEntThreads, plan->num_sms, occ), kEntThreads, kEntSmem, s>>>(a);
    e = cudaGetLastError();
    return e == cudaSuccess ? DCT_OK : cuda_fail(e, "entropy launch");
}

extern "C" double dct_entropy_bits(const uint64_t* stats_host) {
    if (!stats_host) return NAN;
    double bits = (double)stats_host[272];
    for (int part = 0; part < 2; ++part) {
        const int lo = part ? 16 : 0, hi = part ? 272 : 16;
        double n = 0.0;
        for (int i = lo; i < hi; ++i) n += (double)stats_host[i];
        for (int i = lo; i < hi; ++i)
            if (stats_host[i]) bits += (double)stats_host[i] * std::log2(n / (double)stats_host[i]);
    }
    return bits;
}

namespace dctgb {

// Codeword lengths of an optimal prefix code over the symbols with non-zero
// counts, none longer than max_len bits: package-merge (Larmore and
// Hirschberg).  Every level lists the leaves (sorted by count, then symbol)
// merged with the adjacent pairs of the previous level's list, leaves first
// on equal weights; a symbol's length is the number of times its leaf occurs
// among the first 2m - 2 items of the last level (m live symbols).  A lone
// symbol gets one bit.
static void limited_code_lengths(const uint64_t* counts, int n, int max_len, int* len) {
    struct Node {
        uint64_t w;
        int sym;      // leaf symbol, or -1 for a package
        int a, b;     // children of a package
    };
    std::vector<Node> nodes;
    std::vector<int> leaves;
    for (int i = 0; i < n; ++i) {
        len[i] = 0;
        if (counts[i]) {
            nodes.push_back(Node{counts[i], i, -1, -1});
            leaves.push_back((int)nodes.size() - 1);
        }
    }
    const int m = (int)leaves.size();
    if (m == 0) return;
    if (m == 1) {
        len[nodes[leaves[0]].sym] = 1;
        return;
    }
    std::sort(leaves.begin(), leaves.end(), [&](int x, int y) {
        return nodes[x].w != nodes[y].w ? nodes[x].w < nodes[y].w : nodes[x].sym < nodes[y].sym;
    });
    std::vector<int> cur = leaves, next, packages;
    for (int level = 1; level < max_len; ++level) {
        packages.clear();
        for (size_t k = 0; k + 1 < cur.size(); k += 2) {
            nodes.push_back(Node{nodes[cur[k]].w + nodes[cur[k + 1]].w, -1, cur[k], cur[k + 1]});
            packages.push_back((int)nodes.size() - 1);
        }
        next.clear();
        size_t x = 0, y = 0;
        while (x < leaves.size() || y < packages.size()) {
            if (y == packages.size() || (x < leaves.size() && nodes[leaves[x]].w <= nodes[packages[y]].w))
                next.push_back(leaves[x++]);
            else
                next.push_back(packages[y++]);
        }
        cur.swap(next);
    }
    std::vector<int> stack;
    for (int k = 0; k < 2 * m - 2; ++k) {
        stack.push_back(cur[k]);
        while (!stack.empty()) {
            const Node& nd = nodes[stack.back()];
            stack.pop_back();
            if (nd.sym >= 0) {
                ++len[nd.sym];
            } else {
                stack.push_back(nd.a);
                stack.push_back(nd.b);
            }
        }
    }
}

}  // namespace dctgb

extern "C" uint64_t dct_huffman_bits(const uint64_t* stats_host) {
    using namespace dctgb;
    if (!stats_host) return 0;
    uint64_t bits = stats_host[272];
    int len[256];
    for (int part = 0; part < 2; ++part) {
        const int lo = part ? 16 : 0, n = part ? 256 : 16;
        limited_code_lengths(stats_host + lo, n, kMaxCodeLen, len);
        for (int i = 0; i < n; ++i) bits += stats_host[lo + i] * (uint64_t)len[i];
    }
    return bits;
}
