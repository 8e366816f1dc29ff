// Forward-path kernels: level shift, 2-D Cordic-Loeffler DCT, quantiser,
// coefficient store (Sec. 2.5.2, Sec. 3.2): one lane per 8x8 block, with
// the optional statistics pass.
#include "kernels_pair.cuh"

namespace dctgb {

template <unsigned MODE>
static cudaError_t launch_mode(const DirectArgs& a, int num_sms, int threads, cudaStream_t s) {
    while (threads > 64 && (long long)a.ntiles < (long long)num_sms * (threads / 32)) threads /= 2;
    const size_t smem = codec_smem_bytes(threads);
    static OccCache cache;
    int occ = 0;
    cudaError_t e = kernel_occupancy(k_codec<MODE>, cache, threads, smem, codec_smem_bytes(kDirectThreads), occ);
    if (e != cudaSuccess) return e;
    return launch_behind_init(k_codec<MODE>, direct_grid(a.ntiles, threads, num_sms, occ), threads, smem, s, a,
                              (MODE & kStats) != 0);
}

cudaError_t launch_compress(const DirectArgs& a, bool stats, int num_sms, int threads, cudaStream_t s) {
    if (stats) return launch_mode<kLoadPix | kStoreCoef | kStats>(a, num_sms, threads, s);
    return launch_mode<kLoadPix | kStoreCoef>(a, num_sms, threads, s);
}

__global__ void k_init_acc(DirectArgs args, int do_sse, int do_stats) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int pl = 0; pl < args.nplanes; ++pl) {
        if (do_sse && threadIdx.x == 0) *args.p[pl].sse = 0ull;
        if (do_stats)
            for (int w = threadIdx.x; w < kStatsWords; w += blockDim.x)
                args.p[pl].stats[w] = (w == kStMin) ? ~0ull : 0ull;
    }
}

}  // namespace dctgb
