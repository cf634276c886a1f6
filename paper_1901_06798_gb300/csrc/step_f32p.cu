// step_f32p.cu -- FP32 surface-perturbation form of the patch update: state
// (eta' = h + B, hu, hv) and B in FP32.  The surface jump that drives the waves
// is formed from eta' directly, so still water is exactly still and the
// ocean-depth cancellation of h + B never enters the flux.
#include <algorithm>
#include <atomic>
#include "step_tile_f32.cuh"

namespace tsu {

static constexpr int kThreadsF32 = 128;

int step_threads_f32p() { return kThreadsF32; }
int step_strip_width_f32p(int threads, int transverse) { return transverse ? threads - 4 : kTileCols; }

namespace {

static_assert(kTileCols == kTileWidth && kTileRow * sizeof(float) == kTileRowBytes, "the height rule's tile");

// above 48 KiB of dynamic shared memory a kernel has to be told so, once per device
template <typename K> int allow_smem(K kernel, std::atomic<unsigned long long> &told)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    if (dev < 64 && (told.load() >> dev & 1)) return 0;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem_f32(kTileRowsMax));
    if (e == cudaSuccess && dev < 64) told |= 1ull << dev;
    return (int)e;
}

template <int NW, bool GEO, bool BULK> int launch_tile(const StepArgs &a, int n, cudaStream_t st)
{
    static std::atomic<unsigned long long> told{0};
    const int e = allow_smem(step_tile_f32<NW, GEO, BULK>, told);
    if (e) return e;
    return launch_chained(step_tile_f32<NW, GEO, BULK>, n, NW * 32, tile_smem_f32(a.tile_rows), st, a);
}

template <bool GEO> int launch_retake(const StepArgs &a, int n, cudaStream_t st)
{
    static std::atomic<unsigned long long> told{0};
    const int e = allow_smem(retake_tile_f32<GEO>, told);
    if (e) return e;
    StepArgs b = a;
    b.n_items = n;
    return launch_chained(retake_tile_f32<GEO>, std::min(n, kSMs * tile_ctas_f32(a.tile_rows, 128)), 128, tile_smem_f32(a.tile_rows),
                          st, b);
}

template <int NW> int launch_tile_nw(const StepArgs &a, int n, cudaStream_t st)
{
    const bool geo = a.kap != nullptr;
    if (a.bulk_rows) return geo ? launch_tile<NW, true, true>(a, n, st) : launch_tile<NW, false, true>(a, n, st);
    return geo ? launch_tile<NW, true, false>(a, n, st) : launch_tile<NW, false, false>(a, n, st);
}

}  // namespace

// threads per CTA: 32, 64, 128 or 256
int launch_step_f32p(const StepArgs &a, int n_items, int threads, cudaStream_t st)
{
    if (n_items <= 0) return 0;
    if (a.transverse) return launch_unsplit_f32p(a, n_items, threads, st);
    if (a.tile_rows < 1 || a.tile_rows > kTileRowsMax) return (int)cudaErrorInvalidValue;
    // (every launch shape and way of copying gives the same bits)
    if (a.gate != nullptr) return a.kap != nullptr ? launch_retake<true>(a, n_items, st) : launch_retake<false>(a, n_items, st);
    switch (threads) {
    case 32: return launch_tile_nw<1>(a, n_items, st);
    case 64: return launch_tile_nw<2>(a, n_items, st);
    case 128: return launch_tile_nw<4>(a, n_items, st);
    case 256: return launch_tile_nw<8>(a, n_items, st);
    default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace tsu
