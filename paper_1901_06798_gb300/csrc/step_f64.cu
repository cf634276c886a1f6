// step_f64.cu -- FP64 split update (step_tile_f64.cuh).  Built with --fmad=false so
// every multiply and add rounds exactly as the FP64 oracle's.
#include <atomic>
#include "step_tile_f64.cuh"

namespace tsu {

namespace {

constexpr int kThreadsF64 = 128, kThreadsUnsplitF64 = 64;
static_assert(d1::kCols == kTileWidth && d1::kRow * sizeof(double) == kTileRowBytesF64, "the height rule's tile");

template <int NW, bool GEO> int launch_tile(const StepArgs &a, int n, cudaStream_t st)
{
    // above 48 KiB of dynamic shared memory a kernel has to be told so, once per device
    static std::atomic<unsigned long long> told{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    if (dev >= 64 || !(told.load() >> dev & 1)) {
        e = cudaFuncSetAttribute(step_tile_f64<NW, GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem_f64(kTileRowsMaxF64));
        if (e != cudaSuccess) return (int)e;
        if (dev < 64) told |= 1ull << dev;
    }
    // (not launched ahead of the boundaries' end: placed around CTAs that are still
    // there, the tiles spread unevenly over the SMs, 0.33 -> 0.52 ms on 512^2 cells)
    if (a.gate == nullptr) {
        step_tile_f64<NW, GEO><<<n, NW * 32, tile_smem_f64(a.tile_rows), st>>>(a);
        return (int)cudaGetLastError();
    }
    return launch_chained(step_tile_f64<NW, GEO>, n, NW * 32, tile_smem_f64(a.tile_rows), st, a);
}

template <int NW> int launch_geo(const StepArgs &a, int n, cudaStream_t st)
{
    return a.kap != nullptr ? launch_tile<NW, true>(a, n, st) : launch_tile<NW, false>(a, n, st);
}

}  // namespace

int step_threads_f64(int transverse) { return transverse ? kThreadsUnsplitF64 : kThreadsF64; }
int step_strip_width_f64(int threads, int transverse) { return transverse ? threads - 4 : d1::kCols; }

// threads per CTA: 64, 128 or 256
int launch_step_f64(const StepArgs &a, int n_items, int threads, cudaStream_t st)
{
    if (n_items <= 0) return 0;
    if (a.transverse) return launch_unsplit_f64(a, n_items, threads, st);
    if (a.tile_rows < 1 || a.tile_rows > kTileRowsMaxF64) return (int)cudaErrorInvalidValue;
    switch (threads) {
    case 64: return launch_geo<2>(a, n_items, st);
    case 128: return launch_geo<4>(a, n_items, st);
    case 256: return launch_geo<8>(a, n_items, st);
    default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace tsu
