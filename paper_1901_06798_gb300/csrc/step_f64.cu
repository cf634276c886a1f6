// step_f64.cu -- FP64 split update (step_tile_f64.cuh).  Built with --fmad=false so
// every multiply and add rounds exactly as the FP64 oracle's.
#include <algorithm>
#include <atomic>
#include <cmath>
#include "step_tile_f64.cuh"

namespace tsu {

namespace {

constexpr int kThreadsF64 = 128, kThreadsUnsplitF64 = 64;
constexpr int kSMs = 152;
int tile_smem(int rows) { return (rows + 4) * d1::kRow * (int)sizeof(double); }

template <int NW, bool GEO> int launch_tile(const StepArgs &a, int n, cudaStream_t st)
{
    // above 48 KiB of dynamic shared memory a kernel has to be told so, once per device
    static std::atomic<unsigned long long> told{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    if (dev >= 64 || !(told.load() >> dev & 1)) {
        e = cudaFuncSetAttribute(step_tile_f64<NW, GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(kTileRowsMaxF64));
        if (e != cudaSuccess) return (int)e;
        if (dev < 64) told |= 1ull << dev;
    }
    // (not launched ahead of the boundaries' end: placed around CTAs that are still
    // there, the tiles spread unevenly over the SMs, 0.33 -> 0.52 ms on 512^2 cells)
    if (a.gate == nullptr) {
        step_tile_f64<NW, GEO><<<n, NW * 32, tile_smem(a.tile_rows), st>>>(a);
        return (int)cudaGetLastError();
    }
    return launch_chained(step_tile_f64<NW, GEO>, n, NW * 32, tile_smem(a.tile_rows), st, a);
}

template <int NW> int launch_geo(const StepArgs &a, int n, cudaStream_t st)
{
    return a.kap != nullptr ? launch_tile<NW, true>(a, n, st) : launch_tile<NW, false>(a, n, st);
}

}  // namespace

int step_threads_f64(int transverse) { return transverse ? kThreadsUnsplitF64 : kThreadsF64; }
int step_strip_width_f64(int threads, int transverse) { return transverse ? threads - 4 : d1::kCols; }

// The tile height with the least time on the busiest SM.  A tile of R rows costs
// about 2 (R + 4) warp rows of x sweep and 2 (R / 2 + 3) of y march on each half of
// its columns (two segments); an SM's tiles share its FP64 pipe, so they add up.
// The four warps of one CTA leave the pipe idle between dependent instructions:
// alone it takes about 1.75 times, two take 1.2 times as long per unit of work as
// three or more, which is what fits.
// Both sides (us, developed sea): 771 x 602 543 with the rule's height, 941 with 16 rows,
// 687 with 12; 512^2 325 and 380 with 12; 2048^2 3972 and 4124 with 24.  256 threads in place
// of 128: 350 at 512^2, 595 at 771 x 602, but 115 against 127 at 200^2 and 241 against 333 where
// most of 512^2 is at rest; 64 threads: 398, 568, 191, 467.
int tile_rows_f64(int n, const int *nx, const int *ny)
{
    const std::vector<double> strips = strips_by_height(n, nx, ny, d1::kCols);
    int best = 32;
    double bc = 1e300;
    for (int R = 32; R >= 4; R -= 2) {
        const double per = std::ceil(tile_count(strips, R) / kSMs);
        const double c = per * (2.0 * (R + 4) + 4.0 * (R / 2 + 3)) * (per <= 1 ? 1.75 : (per <= 2 ? 1.2 : 1.0));
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

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
