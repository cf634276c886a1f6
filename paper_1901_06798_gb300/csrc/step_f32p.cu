// step_f32p.cu -- FP32 surface-perturbation form of the patch update: state
// (eta' = h + B, hu, hv) and B in FP32.  The surface jump that drives the waves
// is formed from eta' directly, so still water is exactly still and the
// ocean-depth cancellation of h + B never enters the flux.
#include <algorithm>
#include <atomic>
#include <cmath>
#include "step_tile_f32.cuh"

namespace tsu {

static constexpr int kThreadsF32 = 128;

int step_threads_f32p() { return kThreadsF32; }
int step_strip_width_f32p(int threads, int transverse) { return transverse ? threads - 4 : kTileCols; }

namespace {

constexpr int kSMs = 152;
int tile_smem(int rows) { return (rows + 4) * kTileRow * (int)sizeof(float); }

// CTAs of `threads` that fit on an SM: 16 warps of 128 registers, 228 KiB of
// shared memory of which each CTA takes 1 KiB beside its tile
int tile_ctas(int rows, int threads)
{
    return std::max(1, std::min(512 / threads, 228 * 1024 / (tile_smem(rows) + 1024)));
}

// above 48 KiB of dynamic shared memory a kernel has to be told so, once per device
template <typename K> int allow_smem(K kernel, std::atomic<unsigned long long> &told)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    if (dev < 64 && (told.load() >> dev & 1)) return 0;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(kTileRowsMax));
    if (e == cudaSuccess && dev < 64) told |= 1ull << dev;
    return (int)e;
}

template <int NW, bool GEO, bool BULK> int launch_tile(const StepArgs &a, int n, cudaStream_t st)
{
    static std::atomic<unsigned long long> told{0};
    const int e = allow_smem(step_tile_f32<NW, GEO, BULK>, told);
    if (e) return e;
    return launch_chained(step_tile_f32<NW, GEO, BULK>, n, NW * 32, tile_smem(a.tile_rows), st, a);
}

template <bool GEO> int launch_retake(const StepArgs &a, int n, cudaStream_t st)
{
    static std::atomic<unsigned long long> told{0};
    const int e = allow_smem(retake_tile_f32<GEO>, told);
    if (e) return e;
    StepArgs b = a;
    b.n_items = n;
    return launch_chained(retake_tile_f32<GEO>, std::min(n, kSMs * tile_ctas(a.tile_rows, 128)), 128, tile_smem(a.tile_rows),
                          st, b);
}

template <int NW> int launch_tile_nw(const StepArgs &a, int n, cudaStream_t st)
{
    const bool geo = a.kap != nullptr;
    if (a.bulk_rows) return geo ? launch_tile<NW, true, true>(a, n, st) : launch_tile<NW, false, true>(a, n, st);
    return geo ? launch_tile<NW, true, false>(a, n, st) : launch_tile<NW, false, false>(a, n, st);
}

}  // namespace

// The tile height that the model below finds fastest.  A tile of R rows takes
// about R + kOver row times (its ghost rows, the wait for its copies, the ramp of
// the y march); a second to fourth CTA on an SM slows the others by kShare each
// (they share the issue slots that one leaves free); tiles come in waves of as
// many CTAs as fit.
// Both sides of its choices, update alone, developed sea unless noted (us at rows 44 / 20 / 8):
// 4096^2 259 / 309 / 466 (it takes 44), 1531 x 1213 69.5 / 59.2 / 72.7 (24: 60.5),
// 500^2 41.0 / 30.0 / 29.3 (16: 27.2), 200^2 25.0 / 19.4 / 16.8 (12: 17.3); 7000 patches of
// 60^2, 16 steps: 6.7 ms at 60, 7.7 at 20, 8.8 at 16.  With 64 or 256 threads in place of 128
// the best heights take 269 and 289 us at 4096^2.
int tile_rows_f32p(int n, const int *nx, const int *ny, int threads)
{
    static const int cand[] = {4, 6, 8, 10, 12, 16, 20, 24, 30, 36, 44, 60};
    constexpr double kOver = 16.0, kShare = 0.15;
    const std::vector<double> strips = strips_by_height(n, nx, ny, kTileCols);
    int best = 44;
    double bc = 1e300;
    for (int R : cand) {
        const double items = tile_count(strips, R);
        const int occ = tile_ctas(R, threads);
        const double per = items / kSMs, full = std::floor(per / occ), rest = std::ceil(per - full * occ - 1e-9);
        const double one = R + kOver;
        const double c = full * one * (1.0 + kShare * (occ - 1)) + (rest > 0 ? one * (1.0 + kShare * (rest - 1)) : 0.0);
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

// Rows of the unsplit kernels' row segments (strips of threads - 4 columns), each
// of which sweeps 4 more and fills its pipeline.  FP32: about 16 warps run on an
// SM, which share its issue slots as the tiles' do.  FP64: an SM's CTAs share its
// FP64 pipe, so their times add up.
// Both sides (us): FP32 1024^2 took 172 with rows by a fixed 64, 70 with the rule's, 86 with 12;
// FP32 300^2 37 with the rule's and 45 with 64 threads; 2500^2 289 (rule), 286 to 298 at others.
int unsplit_rows(int n, const int *nx, const int *ny, int threads, int precision)
{
    static const int cand[] = {8, 12, 16, 24, 32, 48, 64};
    const bool f64 = precision == 0;
    const int W = threads - 4, occ = std::max(1, 512 / threads);
    const std::vector<double> strips = strips_by_height(n, nx, ny, W);
    int best = f64 ? 128 : 64;
    double bc = 1e300;
    for (int R : cand) {
        const double items = tile_count(strips, R);
        const double per = items / kSMs, full = std::floor(per / occ), rest = std::ceil(per - full * occ - 1e-9);
        const double one = R + 6;
        const double c = f64 ? std::ceil(per) * one
                             : full * one * (1.0 + 0.4 * (occ - 1)) + (rest > 0 ? one * (1.0 + 0.4 * (rest - 1)) : 0.0);
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

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
