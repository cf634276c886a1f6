// tile_rules.h -- heights of the patch update's work items (tiles of the split
// update, row segments of the unsplit one).  Host code without CUDA.
//
// Each rule weighs a list of heights by a model of its kernel and takes the
// fastest.  What a height costs depends on the patches only through the number of
// strips of each patch height: one entry for one patch, so that a step of a grid in
// the caller's memory, which asks on every call, pays for 12 to 15 evaluations (about
// 0.2 us) and no allocation.  A table over all heights from 1 to the patch's, scanned
// for each candidate, took 11 us at 1537 rows and 125 us at 16384 (2050 x 1537 FP32 cells:
// 100 us a step with it, 93 us without).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

namespace tsu {

constexpr int kSMs = 152;
constexpr int kTileWidth = 60;                             // columns of a tile of the split updates
constexpr int kTileRowBytes = 1024, kTileRowBytesF64 = 2048;   // shared memory of a tile's row
constexpr int kTileRowsMax = 124, kTileRowsMaxF64 = 104;   // the most rows of a tile that shared memory holds

// strips of patches of ny rows
struct HeightStrips {
    int ny;
    double strips;
};

inline std::vector<HeightStrips> strips_by_height(int n, const int *nx, const int *ny, int W)
{
    int top = 0;
    for (int k = 0; k < n; k++) top = std::max(top, ny[k]);
    std::vector<double> s((size_t)top + 1, 0.0);
    for (int k = 0; k < n; k++) s[ny[k]] += (double)((nx[k] + W - 1) / W);
    std::vector<HeightStrips> out;
    for (int y = 1; y <= top; y++)
        if (s[y] > 0.0) out.push_back({y, s[y]});
    return out;
}

// work items of at most R rows
inline double tile_count(const HeightStrips *s, int m, int R)
{
    double items = 0.0;
    for (int k = 0; k < m; k++) items += s[k].strips * (double)((s[k].ny + R - 1) / R);
    return items;
}

// rows of a patch's tiles, of at most `cap` rows: equal and even
inline int tile_cut(int ny, int cap)
{
    const int nt = (ny + cap - 1) / cap, r = (ny + nt - 1) / nt;
    return r + (r & 1) <= cap ? r + (r & 1) : r;
}

// FP32 split update: shared memory of a tile, and CTAs of `threads` that fit on an SM:
// 16 warps of 128 registers, 228 KiB of shared memory of which each CTA takes 1 KiB
// beside its tile
inline int tile_smem_f32(int rows) { return (rows + 4) * kTileRowBytes; }
inline int tile_smem_f64(int rows) { return (rows + 4) * kTileRowBytesF64; }
inline int tile_ctas_f32(int rows, int threads)
{
    return std::max(1, std::min(512 / threads, 228 * 1024 / (tile_smem_f32(rows) + 1024)));
}

// FP32 split update: the tile height that the model below finds fastest.  A tile of R
// rows takes about R + kOver row times (its ghost rows, the wait for its copies, the
// ramp of the y march); a second to fourth CTA on an SM slows the others by kShare each
// (they share the issue slots that one leaves free); tiles come in waves of as
// many CTAs as fit.
// Both sides of its choices, update alone, developed sea unless noted (us at rows 44 / 20 / 8):
// 4096^2 259 / 309 / 466 (it takes 44), 1531 x 1213 69.5 / 59.2 / 72.7 (24: 60.5),
// 500^2 41.0 / 30.0 / 29.3 (16: 27.2), 200^2 25.0 / 19.4 / 16.8 (12: 17.3); 7000 patches of
// 60^2, 16 steps: 6.7 ms at 60, 7.7 at 20, 8.8 at 16.  With 64 or 256 threads in place of 128
// the best heights take 269 and 289 us at 4096^2.
inline int tile_rows_f32p(const HeightStrips *s, int m, int threads)
{
    static const int cand[] = {4, 6, 8, 10, 12, 16, 20, 24, 30, 36, 44, 60};
    constexpr double kOver = 16.0, kShare = 0.15;
    int best = 44;
    double bc = 1e300;
    for (int R : cand) {
        const double items = tile_count(s, m, R);
        const int occ = tile_ctas_f32(R, threads);
        const double per = items / kSMs, full = std::floor(per / occ), rest = std::ceil(per - full * occ - 1e-9);
        const double one = R + kOver;
        const double c = full * one * (1.0 + kShare * (occ - 1)) + (rest > 0 ? one * (1.0 + kShare * (rest - 1)) : 0.0);
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

// FP64 split update: the tile height with the least time on the busiest SM.  A tile of R
// rows costs about 2 (R + 4) warp rows of x sweep and 2 (R / 2 + 3) of y march on each
// half of its columns (two segments); an SM's tiles share its FP64 pipe, so they add up.
// The four warps of one CTA leave the pipe idle between dependent instructions:
// alone it takes about 1.75 times, two take 1.2 times as long per unit of work as
// three or more, which is what fits.
// Both sides (us, developed sea): 771 x 602 543 with the rule's height, 941 with 16 rows,
// 687 with 12; 512^2 325 and 380 with 12; 2048^2 3972 and 4124 with 24.  256 threads in place
// of 128: 350 at 512^2, 595 at 771 x 602, but 115 against 127 at 200^2 (before narrow strips
// took two rows of a warp) and 241 against 333 where most of 512^2 is at rest; 64 threads:
// 398, 568, 191, 467.
inline int tile_rows_f64(const HeightStrips *s, int m)
{
    int best = 32;
    double bc = 1e300;
    for (int R = 32; R >= 4; R -= 2) {
        const double per = std::ceil(tile_count(s, m, R) / kSMs);
        const double c = per * (2.0 * (R + 4) + 4.0 * (R / 2 + 3)) * (per <= 1 ? 1.75 : (per <= 2 ? 1.2 : 1.0));
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

// Unsplit update, FP32: rows of its row segments (strips of threads - 4 columns), each
// of which sweeps 4 more and fills its pipeline.  About 16 warps run on an SM, which
// share its issue slots as the tiles' do.
// Both sides (us): 1024^2 took 172 with rows by a fixed 64, 70 with the rule's, 86 with 12;
// 300^2 37 with the rule's and 45 with 64 threads; 2500^2 289 (rule), 286 to 298 at others.
inline int unsplit_rows_f32p(const HeightStrips *s, int m, int threads)
{
    static const int cand[] = {8, 12, 16, 24, 32, 48, 64};
    const int occ = std::max(1, 512 / threads);
    int best = 64;
    double bc = 1e300;
    for (int R : cand) {
        const double items = tile_count(s, m, R);
        const double per = items / kSMs, full = std::floor(per / occ), rest = std::ceil(per - full * occ - 1e-9);
        const double one = R + 6;
        const double c = full * one * (1.0 + 0.4 * (occ - 1)) + (rest > 0 ? one * (1.0 + 0.4 * (rest - 1)) : 0.0);
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

// Unsplit update, FP64: the same segments.  Eight warps fit on an SM (shared memory); in
// units of two warps, a row of one, two or three alone takes 2.1, 2.3 and 3.3 times what
// it takes of the full four, where the FP64 pipe is busy.  Beyond that the SMs take
// segments as they finish: the rows shared out, and the end of the last segments (1.7).
// Both sides (us a step, developed sea, heights 8 / 16 / 32 / 64 / 128, then the rule's):
// 771 x 602 1556 / 1447 / 1569 / 2852 / 5575 (16), 1024^2 3051 / 2800 / 2727 / 3037 / 5588
// (32), 2000^2 10597 / 9699 / 10358 / 10295 / 10398 (16), 4096 x 1000 10577 / 9978 / 10403 /
// 10149 / 10388 (16); 1000 patches of 24^2 2771 / 3019, 2965 in one piece (8), 1600 of
// 60^2 15224 / 14053 / 14207, 14193 in one piece (16).  Counting whole segments an SM,
// whatever the number in flight, took 48 rows for 4096 x 1000: 11401.
inline int unsplit_rows_f64(const HeightStrips *s, int m, int threads)
{
    static const int cand[] = {8, 12, 16, 24, 32, 48, 64, 96, 128};
    static const double alone[] = {0.0, 2.1, 2.3, 3.3, 4.2};
    const double unit = threads / 64.0;
    double rows = 0.0;
    int top = 0;
    for (int k = 0; k < m; k++) {
        rows += s[k].strips * s[k].ny;
        top = std::max(top, s[k].ny);
    }
    int best = 64;
    double bc = 1e300;
    for (int R : cand) {
        const double items = tile_count(s, m, R), in_flight = std::ceil(items / kSMs - 1e-9) * unit, one = std::min(R, top) + 1.0;
        const double c = in_flight <= 4.0 ? one * alone[(int)in_flight] : (rows + items) / kSMs * unit + 1.7 * one;
        if (c < bc) { bc = c; best = R; }
    }
    return best;
}

// FP32 unsplit update: whether a launch of `items` CTAs, of which an SM holds `held`, is
// made ahead of its predecessor's end (chain.cuh).  Placed around CTAs that are still
// there, those of a launch that would leave every SM a slot pile up on some.  Where some SM
// is to hold all it can anyway nothing is lost, and three quarters as many CTAs as SMs find
// room beside the boundaries' CTAs.
// Both sides (us a step, ahead / after): 114 CTAs (300^2) 36.8 / 37.6, 152 (450^2) 48.6 /
// 46.8, 264 (700^2) 64.1 / 59.0, 416 (1500^2) 165.9 / 148.6, 442 (1600^2) 158.8 / 143.9, 469
// (800^2) 56.1 / 58.3, 504 (1700^2) 163.7 / 170.6, 576 (1024^2) 68.7 / 70.7, 1104 (2900^2)
// 398.2 / 398.9, all with 4 held; over 56 sizes 0.1% above the better of the two.
inline bool launch_ahead(int items, int held) { return 4LL * items <= 3LL * kSMs || items > kSMs * (held - 1); }

// The most rows of a work item for n patches of nx[k] x ny[k] cells advanced together,
// in strips of W columns by CTAs of `threads`
inline int work_rows(const HeightStrips *s, int m, int threads, bool split, bool f64)
{
    if (split) return f64 ? tile_rows_f64(s, m) : tile_rows_f32p(s, m, threads);
    return f64 ? unsplit_rows_f64(s, m, threads) : unsplit_rows_f32p(s, m, threads);
}
inline int work_rows(int n, const int *nx, const int *ny, int W, int threads, bool split, bool f64)
{
    if (n == 1) {
        const HeightStrips one{ny[0], (double)((nx[0] + W - 1) / W)};
        return work_rows(&one, 1, threads, split, f64);
    }
    const std::vector<HeightStrips> s = strips_by_height(n, nx, ny, W);
    return work_rows(s.data(), (int)s.size(), threads, split, f64);
}

// The launch shapes the autotuner times (threads, seg_rows): the library's own heights
// (0) and set ones.  None is another one under a second name: every set height is within
// what a tile can hold.
struct LaunchShape {
    int threads, seg_rows;
};
inline std::vector<LaunchShape> launch_shapes(bool split, bool f64)
{
    std::vector<LaunchShape> out;
    const bool tile32 = split && !f64;
    for (int t : {64, 128, 256, 32}) {
        if (t == 32 && !tile32) continue;
        for (int r : {0, 16, 32, 64, 128})
            if ((r != 16 || tile32) && !(split && r == 128)) out.push_back({t, r});
        if (tile32) out.push_back({t, kTileRowsMax});
    }
    return out;
}
// The rows the autotuner reports: those set, else a bound on the library's own, the most
// rows of a work item on any level: 32, 64 or 128 (which they never exceed)
inline int reported_rows(int seg_rows, int most)
{
    return seg_rows > 0 ? seg_rows : (most <= 32 ? 32 : (most <= 64 ? 64 : 128));
}

// The most rows of a work item: what the caller asks for (seg_rows > 0; tiles no taller
// than shared memory holds), else the rule's
inline int item_rows(int seg_rows, int n, const int *nx, const int *ny, int W, int threads, bool split, bool f64)
{
    if (seg_rows <= 0) return work_rows(n, nx, ny, W, threads, split, f64);
    return split ? std::min(seg_rows, f64 ? kTileRowsMaxF64 : kTileRowsMax) : seg_rows;
}

}  // namespace tsu
