// tsu_device.h -- structures shared by the library's host code and kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace tsu {

// One patch of a level: interior box [i0, i0+nx) x [j0, j0+ny) in global
// level indices, stored with 2 ghost cells per side.  The patch's block in the
// arena holds 7 fields of fs elements each: buffer 0 (q0, q1, q2), buffer 1
// (q0, q1, q2), B.  q0 is h (FP64 form) or eta' = h + B (FP32 perturbation
// form); q1 = hu, q2 = hv.  Element (i, j), -2 <= i < nx+2, at
// (j + 2) * pitch + (i + 2).
struct PatchDesc {
    long long off;      // element offset of the block in the arena
    long long fs;       // elements per field
    int i0, j0, nx, ny, pitch;
    int scen;
    int bcmask;         // 1 left, 2 right, 4 bottom, 8 top: ghost cells reach past that domain edge
    int nbr_off, nbr_cnt;      // same-level patches whose interior may feed this patch's ghosts
    int cmap_off, cmap_i0, cmap_j0, cmap_w, cmap_h;  // coarse-level patch index per coarse cell (levels >= 2)
    int ccand_off, ccand_cnt;  // coarse patches overlapping the coarse map's footprint (the map's painters)
    int old_off, old_cnt;      // old same-level patches overlapping (regrid initialisation)
};

// Where one ghost cell of a patch takes its value from, found once per patch
// table (the search over the neighbour boxes does not run at every fill):
// src >= 0 is the element offset in the arena of the same-level neighbour's
// interior cell in field 0 of buffer 0, sfs that patch's field stride; the
// negative codes below mark the other cases.
struct __align__(16) GhostSrc {
    long long src;
    long long sfs;
};
constexpr long long kGhostSkip = -1;     // outside the level's index space (physical boundary)
constexpr long long kGhostInterp = -2;   // no same-level neighbour: space-time interpolation from the coarser level
constexpr long long kGhostNone = -3;     // no neighbour on the coarsest level: a tiling error

// One work item of the patch update: a strip of columns [x0, x0+w) and a row
// segment [y0, y0+h) of one patch (patch-local interior indices).
struct StepItem {
    int patch;
    int x0, y0, w, h;
};

// Device control block of a context: per scenario dt, time, rates, counters.
struct CtrlView {
    double *dt1, *t;
    float *dt1f;                 // FP32 copy of dt1 for the perturbation-form kernel
    double *rate;                // [scen][max_levels]
    double *cell_updates;        // [scen]
    const double *cells;         // [scen][max_levels] interior cells per level
    long long *cfl_viol;         // [scen]
    unsigned long long *smax;    // [scen][2]
    int *retake;                 // [scen] 1: the level-1 step is being retaken (the step kernels' gate)
    long long *retakes;          // [scen] level-1 steps retaken
    int *err;                    // device error flag (TSU_DEV_ERR_*)
    int max_levels;
};

struct GaugeLoc {
    int level, patch;            // finest patch containing the gauge, or patch = -1
};

// What ends a level step (step_tail.cuh), done by the last CTA of the patch-update
// launch unless count is null.  mode as post_level's; end_step: then t += dt^1 and the gauge samples
// (one-level grids), unless a scenario is to be retaken.
struct TailArgs {
    CtrlView cv;
    unsigned *count;             // CTAs done, zero between launches
    int *any_retake;             // a scenario is marked for a retake (null: the step is never retaken)
    int level, nscen, mode, end_step;
    double R, dx, dy, cfl_max, cfl_desired;
    int ngauges;
    const GaugeLoc *gloc;        // [scen][gauge]
    const double *gxy;
    double *geta, *gt;
    long long *nsamp;
    double x0, y0, gdx, gdy;     // the level's origin and cell size in the gauges' coordinates
    double *speeds_out;          // set: only the two largest speeds go there (host memory)
};

// The most CTAs of a launch that are counted: two waves of the FP32 split update's (the
// launch saved, against the wait at the end of each wave).  Levels above the first,
// where counting saves one launch and not two, are counted up to a quarter of it.  The
// line matters little there: 3-level runs of 14 + 159 and 46 + 528 patches took 1.89 and
// 3.00 ms a coarse step with no finer level counted, 1.89 and 3.04 with this line, 1.90
// and 3.03 with all up to 1216; four scenarios with 33 patches in all 244, 244, 237 us.
constexpr int kTailMaxCtas = 1216;

struct StepArgs {
    const PatchDesc *descs;
    const StepItem *items;
    void *arena;
    int cur;                    // current buffer of this level (0 or 1)
    const double *dt1;          // level-1 time step per scenario
    unsigned long long *smax;   // per scenario: [2] max speed bits (x, y)
    double R;                   // refinement of this level relative to level 1
    double dx, dy, g, drytol;
    // FP32 copies for the perturbation-form kernel (no FP64 work per CTA)
    const float *dt1f;          // level-1 time step per scenario, FP32
    float rdx, rdy;             // 1 / (R dx), 1 / (R dy)
    float gf, drytolf, sqrtgf;
    int transverse;             // 1: unsplit update with transverse corrections
    double manning;             // n^2 g of the friction step (0: none)
    float manningf;
    float rR;                   // 1 / R (FP32 level time step = dt1f * rR)
    // latitude-longitude grids (capacity form): dx, dy above are the physical
    // sizes of an equatorial cell; capacity of global row J at kap[J + 2], relative
    // length of the latitude edge below row J at ced[J + 2]; null on Cartesian grids
    const double *kap, *ced;
    const float *kapf, *cedf;
    // FP32: 1 / capacity of row J at [J + 2]; length of the edge below row J over the mean capacity of its
    // two cells at [J + 2] (J >= -1)
    const float *rkapf, *cratf;
    // split update (step_tile_f32.cuh, step_tile_f64.cuh): the most rows of a work item, and,
    // with null items, the tile columns of the one patch the launch covers
    int tile_rows, tile_nsx;
    // FP32 split update: ghost-cell sources of the level's patches in ghost-ring order, patch k's from
    // gmap[goff[k]]; a tile of a patch inside the domain takes its ghost cells from there (null: from the
    // patch's own ghost ring)
    const GhostSrc *gmap;
    const long long *goff;
    // CFL retake of a level-1 step: when set, a work item of scenario s runs
    // only if gate[s] != 0 (null: every item runs)
    const int *gate;
    // device error flag (TSU_DEV_ERR_* bits; null: not reported); FP32 split
    // update: bulk copies of the tile's rows (0: per-thread cp.async) and the
    // polls a thread spends waiting for them before it gives up
    int *err;
    int bulk_rows;
    unsigned wait_polls;
    int n_items;                // work items (the FP32 split update's retake launch strides over them)
    TailArgs tail;
};

// device error flag bits: 1, 2, 4 a ghost, coarse or parent cell without a
// covering patch (nesting); 8 a non-finite wave speed or depth; 16 a wait for a
// bulk copy ran out of polls; 32 patch storage not aligned for bulk copies
enum { TSU_DEV_ERR_NESTING = 7, TSU_DEV_ERR_NAN = 8, TSU_DEV_ERR_TIMEOUT = 16, TSU_DEV_ERR_LAYOUT = 32 };

// FP32 launch constants of a level
inline void set_f32_constants(StepArgs &a)
{
    a.rdx = (float)(1.0 / (a.R * a.dx));
    a.rdy = (float)(1.0 / (a.R * a.dy));
    a.gf = (float)a.g;
    a.drytolf = (float)a.drytol;
    a.sqrtgf = (float)__builtin_sqrt(a.g);
    a.manningf = (float)a.manning;
    a.rR = (float)(1.0 / a.R);
}

// Launch helpers implemented in the .cu files.
int launch_step_f64(const StepArgs &a, int n_items, int threads, cudaStream_t st);
int launch_step_f32p(const StepArgs &a, int n_items, int threads, cudaStream_t st);
int launch_unsplit_f64(const StepArgs &a, int n_items, int threads, cudaStream_t st);
int launch_unsplit_f32p(const StepArgs &a, int n_items, int threads, cudaStream_t st);
int step_threads_f64(int transverse);
int step_threads_f32p();
// columns one work item of the patch update covers, for a launch of `threads`
// per CTA (the unsplit kernels take one column per thread in both precisions)
int step_strip_width_f64(int threads, int transverse);
int step_strip_width_f32p(int threads, int transverse);

}  // namespace tsu
