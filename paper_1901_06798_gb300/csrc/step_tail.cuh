// step_tail.cuh -- the end of a level step: the level's rate and CFL check
// (Sec. 2.2), and on a one-level grid the end of the coarse step and its gauge
// samples.  These were three launches of one block, about 2.2 us each in a
// replayed step.  They are one piece of work now, done by the last CTA of the patch
// update to finish where that launch is small, and else by a launch of its own
// (tail_kernel): counting CTAs makes each wait for its stores to land before it
// leaves, about 2 us for every wave of CTAs.  One step of a 200^2 grid 19.3 ->
// 17.1 us; with the count in every launch, a step of 14,000 AMR tiles took 43 us
// more than with none.
#pragma once
#include <cuda_runtime.h>
#include "chain.cuh"
#include "tsu_device.h"

namespace tsu {

// Scenario s after a level's step: the level's rate max(sx/dx, sy/dy) from the
// largest speeds sx, sy.
//   mode 0: a kept step -- count its cells, a violation if dt rate > cfl_max,
//           and fold the rate into the level's maximum;
//   mode 1: cell speeds of new patches -- the rate only;
//   mode 2: a level-1 step that may be retaken (Sec. 2.2 CFL condition): if
//           dt rate > cfl_max, mark the scenario for a retake and set
//           dt^1 = cfl_desired / rate (the state is still in the untouched
//           buffer); otherwise keep it as in mode 0;
//   mode 3: after the retake launch -- keep the retaken steps as in mode 0.
// A rate that is not a finite number (a NaN or infinite speed) sets the error
// flag to TSU_DEV_ERR_NAN.  Returns whether the scenario is to be retaken.
__device__ __forceinline__ bool post_level(const CtrlView &cv, int s, int level, double sx, double sy, double R, double dx,
                                           double dy, double cfl_max, double cfl_desired, int mode)
{
    if (mode == 3 && cv.retake[s] == 0) return false;
    const double rate = fmax(sx / dx, sy / dy);
    if (!(sx <= 1.0e300 && sy <= 1.0e300)) atomicOr(cv.err, TSU_DEV_ERR_NAN);
    double *ra = cv.rate + (long long)s * cv.max_levels + level;
    if (mode != 1) {
        const double dt = cv.dt1[s] / R;
        if (dt * rate > cfl_max) {
            if (mode == 2) {
                cv.retake[s] = 1;
                cv.retakes[s] += 1;
                cv.dt1[s] = cfl_desired / rate;
                cv.dt1f[s] = (float)cv.dt1[s];
                return true;
            }
            cv.cfl_viol[s] += 1;
        }
        if (mode == 2 || mode == 3) cv.retake[s] = 0;
        cv.cell_updates[s] += cv.cells[(long long)s * cv.max_levels + level];
    }
    *ra = fmax(*ra, rate);
    return false;
}

// eta at gauge c of the level's patches, bilinear between cell centres.  Rounds
// every operation (whatever the contraction mode of the file) as the gauges of
// refined runs do.
template <typename T, bool PERT>
__device__ __forceinline__ double gauge_eta(const PatchDesc &P, const T *blk, int cur, double gx, double gy, double x0,
                                            double y0, double dx, double dy)
{
    const double fx = __dadd_rn(__dadd_rn(gx, -x0) / dx, -0.5), fy = __dadd_rn(__dadd_rn(gy, -y0) / dy, -0.5);
    int ia = (int)floor(fx), ja = (int)floor(fy);
    double tx = __dadd_rn(fx, -(double)ia), ty = __dadd_rn(fy, -(double)ja);
    if (ia < P.i0) { ia = P.i0; tx = 0.0; }
    if (ia > P.i0 + P.nx - 2) { ia = P.i0 + P.nx - 2; tx = 1.0; }
    if (ja < P.j0) { ja = P.j0; ty = 0.0; }
    if (ja > P.j0 + P.ny - 2) { ja = P.j0 + P.ny - 2; ty = 1.0; }
    const T *q0 = blk + (long long)(cur * 3) * P.fs, *B = blk + 6LL * P.fs;
    double e[4];
#pragma unroll
    for (int m = 0; m < 4; m++) {
        const long long k = (long long)(ja - P.j0 + (m >> 1) + 2) * P.pitch + (ia - P.i0 + (m & 1) + 2);
        const double q = (double)__ldcg(q0 + k);   // written by other CTAs of this launch: not through L1
        e[m] = PERT ? q : __dadd_rn(q, (double)__ldcg(B + k));
    }
    const double a = __dadd_rn(e[0], __dmul_rn(tx, __dadd_rn(e[1], -e[0])));
    const double b = __dadd_rn(e[2], __dmul_rn(tx, __dadd_rn(e[3], -e[2])));
    return __dadd_rn(a, __dmul_rn(ty, __dadd_rn(b, -a)));
}

// First call of every patch-update kernel: whether this launch has anything to do: a retake launch (a.gate set) has not
// when no scenario is marked
__device__ __forceinline__ bool launch_live(const StepArgs &a)
{
    chain_begin();
    return a.gate == nullptr || a.tail.any_retake == nullptr || *a.tail.any_retake != 0;
}

template <typename T, bool PERT> __device__ __forceinline__ void end_level(const StepArgs &a)
{
    const TailArgs &tl = a.tail;
    if (tl.speeds_out != nullptr) {
        if (threadIdx.x < 2)
            tl.speeds_out[threadIdx.x] = __longlong_as_double((long long)atomicExch(a.smax + threadIdx.x, 0ull));
        return;
    }
    bool any = false;
    for (int s = threadIdx.x; s < tl.nscen; s += blockDim.x) {
        const double sx = __longlong_as_double((long long)atomicExch(tl.cv.smax + 2 * s, 0ull));
        const double sy = __longlong_as_double((long long)atomicExch(tl.cv.smax + 2 * s + 1, 0ull));
        any |= post_level(tl.cv, s, tl.level, sx, sy, tl.R, tl.dx, tl.dy, tl.cfl_max, tl.cfl_desired, tl.mode);
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0 && tl.any_retake) *tl.any_retake = any ? 1 : 0;
    if (any || !tl.end_step) return;   // the retake launch, or the caller, ends the step
    for (int s = threadIdx.x; s < tl.nscen; s += blockDim.x) tl.cv.t[s] = __dadd_rn(tl.cv.t[s], tl.cv.dt1[s]);
    if (tl.ngauges <= 0) return;
    __syncthreads();
    const long long sample = *tl.nsamp;
    for (int c = threadIdx.x; c < tl.nscen * tl.ngauges; c += blockDim.x) {
        const int s = c / tl.ngauges, q = c - s * tl.ngauges;
        double eta = __longlong_as_double(0x7ff8000000000000LL);
        const int p = tl.gloc[c].patch;
        if (p >= 0) {
            const PatchDesc P = a.descs[p];
            eta = gauge_eta<T, PERT>(P, reinterpret_cast<const T *>(a.arena) + P.off, 1 - a.cur, tl.gxy[2 * q],
                                     tl.gxy[2 * q + 1], tl.x0, tl.y0, tl.gdx, tl.gdy);
        }
        tl.geta[(sample * tl.nscen + s) * tl.ngauges + q] = eta;
        if (q == 0) tl.gt[sample * tl.nscen + s] = tl.cv.t[s];
    }
    __syncthreads();
    if (threadIdx.x == 0) *tl.nsamp = sample + 1;
}

// Every thread of every CTA of the launch calls it once, after its last work.
template <typename T, bool PERT> __device__ __forceinline__ void step_tail(const StepArgs &a)
{
    if (a.tail.count == nullptr) return;   // uniform over the launch
    __shared__ int role;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();   // the CTA's stores and speeds before its count
        role = atomicAdd(a.tail.count, 1u) + 1u == gridDim.x ? 1 : 0;
        if (role) *a.tail.count = 0u;
        __threadfence();
    }
    __syncthreads();
    if (role) end_level<T, PERT>(a);
}

}  // namespace tsu
