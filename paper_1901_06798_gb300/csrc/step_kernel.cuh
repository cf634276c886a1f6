// step_kernel.cuh -- device functions of the patch update shared by its kernels:
// the normal Riemann solver with bed steps, dry states and walls, the MC-limited
// fluctuations and correction fluxes (Sec. 2.2 Eqs. wave_propagation_2nd_order,
// theta), wet/dry post-processing, Manning friction, and the copies into shared
// memory.
// The arithmetic of riemann()/limit() follows the FP64 oracle operation by
// operation; the FP64 instantiation is compiled without contraction so the
// two agree to the last bit.
#pragma once
#include <cuda_runtime.h>
#include "step_tail.cuh"
#include "tsu_device.h"

namespace tsu {

template <typename T> struct Wave {
    T Z[3][3];   // f-wave p, component (mass, normal, transverse)
    T s[3];
    int wall;    // 1: left side replaced by the wall mirror, 2: right side
};

template <typename T> __device__ __forceinline__ T dsqrt(T x);
template <> __device__ __forceinline__ double dsqrt<double>(double x) { return sqrt(x); }
template <> __device__ __forceinline__ float dsqrt<float>(float x) { return sqrtf(x); }
template <typename T> __device__ __forceinline__ T dmin(T a, T b);
template <> __device__ __forceinline__ double dmin<double>(double a, double b) { return fmin(a, b); }
template <> __device__ __forceinline__ float dmin<float>(float a, float b) { return fminf(a, b); }
template <typename T> __device__ __forceinline__ T dmax(T a, T b);
template <> __device__ __forceinline__ double dmax<double>(double a, double b) { return fmax(a, b); }
template <> __device__ __forceinline__ float dmax<float>(float a, float b) { return fmaxf(a, b); }
template <typename T> __device__ __forceinline__ T dabs(T a);
template <> __device__ __forceinline__ double dabs<double>(double a) { return fabs(a); }
template <> __device__ __forceinline__ float dabs<float>(float a) { return fabsf(a); }

// One cell as seen by a normal-direction Riemann problem: stored state (q0 is
// h, or eta' in the perturbation form), bed, and the quantities derived from
// it once per sweep -- depth, velocities, sqrt(g h), sqrt(h).
template <typename T> struct Cell {
    T q0, hn, ht, B;
    T h, u, v, c, sq;
    bool wet;
};

template <typename T, bool PERT>
__device__ __forceinline__ void derive(Cell<T> &z, T g, T drytol)
{
    z.h = PERT ? z.q0 - z.B : z.q0;
    z.wet = z.h >= drytol;
    z.u = T(0); z.v = T(0); z.c = T(0); z.sq = T(0);
    if (z.wet) {
        z.u = z.hn / z.h;
        z.v = z.ht / z.h;
        z.c = dsqrt<T>(g * z.h);
        z.sq = dsqrt<T>(z.h);
    }
}

// Normal-direction Riemann solver.  Augmented HLLE-type f-wave decomposition
// with the bathymetry source folded into the momentum flux jump,
// Einfeldt-type speeds from Roe averages, dry-bed speeds, a reflecting wall
// where a dry bed lies above the wet side's middle-state surface, a bed-step
// depth jump bounded so every state of the fan keeps h >= 0 (Sec. 2.2), and a
// contact wave at the Roe speed for the transverse momentum.
template <typename T, bool PERT>
__device__ __forceinline__ void riemann(const T g, const Cell<T> &cl, const Cell<T> &cr, Wave<T> &r)
{
    const T zero = T(0);
    r.wall = 0;
    if (!cl.wet && !cr.wet) {
#pragma unroll
        for (int p = 0; p < 3; p++) {
            r.s[p] = zero;
#pragma unroll
            for (int m = 0; m < 3; m++) r.Z[p][m] = zero;
        }
        return;
    }
    T qL = cl.q0, hnL = cl.hn, BL = cl.B, hL = cl.h, uL = cl.u, vL = cl.v, cL = cl.c, sqL = cl.sq;
    T qR = cr.q0, hnR = cr.hn, BR = cr.B, hR = cr.h, uR = cr.u, vR = cr.v, cR = cr.c, sqR = cr.sq;
    bool wetL = cl.wet, wetR = cr.wet;
    if (wetL && !wetR) {
        T a = cL + T(0.5) * uL;
        T hm = a > zero ? a * a / g : zero;
        if (hm + BL <= BR) {
            r.wall = 2;
            hR = hL; hnR = -hnL; BR = BL; uR = -uL; vR = vL; wetR = true; qR = qL; cR = cL; sqR = sqL;
        }
    } else if (!wetL && wetR) {
        T a = cR - T(0.5) * uR;
        T hm = a > zero ? a * a / g : zero;
        if (hm + BR <= BL) {
            r.wall = 1;
            hL = hR; hnL = -hnR; BL = BR; uL = -uR; vL = vR; wetL = true; qL = qR; cL = cR; sqL = sqR;
        }
    }

    T s1, s2, s3;
    if (wetL && wetR) {
        T uhat = (sqL * uL + sqR * uR) / (sqL + sqR);
        T chat = dsqrt<T>(g * (T(0.5) * (hL + hR)));
        s1 = dmin<T>(uL - cL, uhat - chat);
        s3 = dmax<T>(uR + cR, uhat + chat);
        s2 = uhat;
    } else if (wetL) {
        s1 = uL - cL;
        s3 = uL + T(2) * cL;
        s2 = uL;
    } else {
        s1 = uR - T(2) * cR;
        s3 = uR + cR;
        s2 = uR;
    }

    T hbar = T(0.5) * (hL + hR);
    T deta = PERT ? qR - qL : (hR + BR) - (hL + BL);
    T d2 = hnR - hnL;
    T d3 = (hnR * uR - hnL * uL) + (g * hbar) * deta;
    T d4 = hnR * vR - hnL * vL;
    T den = s3 - s1;
    // Non-negative depth: the bed step is a stationary wave across which the
    // depth jumps by delta (BL - BR keeps still water still).  With
    // M = s3 hR - s1 hL - d(hu), the fan's constant states have depths
    //   s1 < 0 < s3: (M - s3 delta)/den and (M - s1 delta)/den either side of x = 0;
    //   s1 >= 0:     hL + delta, then (M - s1 delta)/den;
    //   s3 <= 0:     (M - s3 delta)/den, then hR - delta.
    // A delta that would make one negative is moved to make it zero, and the
    // acoustic waves carry dh - delta instead of d(eta).
    T M = (s3 * hR - s1 * hL) - d2;
    T delta = BL - BR;
    bool bounded = false;
    if (s1 < zero && s3 > zero) {
        if (M - s3 * delta < zero) { delta = M / s3; bounded = true; }
        else if (M - s1 * delta < zero) { delta = M / s1; bounded = true; }
    } else if (s1 >= zero) {
        if (hL + delta < zero) { delta = -hL; bounded = true; }
        else if (s1 > zero && M - s1 * delta < zero) { delta = M / s1; bounded = true; }
    } else {
        if (hR - delta < zero) { delta = hR; bounded = true; }
        else if (s3 < zero && M - s3 * delta < zero) { delta = M / s3; bounded = true; }
    }
    T d1 = bounded ? (hR - hL) - delta : deta;
    T w1m = (s3 * d1 - d2) / den;
    T w1n = (s3 * d2 - d3) / den;
    T b1 = s1 * w1m, g1 = s1 * w1n;
    T b3 = s3 * (d1 - w1m), g3 = s3 * (d2 - w1n);

    r.Z[0][0] = b1; r.Z[0][1] = g1; r.Z[0][2] = b1 * vL;
    r.Z[2][0] = b3; r.Z[2][1] = g3; r.Z[2][2] = b3 * vR;
    r.Z[1][0] = zero; r.Z[1][1] = zero; r.Z[1][2] = (d4 - b1 * vL) - b3 * vR;
    r.s[0] = s1; r.s[1] = s2; r.s[2] = s3;
}

template <typename T> __device__ __forceinline__ T wleft(T s) { return s < T(0) ? T(1) : (s == T(0) ? T(0.5) : T(0)); }
template <typename T> __device__ __forceinline__ T wright(T s) { return s > T(0) ? T(1) : (s == T(0) ? T(0.5) : T(0)); }

template <typename T> __device__ __forceinline__ T mc_limiter(T theta)
{
    T t = T(0.5) * (T(1) + theta);
    t = dmin<T>(t, T(2));
    t = dmin<T>(t, T(2) * theta);
    return dmax<T>(T(0), t);
}

// Fluctuations and limited correction flux of one edge.  ZI[p][m]: the f-waves
// of the upwind neighbour chosen per wave (I = i-1 if s >= 0, else i+1).
template <typename T>
__device__ __forceinline__ void limit(const Wave<T> &r, const T (&ZI)[3][3], T dtdx,
                                      T (&amdq)[3], T (&apdq)[3], T (&F)[3])
{
    T wl0 = wleft<T>(r.s[0]), wl1 = wleft<T>(r.s[1]), wl2 = wleft<T>(r.s[2]);
    T wr0 = wright<T>(r.s[0]), wr1 = wright<T>(r.s[1]), wr2 = wright<T>(r.s[2]);
#pragma unroll
    for (int m = 0; m < 3; m++) {
        amdq[m] = (wl0 * r.Z[0][m] + wl1 * r.Z[1][m]) + wl2 * r.Z[2][m];
        apdq[m] = (wr0 * r.Z[0][m] + wr1 * r.Z[1][m]) + wr2 * r.Z[2][m];
    }
    if (r.wall == 2) { apdq[0] = T(0); apdq[1] = T(0); apdq[2] = T(0); }
    if (r.wall == 1) { amdq[0] = T(0); amdq[1] = T(0); amdq[2] = T(0); }
    T c[3] = {T(0), T(0), T(0)};
    if (r.wall == 0) {
#pragma unroll
        for (int p = 0; p < 3; p++) {
            const T *Zi = r.Z[p];
            T dii = (Zi[0] * Zi[0] + Zi[1] * Zi[1]) + Zi[2] * Zi[2];
            T phi = T(0);
            if (dii != T(0)) {
                T dIi = (ZI[p][0] * Zi[0] + ZI[p][1] * Zi[1]) + ZI[p][2] * Zi[2];
                phi = mc_limiter<T>(dIi / dii);
            }
            T s = r.s[p];
            T cp = (T(1) - dtdx * dabs<T>(s)) * phi;
            if (s < T(0)) cp = -cp;
            else if (s == T(0)) cp = T(0);
            c[p] = cp;
        }
    }
#pragma unroll
    for (int m = 0; m < 3; m++)
        F[m] = T(0.5) * ((c[0] * r.Z[0][m] + c[1] * r.Z[1][m]) + c[2] * r.Z[2][m]);
}

template <typename T, bool PERT>
__device__ __forceinline__ void postprocess(T &q0, T &qn, T &qt, T B, T drytol)
{
    if (PERT) {
        T h = q0 - B;
        if (h < T(0)) { q0 = B; h = T(0); }
        if (h < drytol) { qn = T(0); qt = T(0); }
    } else {
        if (q0 < T(0)) q0 = T(0);
        if (q0 < drytol) { qn = T(0); qt = T(0); }
    }
}

// Manning friction of one updated cell (Sec. 2.1 drag, read with the momentum
// magnitude: D = n^2 g sqrt(hu^2 + hv^2) / h^(7/3)), implicit in the
// momentum: hu, hv <- hu, hv / (1 + dt D) on a wet cell.  coef = n^2 g.
template <typename T> __device__ __forceinline__ T dpow(T x, T y);
template <> __device__ __forceinline__ double dpow<double>(double x, double y) { return pow(x, y); }
template <> __device__ __forceinline__ float dpow<float>(float x, float y) { return powf(x, y); }
template <typename T, bool PERT>
__device__ __forceinline__ void friction(T q0, T &hu, T &hv, T B, T drytol, T coef, T dt)
{
    const T h = PERT ? q0 - B : q0;
    if (!(h >= drytol)) return;
    const T D = (coef * dpow<T>(h, T(-7.0 / 3.0))) * dsqrt<T>(hu * hu + hv * hv);
    const T f = T(1) + dt * D;
    hu = hu / f;
    hv = hv / f;
}

__device__ __forceinline__ void cp_async_elem(void *smem, const void *gmem, int bytes)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if (bytes == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Bulk copies into shared memory completing on an mbarrier (one thread arms
// the barrier with the bytes to expect and issues the copies; every consumer
// polls the phase).  Waits are bounded: mbar_wait gives up after `polls` tests.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
// makes initialised barriers visible to the bulk copies (the async proxy)
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *b, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// bytes (a multiple of 16) from 16-byte aligned global src to 16-byte aligned shared dst
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *b)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(b))
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long *b, unsigned parity)
{
    unsigned r;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(r)
                 : "r"(smem_u32(b)), "r"(parity)
                 : "memory");
    return r != 0;
}
// true once the phase of the given parity has completed; false if it has not
// after `polls` tests
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity, unsigned polls)
{
    for (unsigned i = 0; i < polls; i++)
        if (mbar_test(b, parity)) return true;
    return false;
}
// polls of the final wait for copies still in flight after a wait gave up
constexpr unsigned kDrainPolls = 1u << 26;

__device__ __forceinline__ void atomic_max_speed(unsigned long long *dst, double v)
{
    atomicMax(dst, (unsigned long long)__double_as_longlong(v));
}

}  // namespace tsu
