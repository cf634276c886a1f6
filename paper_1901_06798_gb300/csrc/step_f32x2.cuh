// step_f32x2.cuh -- device functions of the FP32 surface-perturbation patch
// update (dimensionally split, Sec. 2.2) on Blackwell's paired FP32
// instructions.
//
// Every per-cell and per-edge formula runs on float2 (__ffma2_rn, __fadd2_rn,
// __fmul2_rn): one issue slot for two edges or two cells.  Per-lane operations
// (reciprocal, square root, min/max, compares, selects) stay scalar.  The
// arithmetic is organised where FP32 rounding is held to the 1e-4 m surface bar
// rather than to the FP64 oracle's operation order:
//   * the wet-wet subsonic Riemann problem (the ocean) takes a short form; dry
//     beds, walls, dry pairs, supersonic fans and bounded bed steps take the
//     general solver.  The choice is made per edge, so an edge's waves do not
//     depend on which edge shares its pair, nor on the launch shape;
//   * A-dQ and A+dQ are sums of the waves weighted by the side each goes to:
//     1, 0, or 1/2 for a wave of speed 0, as in the oracle;
//   * the contact wave has only a transverse component, so an edge has 7 wave
//     components, and its limiter ratio is a quotient of scalars;
//   * no zero-norm test before theta = Z_I.Z / Z.Z: a zero wave contributes
//     0 to the correction whatever phi becomes (phi stays finite);
//   * phi / 2 = sat(min((1 + theta) / 4, theta)) is the MC limiter halved,
//     with the clamps to [0, 1] as one saturation.
// The limiter has two forms of the same operations: limit2 for any pair of
// edges, and limit2_ocean for pairs whose edges both took the short Riemann
// form.  There s1 < 0 < s3, so the acoustic waves' sides, signs and upwind
// neighbours are known and only the contact wave's are looked up; every weight
// left out multiplies an exact 0 or 1, so the two give the same bits.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include "step_kernel.cuh"

namespace tsu {
namespace x2 {

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b as one paired FMA
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
// c - a b
__device__ __forceinline__ float2 fnma(float2 a, float2 b, float2 c)
{
    return __ffma2_rn(make_float2(-a.x, -a.y), b, c);
}
__device__ __forceinline__ float2 fmin2(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
__device__ __forceinline__ float2 fmax2(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ float rcp1(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
// min and max that pass a NaN on
__device__ __forceinline__ float min_nan(float a, float b)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 rcp(float2 a) { return make_float2(rcp1(a.x), rcp1(a.y)); }
__device__ __forceinline__ float2 sqrt2(float2 a) { return make_float2(sqrtf(a.x), sqrtf(a.y)); }

// two cells in the roles of one sweep: q0 = eta', hn normal, ht transverse
// momentum, B; derived h, velocities, sqrt(g h), sqrt(h), momentum fluxes hn u, hn v
struct C2 {
    float2 q0, hn, ht, B;
    float2 h, u, v, c, sq, pn, pt;
    bool wx, wy;
};

// Two edges' waves: the first one negated (y0 = -Z^1, which saves the limiter a
// sign), the contact wave's transverse component, the third one; speeds, the
// first one negated too.
struct W2 {
    float2 y0m, y0n, y0t, z1t, z2m, z2n, z2t;
    float2 n0, s1, s2;
    int wallx, wally;
};

__device__ __forceinline__ void zero_waves(W2 &r)
{
    r.y0m = r.y0n = r.y0t = r.z1t = r.z2m = r.z2n = r.z2t = r.n0 = r.s1 = r.s2 = f2(0.0f);
    r.wallx = 0; r.wally = 0;
}

__device__ __forceinline__ void derive(C2 &z, float sqrtg, float drytol)
{
    z.h = sub(z.q0, z.B);
    z.wx = z.h.x >= drytol;
    z.wy = z.h.y >= drytol;
    const float2 rh = make_float2(z.wx ? rcp1(z.h.x) : 0.0f, z.wy ? rcp1(z.h.y) : 0.0f);
    z.u = mul(z.hn, rh);
    z.v = mul(z.ht, rh);
    z.sq = make_float2(sqrtf(z.wx ? z.h.x : 0.0f), sqrtf(z.wy ? z.h.y : 0.0f));
    z.c = mul(f2(sqrtg), z.sq);
    z.pn = mul(z.hn, z.u);
    z.pt = mul(z.hn, z.v);
}

// two wet cells whose depth z.h is set: the same values without the selects
__device__ __forceinline__ void derive_wet(C2 &z, float sqrtg)
{
    const float2 rh = rcp(z.h);
    z.wx = true; z.wy = true;
    z.u = mul(z.hn, rh);
    z.v = mul(z.ht, rh);
    z.sq = sqrt2(z.h);
    z.c = mul(f2(sqrtg), z.sq);
    z.pn = mul(z.hn, z.u);
    z.pt = mul(z.hn, z.v);
}

__device__ __forceinline__ void lane_in(const C2 &z, int l, Cell<float> &o)
{
    o.q0 = l ? z.q0.y : z.q0.x; o.hn = l ? z.hn.y : z.hn.x; o.ht = l ? z.ht.y : z.ht.x; o.B = l ? z.B.y : z.B.x;
    o.h = l ? z.h.y : z.h.x; o.u = l ? z.u.y : z.u.x; o.v = l ? z.v.y : z.v.x; o.c = l ? z.c.y : z.c.x;
    o.sq = l ? z.sq.y : z.sq.x; o.wet = l ? z.wy : z.wx;
}

// the general solver on lane l (0: x, 1: y) of two edges, into that lane of r
__device__ __forceinline__ void riemann2_lane(float g, const C2 &L, const C2 &R, int l, W2 &r)
{
    Cell<float> a, b;
    lane_in(L, l, a);
    lane_in(R, l, b);
    Wave<float> w;
    riemann<float, true>(g, a, b, w);
    if (l == 0) {
        r.y0m.x = -w.Z[0][0]; r.y0n.x = -w.Z[0][1]; r.y0t.x = -w.Z[0][2]; r.z1t.x = w.Z[1][2];
        r.z2m.x = w.Z[2][0]; r.z2n.x = w.Z[2][1]; r.z2t.x = w.Z[2][2];
        r.n0.x = -w.s[0]; r.s1.x = w.s[1]; r.s2.x = w.s[2];
        r.wallx = w.wall;
    } else {
        r.y0m.y = -w.Z[0][0]; r.y0n.y = -w.Z[0][1]; r.y0t.y = -w.Z[0][2]; r.z1t.y = w.Z[1][2];
        r.z2m.y = w.Z[2][0]; r.z2n.y = w.Z[2][1]; r.z2t.y = w.Z[2][2];
        r.n0.y = -w.s[0]; r.s1.y = w.s[1]; r.s2.y = w.s[2];
        r.wally = w.wall;
    }
}

// Riemann problems of two edges (L[i] | R[i]) for lanes i = x, y, in the short
// wet-wet form.  Returns per lane the least of the quantities that have to be
// positive for it to hold: -s1 and s3 (subsonic), and the middle depths either
// side of the bed step with the still-water jump, hL + W1 and hR - W3 (the
// depth bound is not needed).
__device__ __forceinline__ float2 riemann2_ocean(float g, const C2 &L, const C2 &R, W2 &r)
{
    const float2 num = fma(L.sq, L.u, mul(R.sq, R.u));
    const float2 uhat = mul(num, rcp(add(L.sq, R.sq)));
    const float2 h2 = add(L.h, R.h);
    const float2 chat = sqrt2(mul(f2(0.5f * g), h2)), ngh = mul(f2(-0.5f * g), h2);   // +- g times the mean depth
    const float2 n0 = fmax2(sub(L.c, L.u), sub(chat, uhat));
    const float2 s2 = fmax2(add(R.u, R.c), add(uhat, chat));
    const float2 d1 = sub(R.q0, L.q0);
    const float2 d2 = sub(R.hn, L.hn), nd2 = sub(L.hn, R.hn);
    const float2 nd3 = fma(ngh, d1, sub(L.pn, R.pn));
    const float2 rden = rcp(add(s2, n0));
    const float2 w1m = mul(fma(s2, d1, nd2), rden);
    const float2 w1n = mul(fma(s2, d2, nd3), rden);
    const float2 w3m = sub(d1, w1m);
    const float2 hl = add(L.h, w1m), hr = sub(R.h, w3m);
    r.y0m = mul(n0, w1m); r.y0n = mul(n0, w1n); r.y0t = mul(r.y0m, L.v);
    r.z2m = mul(s2, w3m); r.z2n = mul(s2, sub(d2, w1n)); r.z2t = mul(r.z2m, R.v);
    r.z1t = sub(add(sub(R.pt, L.pt), r.y0t), r.z2t);
    r.n0 = n0; r.s1 = uhat; r.s2 = s2;
    return make_float2(fminf(fminf(hl.x, hr.x), fminf(n0.x, s2.x)), fminf(fminf(hl.y, hr.y), fminf(n0.y, s2.y)));
}

// the same for any two edges: a lane whose cells are not both wet, or that the
// short form does not cover, is solved again by the general solver
__device__ __forceinline__ void riemann2(float g, const C2 &L, const C2 &R, W2 &r)
{
    const float2 ok = riemann2_ocean(g, L, R, r);
    r.wallx = 0; r.wally = 0;
    if (!(L.wx && R.wx && ok.x > 0.0f)) riemann2_lane(g, L, R, 0, r);
    if (!(L.wy && R.wy && ok.y > 0.0f)) riemann2_lane(g, L, R, 1, r);
}

// the share of a wave of speed s that goes to the right: 1, 0, or 1/2 at s = 0
__device__ __forceinline__ float2 right_share(float2 s)
{
    return make_float2(__saturatef(fmaf(s.x, 1e30f, 0.5f)), __saturatef(fmaf(s.y, 1e30f, 0.5f)));
}
// the products of an edge's waves with its upwind neighbour's
__device__ __forceinline__ float2 dot3(float2 am, float2 an, float2 at, float2 bm, float2 bn, float2 bt)
{
    return fma(am, bm, fma(an, bn, mul(at, bt)));
}
// half the MC limiter: phi / 2 = max(0, min((1 + th) / 4, 1, th)) = sat(min((1 + th) / 4, th))
__device__ __forceinline__ float2 mc_half(float2 th)
{
    const float2 a = fma(f2(0.25f), th, f2(0.25f));
    return make_float2(__saturatef(fminf(a.x, th.x)), __saturatef(fminf(a.y, th.y)));
}

// What two edges give their cells: S = A-dQ + F~ to the cell on the left (below),
// D = A+dQ - F~ to the one on the right (above).  d0, d2: products of the first
// and third waves with their upwind neighbours'; t1: the upwind contact waves.
// Correction factors c_p = 1/2 sgn(s)(1 - dt/dx |s|) phi = (sgn(s) - dt/dx s)(phi / 2).
// Any edges.
__device__ __forceinline__ void limit2(const W2 &r, float2 d0, float2 t1, float2 d2, float2 dtdx, float2 (&S)[3],
                                       float2 (&D)[3])
{
    const float2 one = f2(1.0f), mdt = make_float2(-dtdx.x, -dtdx.y);
    const float2 wl0 = right_share(r.n0), wr1 = right_share(r.s1), wr2 = right_share(r.s2);
    const float2 wr0 = sub(one, wl0), wl1 = sub(one, wr1), wl2 = sub(one, wr2);
    const float2 ng0 = sub(wl0, wr0), g1 = sub(wr1, wl1), g2 = sub(wr2, wl2);   // -sgn(s0), sgn(s1), sgn(s2)
    const float2 q0 = dot3(r.y0m, r.y0n, r.y0t, r.y0m, r.y0n, r.y0t), q2 = dot3(r.z2m, r.z2n, r.z2t, r.z2m, r.z2n, r.z2t);
    const float2 c0 = mul(fma(mdt, r.n0, ng0), mc_half(mul(d0, rcp(q0))));
    const float2 c1 = mul(fma(mdt, r.s1, g1), mc_half(mul(t1, rcp(r.z1t))));
    const float2 c2 = mul(fma(mdt, r.s2, g2), mc_half(mul(d2, rcp(q2))));
    const float2 F[3] = {fma(c0, r.y0m, mul(c2, r.z2m)), fma(c0, r.y0n, mul(c2, r.z2n)),
                         fma(c1, r.z1t, fma(c0, r.y0t, mul(c2, r.z2t)))};
    const float2 am[3] = {fnma(wl0, r.y0m, mul(wl2, r.z2m)), fnma(wl0, r.y0n, mul(wl2, r.z2n)),
                          fnma(wl0, r.y0t, mul(wl2, r.z2t))};
    const float2 ap[3] = {fma(wr2, r.z2m, mul(wr0, mul(f2(-1.0f), r.y0m))), fma(wr2, r.z2n, mul(wr0, mul(f2(-1.0f), r.y0n))),
                          fma(wr2, r.z2t, mul(wr0, mul(f2(-1.0f), r.y0t)))};
    S[0] = add(am[0], F[0]); D[0] = sub(ap[0], F[0]);
    S[1] = add(am[1], F[1]); D[1] = sub(ap[1], F[1]);
    S[2] = add(fma(wl1, r.z1t, F[2]), am[2]);
    D[2] = sub(fma(wr1, r.z1t, ap[2]), F[2]);
    if (r.wallx | r.wally) {
        // a wall edge: no fluctuation into the dry side, no correction
        const float2 at = fma(wl1, r.z1t, am[2]), bt = fma(wr1, r.z1t, ap[2]);
        if (r.wallx) {
            const bool l = r.wallx == 2;
            S[0].x = l ? am[0].x : 0.0f; S[1].x = l ? am[1].x : 0.0f; S[2].x = l ? at.x : 0.0f;
            D[0].x = l ? 0.0f : ap[0].x; D[1].x = l ? 0.0f : ap[1].x; D[2].x = l ? 0.0f : bt.x;
        }
        if (r.wally) {
            const bool l = r.wally == 2;
            S[0].y = l ? am[0].y : 0.0f; S[1].y = l ? am[1].y : 0.0f; S[2].y = l ? at.y : 0.0f;
            D[0].y = l ? 0.0f : ap[0].y; D[1].y = l ? 0.0f : ap[1].y; D[2].y = l ? 0.0f : bt.y;
        }
    }
}

// The same where both edges took the short Riemann form (s1 < 0 < s3), with the
// factor of the third wave apart: it needs only the edge on the left (below), so
// a march can form it as soon as the edge is solved.
__device__ __forceinline__ float2 third_factor(const W2 &r, float2 d2, float2 mdt)
{
    return mul(fma(mdt, r.s2, f2(1.0f)), mc_half(mul(d2, rcp(dot3(r.z2m, r.z2n, r.z2t, r.z2m, r.z2n, r.z2t)))));
}
__device__ __forceinline__ void limit2_ocean(const W2 &r, float2 d0, float2 t1, float2 c2, float2 mdt, float2 (&S)[3],
                                             float2 (&D)[3])
{
    const float2 one = f2(1.0f);
    const float2 wr1 = right_share(r.s1), wl1 = sub(one, wr1), g1 = sub(wr1, wl1);
    const float2 c0 = mul(fma(mdt, r.n0, one), mc_half(mul(d0, rcp(dot3(r.y0m, r.y0n, r.y0t, r.y0m, r.y0n, r.y0t)))));
    const float2 c1 = mul(fma(mdt, r.s1, g1), mc_half(mul(t1, rcp(r.z1t))));
    const float2 Fm = fma(c0, r.y0m, mul(c2, r.z2m));
    const float2 Fn = fma(c0, r.y0n, mul(c2, r.z2n));
    const float2 Ft = fma(c1, r.z1t, fma(c0, r.y0t, mul(c2, r.z2t)));
    S[0] = sub(Fm, r.y0m); D[0] = sub(r.z2m, Fm);
    S[1] = sub(Fn, r.y0n); D[1] = sub(r.z2n, Fn);
    S[2] = sub(fma(wl1, r.z1t, Ft), r.y0t);
    D[2] = sub(fma(wr1, r.z1t, r.z2t), Ft);
}

// Manning friction of two updated cells (as friction() in step_kernel.cuh)
__device__ __forceinline__ void friction2(float2 q0, float2 &hu, float2 &hv, float2 B, float drytol, float coef,
                                          float dt)
{
    const float2 h = sub(q0, B);
    const float2 m2 = fma(hu, hu, mul(hv, hv));
    float fx = 1.0f, fy = 1.0f;
    if (h.x >= drytol) fx = fmaf(dt, coef * __powf(h.x, -7.0f / 3.0f) * sqrtf(m2.x), 1.0f);
    if (h.y >= drytol) fy = fmaf(dt, coef * __powf(h.y, -7.0f / 3.0f) * sqrtf(m2.y), 1.0f);
    const float2 r = make_float2(__fdividef(1.0f, fx), __fdividef(1.0f, fy));
    hu = mul(hu, r);
    hv = mul(hv, r);
}

// wet/dry post-processing of two updated cells (perturbation form)
__device__ __forceinline__ void post2(float2 &q0, float2 &qn, float2 &qt, float2 B, float drytol)
{
    const float2 h = sub(q0, B);
    if (h.x < 0.0f) q0.x = B.x;
    if (h.y < 0.0f) q0.y = B.y;
    if (!(h.x >= drytol)) { qn.x = 0.0f; qt.x = 0.0f; }
    if (!(h.y >= drytol)) { qn.y = 0.0f; qt.y = 0.0f; }
}

__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void st2(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }

}  // namespace x2

}  // namespace tsu
