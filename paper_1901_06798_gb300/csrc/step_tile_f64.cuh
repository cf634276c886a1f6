// step_tile_f64.cuh -- the FP64 split step (Sec. 2.2, x sweep then y sweep) of
// every patch of a level in one launch, bit for bit the FP64 oracle's.
//
// GB300 issues an FP64 warp instruction once in 16 cycles per SM, two orders below
// its other pipes, so the FP64 instructions are what the step costs and everything
// here serves to issue fewer of them and to keep all SMs' FP64 pipes busy:
//   * a CTA takes a tile of up to 60 columns x h rows with its two ghost cells per
//     side in shared memory, sweeps it in x in place and then in y to the output
//     (as step_tile_f32.cuh); tile heights follow the size of the level so that a
//     512^2 grid spreads over the whole chip;
//   * compares, selects, minima, maxima, signs and the halvings and quarterings of
//     the limiter are integer operations on the bit patterns;
//   * quantities of one cell (hn u, hn v, sqrt(h) u, u +- c, h + B) are formed once
//     and not at each of its edges;
//   * where every cell of a warp's row is wet and every edge subsonic with no
//     bounded bed step, the terms that are an exact 0 or a factor of exactly 1 are
//     left out of the limiter (wave 1 goes left, wave 3 right; the contact wave has
//     only a transverse component).  That the depth bound does not act is decided
//     in FP32 with a margin far above its rounding;
//   * where every cell is wet and at rest under a level surface, nothing is solved:
//     all waves are exact zeros, and the largest speed is sqrt(g h) of the deepest
//     cell, as the edge's mean depth lies between its cells' and every operation
//     is monotone.
// What remains is the oracle's arithmetic, operation for operation.  The FP64 pipe is
// 84% busy while CTAs run.  A fused kernel of one-column threads over 32-row segments
// with FP64 compares and selects took 3642 us for a 512^2 step mostly at rest (36
// CTAs) and 3170 us for 771 x 602 developed cells; this one takes 335 and 557 us.
// GEO: latitude-longitude grid in capacity form (Sec. 2.1 spherical coordinates):
// the x sweep of row j runs with dt / (kap_j dx) and reports speeds / kap_j; a
// y-edge's fluctuations and correction flux are weighted by its relative length
// ced_e, its Courant number uses dt ced_e / (kbar_e dy) (kbar_e the mean capacity
// of its two cells), the cell update divides by kap_j, and the mass gets the term
// (ced_{j+1} - ced_j) hv_j of the varying edge length.
#pragma once
#include <type_traits>
#include "step_kernel.cuh"
#include "tile_rules.h"

namespace tsu {
namespace d1 {

constexpr int kCols = 60, kRing = 64;   // columns a tile updates and holds
constexpr int kRow = 4 * kRing;         // doubles of one tile row: h, hu, hv, B

__device__ __forceinline__ long long bits(double a) { return __double_as_longlong(a); }
// bit patterns in the order of the values
__device__ __forceinline__ long long key(double a)
{
    const long long b = bits(a);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double imin(double a, double b) { return key(a) <= key(b) ? a : b; }
__device__ __forceinline__ double imax(double a, double b) { return key(a) >= key(b) ? a : b; }
__device__ __forceinline__ double pmax(double a, double b) { return bits(a) >= bits(b) ? a : b; }   // neither negative
__device__ __forceinline__ bool neg(double a) { return bits(a) < 0; }
__device__ __forceinline__ bool zero(double a) { return (bits(a) << 1) == 0; }
__device__ __forceinline__ double flip(double a, bool f) { return __longlong_as_double(bits(a) ^ (f ? (long long)0x8000000000000000ull : 0)); }
// a normal a times 2^-n
__device__ __forceinline__ double down(double a, int n) { return __longlong_as_double(bits(a) - ((long long)n << 52)); }
// the float next to a towards zero; 0 below the float range, infinity above it
__device__ __forceinline__ float tof(double a)
{
    const unsigned hi = (unsigned)((unsigned long long)bits(a) >> 32), lo = (unsigned)bits(a);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned r = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : ((unsigned)e << 23) | m);
    return __uint_as_float(r | (hi & 0x80000000u));
}

// a cell with what its edges take from it
struct CellD {
    Cell<double> z;
    double e, su, um, up, pn, pt;   // h + B, sqrt(h) u, u - c, u + c, hn u, hn v
};

__device__ __forceinline__ void load_cell(CellD &c, double h, double hn, double ht, double B, long long tol)
{
    c.z.q0 = h; c.z.hn = hn; c.z.ht = ht; c.z.B = B;
    c.z.h = h;
    c.z.wet = bits(h) >= tol;
}
__device__ __forceinline__ bool still(const CellD &c) { return zero(c.z.hn) && zero(c.z.ht); }
// derived quantities (as derive()); dry cells get zeros
__device__ __forceinline__ void derive(CellD &c, double g)
{
    Cell<double> &z = c.z;
    z.u = 0.0; z.v = 0.0; z.c = 0.0; z.sq = 0.0;
    if (z.wet) {
        z.u = z.hn / z.h;
        z.v = z.ht / z.h;
        z.c = sqrt(g * z.h);
        z.sq = sqrt(z.h);
    }
    c.su = z.sq * z.u;
    c.um = z.u - z.c;
    c.up = z.u + z.c;
    c.pn = z.hn * z.u;
    c.pt = z.hn * z.v;
}

// riemann() for two wet cells, subsonic, with no bounded bed step; false where that
// is not so or not certain (r is then not to be used)
__device__ __forceinline__ bool riemann_ocean(double hg, const CellD &L, const CellD &R, Wave<double> &r)
{
    const double uh = (L.su + R.su) / (L.z.sq + R.z.sq);
    const double ghb = hg * (L.z.h + R.z.h);   // g (h_L + h_R) / 2: halving is exact
    const double ch = sqrt(ghb);
    const double s1 = imin(L.um, uh - ch), s3 = imax(R.up, uh + ch);
    const double deta = R.e - L.e, d2 = R.z.hn - L.z.hn;
    const double d3 = (R.pn - L.pn) + ghb * deta;
    const double d4 = R.pt - L.pt;
    const double den = s3 - s1;
    const double w1m = (s3 * deta - d2) / den;
    const double w1n = (s3 * d2 - d3) / den;
    const double b1 = s1 * w1m, g1 = s1 * w1n;
    const double b3 = s3 * (deta - w1m), g3 = s3 * (d2 - w1n);
    const double t1 = b1 * L.z.v, t3 = b3 * R.z.v;
    r.Z[0][0] = b1; r.Z[0][1] = g1; r.Z[0][2] = t1;
    r.Z[1][0] = 0.0; r.Z[1][1] = 0.0; r.Z[1][2] = (d4 - t1) - t3;
    r.Z[2][0] = b3; r.Z[2][1] = g3; r.Z[2][2] = t3;
    r.s[0] = s1; r.s[1] = uh; r.s[2] = s3;
    r.wall = 0;
    // the states either side of the bed step keep h >= 0: M - s3 delta and M - s1
    // delta positive by more than FP32 can have wrong in them
    const float f1 = tof(s1), f3 = tof(s3), a = f3 * tof(R.z.h), b = f1 * tof(L.z.h), c = tof(d2);
    const float dl = tof(L.z.B - R.z.B);
    const float M = (a - b) - c, p3 = f3 * dl, p1 = f1 * dl;
    const float lim = 1e-4f * ((a - b) + fabsf(c) + fabsf(p3) + fabsf(p1));
    return L.z.wet && R.z.wet && neg(s1) && !neg(s3) && f1 < 0.0f && f3 > 0.0f && M - p3 > lim && M - p1 > lim;
}

// half the MC limiter of dIi / dii, max(0, min((1 + theta)/4, 1, theta)): halving
// and quartering are exact, so c_p carries the 1/2 of the correction flux
__device__ __forceinline__ double mc_half(double dIi, double dii)
{
    if (zero(dii)) return 0.0;
    const double th = dIi / dii;
    if (bits(th) <= 0) return 0.0;
    const double q = down(1.0 + th, 2);   // theta > 0: 1 + theta is normal
    double m = bits(q) < bits(th) ? q : th;
    if (bits(m) > 0x3ff0000000000000LL) m = 1.0;
    return m;
}
__device__ __forceinline__ double factor(double s, double r, double ph)   // 1/2 sgn(s)(1 - r |s|) phi
{
    return flip((1.0 - r * fabs(s)) * ph, neg(s));
}
__device__ __forceinline__ double dot3(const double (&a)[3], const double (&b)[3])
{
    return (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2];
}

// limit() of an edge that riemann_ocean solved: wave 0 with its right neighbour's,
// wave 2 with its left neighbour's, t1 the upwind contact wave
__device__ __forceinline__ void limit_ocean(const Wave<double> &r, const double (&I0)[3], double t1, const double (&I2)[3],
                                            double dtdx, double (&am)[3], double (&ap)[3], double (&F)[3])
{
    const double c0 = factor(r.s[0], dtdx, mc_half(dot3(I0, r.Z[0]), dot3(r.Z[0], r.Z[0])));
    const double c2 = factor(r.s[2], dtdx, mc_half(dot3(I2, r.Z[2]), dot3(r.Z[2], r.Z[2])));
    const double z1 = r.Z[1][2];
    double c1 = 0.0, l1 = 0.0, r1 = 0.0;   // the contact wave's factor and its shares
    if (!zero(z1)) {
        if (zero(r.s[1])) { l1 = 0.5 * z1; r1 = l1; }
        else {
            if (neg(r.s[1])) l1 = z1; else r1 = z1;
            c1 = factor(r.s[1], dtdx, mc_half(t1 * z1, z1 * z1));
        }
    }
    am[0] = r.Z[0][0]; ap[0] = r.Z[2][0]; F[0] = c0 * r.Z[0][0] + c2 * r.Z[2][0];
    am[1] = r.Z[0][1]; ap[1] = r.Z[2][1]; F[1] = c0 * r.Z[0][1] + c2 * r.Z[2][1];
    am[2] = r.Z[0][2] + l1; ap[2] = r1 + r.Z[2][2];
    F[2] = (c0 * r.Z[0][2] + c1 * z1) + c2 * r.Z[2][2];
}

// limit() of any edge.  Waves go to a side by selection (half each at speed 0); the
// contact wave has only a transverse component here too.
__device__ __forceinline__ void share(double z, double s, double &l, double &r)
{
    l = neg(s) ? z : 0.0;
    r = neg(s) ? 0.0 : z;
    if (zero(s)) { l = 0.5 * z; r = l; }
}
__device__ __forceinline__ void limit_any(const Wave<double> &r, const double (&I0)[3], double t1, const double (&I2)[3],
                                          double dtdx, double (&am)[3], double (&ap)[3], double (&F)[3])
{
    double l0[3], r0[3], l2[3], r2[3], l1, r1;
#pragma unroll
    for (int m = 0; m < 3; m++) { share(r.Z[0][m], r.s[0], l0[m], r0[m]); share(r.Z[2][m], r.s[2], l2[m], r2[m]); }
    const double z1 = r.Z[1][2];
    share(z1, r.s[1], l1, r1);
    double c0 = 0.0, c1 = 0.0, c2 = 0.0;
    if (r.wall == 0) {
        if (!zero(r.s[0])) c0 = factor(r.s[0], dtdx, mc_half(dot3(I0, r.Z[0]), dot3(r.Z[0], r.Z[0])));
        if (!zero(r.s[1])) c1 = factor(r.s[1], dtdx, mc_half(t1 * z1, z1 * z1));
        if (!zero(r.s[2])) c2 = factor(r.s[2], dtdx, mc_half(dot3(I2, r.Z[2]), dot3(r.Z[2], r.Z[2])));
    }
#pragma unroll
    for (int m = 0; m < 2; m++) {
        am[m] = l0[m] + l2[m];
        ap[m] = r0[m] + r2[m];
        F[m] = c0 * r.Z[0][m] + c2 * r.Z[2][m];
    }
    am[2] = (l0[2] + l1) + l2[2];
    ap[2] = (r0[2] + r1) + r2[2];
    F[2] = (c0 * r.Z[0][2] + c1 * z1) + c2 * r.Z[2][2];
    if (r.wall == 2) { ap[0] = 0.0; ap[1] = 0.0; ap[2] = 0.0; }
    if (r.wall == 1) { am[0] = 0.0; am[1] = 0.0; am[2] = 0.0; }
}

// the neighbour's value among GW lanes of a row; its first or last lane: its own
template <int GW> __device__ __forceinline__ double shfl_up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1, GW); }
template <int GW> __device__ __forceinline__ double shfl_down1(double v) { return __shfl_down_sync(0xffffffffu, v, 1, GW); }

// postprocess(); false where h is not a finite number (or absurd), which is left as it is
__device__ __forceinline__ bool post(double &h, double &qn, double &qt, long long tol)
{
    const long long mag = bits(h) & 0x7fffffffffffffffLL;
    if (mag >= 0x46293e5939a08ceaLL && !(neg(h) && mag <= 0x7ff0000000000000LL)) return false;   // 1e30 and above, NaN
    if (neg(h)) h = 0.0;
    if (bits(h) < tol) { qn = 0.0; qt = 0.0; }
    return true;
}

}  // namespace d1

template <int NW, bool GEO> __device__ __forceinline__ void tile64_item(const StepArgs &a, int item)
{
    using namespace d1;
    constexpr unsigned ALL = 0xffffffffu;
    constexpr int NT = NW * 32;
    extern __shared__ __align__(128) double tile64[];   // [row][field][column]
    __shared__ double red[2][NW];

    StepItem it;
    if (a.items) it = a.items[item];
    else {   // one patch cut into tiles of a.tile_rows rows
        const int nsx = a.tile_nsx, sy = item / nsx, sx = item - sy * nsx;
        const PatchDesc &P0 = a.descs[0];
        it.patch = 0;
        it.x0 = sx * kCols; it.y0 = sy * a.tile_rows;
        it.w = min(kCols, P0.nx - it.x0); it.h = min(a.tile_rows, P0.ny - it.y0);
    }
    if (it.w > kCols || it.w < 1 || it.h < 1 || it.h > a.tile_rows) return;   // not an item of this launch
    const PatchDesc P = a.descs[it.patch];
    if (a.gate != nullptr && a.gate[P.scen] == 0) return;   // not retaken (uniform over the CTA)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int cur = a.cur, pitch = P.pitch;
    const long long fs = P.fs;
    double *base = reinterpret_cast<double *>(a.arena) + P.off;
    const double g = a.g, hg = 0.5 * a.g, drytol = a.drytol;
    const long long tol = bits(drytol);
    const double dt = a.dt1[P.scen] / a.R;
    const double dtdx0 = dt / a.dx, dtdy0 = dt / a.dy;
    const int x0 = it.x0, y0 = it.y0, w = it.w, h = it.h;
    const int nrows = h + 4, ncols = w + 4;
    // tile row k, column c <-> patch row y0 - 2 + k, column x0 - 2 + c
    const double *src = base + (long long)(cur * 3) * fs + (long long)y0 * pitch + x0;
    const long long fB = (long long)(6 - cur * 3) * fs;
    for (int e = t; e < nrows * 256; e += NT) {
        const int k = e >> 8, f = (e >> 6) & 3, c = e & 63;
        // columns past a narrow tile repeat its last: no waves between them
        cp_async_elem(tile64 + k * kRow + f * kRing + c, src + (f < 3 ? f * fs : fB) + (long long)k * pitch + min(c, ncols - 1), 8);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();

    const double *kapP = GEO ? a.kap + (P.j0 + 2) : nullptr;   // capacity of patch row j at kapP[j]
    const double *cedP = GEO ? a.ced + (P.j0 + 2) : nullptr;   // relative length of the y-edge below it at cedP[j]
    double smx = 0.0, smy = 0.0, deep_x = 0.0, deep_y = 0.0;   // largest speeds; deepest resting cells

    // ---- x sweep, two adjacent columns per lane and their left edges: a row per warp, or
    // two where a row fits half of one.  (Patches of 16 columns, 3600 of them: 2958 us a
    // step with a row per warp whatever its width, 1970 us; 28 columns 1627 and 1046.  The
    // width fixed at compile time: with it in a register wide rows lose 0.5%.)
    auto sweep_x = [&](auto width) {
        constexpr int GW = decltype(width)::value, RW = 32 / GW;   // lanes of a row, rows of a warp
        const int c0 = 2 * (lane & (GW - 1));
        const bool lim[2] = {c0 >= 2 && c0 <= w + 2, c0 + 1 >= 2 && c0 + 1 <= w + 2};   // edges of updated columns
        for (int kw = warp * RW; kw < nrows; kw += NW * RW) {
            const int k = RW == 1 ? kw : min(kw + lane / GW, nrows - 1);
            const bool live = RW == 1 || kw + lane / GW < nrows;   // (past the last row: its values, unused)
            const bool out[2] = {live && c0 >= 2 && c0 < w + 2, live && c0 + 1 >= 2 && c0 + 1 < w + 2};   // updated columns
            double *row = tile64 + k * kRow + c0;
            CellD z[2], L;
#pragma unroll
            for (int q = 0; q < 2; q++) {
                load_cell(z[q], row[q], row[kRing + q], row[2 * kRing + q], row[3 * kRing + q], tol);
                z[q].e = z[q].z.h + z[q].z.B;
            }
            const int j = y0 - 2 + k;
            const bool rowint = live && j >= 0 && j < P.ny;
            const double kr = GEO ? kapP[j] : 1.0;
            const double dtdx = GEO ? dt / (kr * a.dx) : dtdx0;
            const bool wet = z[0].z.wet && z[1].z.wet;
            L.e = shfl_up1<GW>(z[1].e);
            L.z.h = shfl_up1<GW>(z[1].z.h);
            const bool flat = wet && bits(L.e) == bits(z[0].e) && bits(z[0].e) == bits(z[1].e) && still(z[0]) && still(z[1]);
            if (__all_sync(ALL, flat)) {
                if (rowint) {
                    double d = 0.0;
                    if (lim[0]) d = pmax(L.z.h, z[0].z.h);
                    if (lim[1]) d = pmax(d, pmax(z[0].z.h, z[1].z.h));
                    if (GEO) { if (d > 0.0) smx = pmax(smx, sqrt(g * d) / kr); }
                    else deep_x = pmax(deep_x, d);
                }
                continue;
            }
            if (!__any_sync(ALL, z[0].z.wet || z[1].z.wet)) {   // no edge has waves
#pragma unroll
                for (int q = 0; q < 2; q++)
                    if (out[q]) {
                        double q0 = z[q].z.h, q1 = z[q].z.hn, q2 = z[q].z.ht;
                        postprocess<double, false>(q0, q1, q2, z[q].z.B, drytol);
                        row[q] = q0; row[kRing + q] = q1; row[2 * kRing + q] = q2;
                    }
                continue;
            }
            derive(z[0], g);
            derive(z[1], g);
            L.z.q0 = L.z.h; L.z.wet = bits(L.z.h) >= tol;
            L.z.hn = shfl_up1<GW>(z[1].z.hn); L.z.ht = shfl_up1<GW>(z[1].z.ht); L.z.B = shfl_up1<GW>(z[1].z.B);
            L.z.u = shfl_up1<GW>(z[1].z.u); L.z.v = shfl_up1<GW>(z[1].z.v); L.z.c = shfl_up1<GW>(z[1].z.c); L.z.sq = shfl_up1<GW>(z[1].z.sq);
            L.su = shfl_up1<GW>(z[1].su); L.um = shfl_up1<GW>(z[1].um); L.pn = shfl_up1<GW>(z[1].pn); L.pt = shfl_up1<GW>(z[1].pt);
            Wave<double> e[2];
            double am[2][3], ap[2][3], F[2][3];
            // (a row with a dry cell goes to the general solver at once)
            const bool tried = __all_sync(ALL, wet);
            const bool oc = tried && (riemann_ocean(hg, L, z[0], e[0]) & riemann_ocean(hg, z[0], z[1], e[1]));
            if (__all_sync(ALL, oc)) {
                double rt[3], lt[3];
#pragma unroll
                for (int m = 0; m < 3; m++) { rt[m] = shfl_down1<GW>(e[0].Z[0][m]); lt[m] = shfl_up1<GW>(e[1].Z[2][m]); }
                const double tl = shfl_up1<GW>(e[1].Z[1][2]), tr = shfl_down1<GW>(e[0].Z[1][2]);
                limit_ocean(e[0], e[1].Z[0], neg(e[0].s[1]) ? e[1].Z[1][2] : tl, lt, dtdx, am[0], ap[0], F[0]);
                limit_ocean(e[1], rt, neg(e[1].s[1]) ? tr : e[0].Z[1][2], e[0].Z[2], dtdx, am[1], ap[1], F[1]);
            } else {
                if (!oc) {
                    riemann<double, false>(g, L.z, z[0].z, e[0]);
                    riemann<double, false>(g, z[0].z, z[1].z, e[1]);
                }
                double I00[3], I02[3], I10[3], I12[3];   // upwind waves of the two edges
                auto pick = [&](int p, int m, double &x0, double &x1) {
                    const double l = shfl_up1<GW>(e[1].Z[p][m]), r = shfl_down1<GW>(e[0].Z[p][m]);
                    x0 = neg(e[0].s[p]) ? e[1].Z[p][m] : l;
                    x1 = neg(e[1].s[p]) ? r : e[0].Z[p][m];
                };
                double t0, t1;
#pragma unroll
                for (int m = 0; m < 3; m++) { pick(0, m, I00[m], I10[m]); pick(2, m, I02[m], I12[m]); }
                pick(1, 2, t0, t1);
                limit_any(e[0], I00, t0, I02, dtdx, am[0], ap[0], F[0]);
                limit_any(e[1], I10, t1, I12, dtdx, am[1], ap[1], F[1]);
            }
            if (rowint) {
#pragma unroll
                for (int q = 0; q < 2; q++)
                    if (lim[q]) {
                        const double se = imax(flip(e[q].s[0], true), e[q].s[2]);
                        smx = imax(smx, GEO ? se / kr : se);
                    }
            }
            double amr[3], Fr[3];   // of the right lane's first edge
#pragma unroll
            for (int m = 0; m < 3; m++) { amr[m] = shfl_down1<GW>(am[0][m]); Fr[m] = shfl_down1<GW>(F[0][m]); }
#pragma unroll
            for (int q = 0; q < 2; q++) {
                double qs[3] = {z[q].z.q0, z[q].z.hn, z[q].z.ht};
#pragma unroll
                for (int m = 0; m < 3; m++) {
                    const double u = (ap[q][m] + (q ? amr[m] : am[1][m])) + ((q ? Fr[m] : F[1][m]) - F[q][m]);
                    qs[m] = qs[m] - dtdx * u;
                }
                post(qs[0], qs[1], qs[2], tol);
                if (out[q]) { row[q] = qs[0]; row[kRing + q] = qs[1]; row[2 * kRing + q] = qs[2]; }
            }
        }
    };
    if (w <= 28) sweep_x(std::integral_constant<int, 16>());
    else sweep_x(std::integral_constant<int, 32>());
    __syncthreads();

    // ---- y sweep: a warp takes 32 columns and a segment of rows, one column per
    // lane, and marches up.  Ring row k = 0 .. hs + 3 of the segment is tile row s0 +
    // k; y-edge k lies between ring rows k - 1 and k.  Iteration k solves edge k,
    // limits edge k - 1 and updates row k - 2.
    constexpr int NSEG = NW >= 2 ? NW / 2 : 1;
    const int sl = (h + NSEG - 1) / NSEG;
    double *dst = base + (long long)((1 - cur) * 3) * fs;
    for (int un = warp; un < 2 * NSEG; un += NW) {
        const int half = un & 1, s0 = (un >> 1) * sl, hs = min(sl, h - s0);
        if (32 * half >= w || hs <= 0) continue;   // uniform over the warp
        const int col = 32 * half + lane;
        const bool valid = col < w;
        const double *cs = tile64 + s0 * kRow + min(col, w - 1) + 2;   // lanes past the tile repeat its last column
        const long long o0 = (long long)(y0 + s0) * pitch + (x0 + col + 2);   // ring row k at o0 + k pitch
        const int jr = y0 + s0 - 2;   // patch row of ring row 0
        CellD p, c;
        Wave<double> wo, wm, wn;   // edges k - 2, k - 1, k
        double apl[3] = {0.0, 0.0, 0.0}, Fl[3] = {0.0, 0.0, 0.0};   // A+dQ and F~ of edge k - 2
        bool pder = false;         // p's derived quantities are set
        bool okm = false, rm = true, rp = true;   // edge k - 1 solved by riemann_ocean; edges k - 1, k - 2 without waves
        auto clear = [](Wave<double> &x) {
#pragma unroll
            for (int q = 0; q < 3; q++) {
                x.s[q] = 0.0;
#pragma unroll
                for (int m = 0; m < 3; m++) x.Z[q][m] = 0.0;
            }
            x.wall = 0;
        };
        clear(wo); clear(wm); clear(wn);
        for (int k = 0; k <= hs + 3; k++) {
            const double *r = cs + k * kRow;
            load_cell(c, r[0], r[2 * kRing], r[kRing], r[3 * kRing], tol);   // y roles: hn = hv, ht = hu
            c.e = c.z.h + c.z.B;
            bool rn = true, okn = false, cder = false;
            if (k >= 1) {
                const bool counts = valid && k >= 2 && k <= hs + 2;   // a y-edge of a row of the segment
                const double cr = GEO ? cedP[jr + k] / (0.5 * (kapP[jr + k - 1] + kapP[jr + k])) : 1.0;
                const bool flat = c.z.wet && p.z.wet && bits(c.e) == bits(p.e) && still(c) && still(p);
                if (__all_sync(ALL, flat)) {
                    const double d = pmax(p.z.h, c.z.h);
                    if (GEO) { if (counts) smy = pmax(smy, sqrt(g * d) * cr); }
                    else if (counts) deep_y = pmax(deep_y, d);
                    clear(wn);
                } else if (!__any_sync(ALL, c.z.wet || p.z.wet)) {
                    clear(wn);
                } else {
                    rn = false;
                    if (!pder) derive(p, g);
                    derive(c, g);
                    cder = true;
                    // (with a dry cell among the warp's, the general solver at once)
                    const bool tried = __all_sync(ALL, c.z.wet && p.z.wet);
                    const bool oc = tried && riemann_ocean(hg, p, c, wn);
                    okn = __all_sync(ALL, oc);
                    if (!oc) riemann<double, false>(g, p.z, c.z, wn);
                    if (counts) {
                        const double se = imax(flip(wn.s[0], true), wn.s[2]);
                        smy = imax(smy, GEO ? se * cr : se);
                    }
                }
            }
            if (k >= 3) {
                double am[3] = {0.0, 0.0, 0.0}, ap[3] = {0.0, 0.0, 0.0}, F[3] = {0.0, 0.0, 0.0};
                if (!rm) {
                    double dtdy = dtdy0;
                    if (GEO) {
                        const double kbar = 0.5 * (kapP[jr + k - 2] + kapP[jr + k - 1]);
                        dtdy = (dt * cedP[jr + k - 1]) / (kbar * a.dy);
                    }
                    if (okm) {
                        limit_ocean(wm, wn.Z[0], neg(wm.s[1]) ? wn.Z[1][2] : wo.Z[1][2], wo.Z[2], dtdy, am, ap, F);
                    } else {
                        double I0[3], I2[3];
#pragma unroll
                        for (int m = 0; m < 3; m++) {
                            I0[m] = neg(wm.s[0]) ? wn.Z[0][m] : wo.Z[0][m];
                            I2[m] = neg(wm.s[2]) ? wn.Z[2][m] : wo.Z[2][m];
                        }
                        limit_any(wm, I0, neg(wm.s[1]) ? wn.Z[1][2] : wo.Z[1][2], I2, dtdy, am, ap, F);
                    }
                }
                if (k >= 4) {
                    const double *q = cs + (k - 2) * kRow;
                    double qn[3] = {q[0], q[2 * kRing], q[kRing]};   // (mass, normal = hv, transverse = hu)
                    if (!(rm && rp)) {
                        if (GEO) {
                            const int rc = jr + k - 2;
                            const double clo = cedP[rc], chi = cedP[rc + 1];
                            const double dtk = dt / (kapP[rc] * a.dy);
                            const double hv = qn[1];
#pragma unroll
                            for (int m = 0; m < 3; m++) {
                                double u = (clo * apl[m] + chi * am[m]) + (chi * F[m] - clo * Fl[m]);
                                if (m == 0) u = u + (chi - clo) * hv;
                                qn[m] = qn[m] - dtk * u;
                            }
                        } else {
#pragma unroll
                            for (int m = 0; m < 3; m++) {
                                const double u = (apl[m] + am[m]) + (F[m] - Fl[m]);
                                qn[m] = qn[m] - dtdy0 * u;
                            }
                        }
                    }
                    // (a depth that is not a finite number reaches the host as an infinite speed)
                    if (!post(qn[0], qn[1], qn[2], tol) && valid) smy = INFINITY;
                    if (a.manning > 0.0)   // y frame: qn[2] = hu, qn[1] = hv
                        friction<double, false>(qn[0], qn[2], qn[1], q[3 * kRing], drytol, a.manning, dt);
                    if (valid) {
                        const long long o = o0 + (long long)(k - 2) * pitch;
                        dst[o] = qn[0];
                        dst[fs + o] = qn[2];
                        dst[2 * fs + o] = qn[1];
                    }
                }
#pragma unroll
                for (int m = 0; m < 3; m++) { apl[m] = ap[m]; Fl[m] = F[m]; }
                rp = rm;
            }
            wo = wm; wm = wn;
            okm = okn; rm = rn;
            p = c; pder = cder;
        }
    }
    if (!GEO) {
        if (deep_x > 0.0) smx = pmax(smx, sqrt(g * deep_x));
        if (deep_y > 0.0) smy = pmax(smy, sqrt(g * deep_y));
    }

    // ---- the CTA's largest speeds
    if (!(smx > 0.0)) smx = 0.0;
    if (!(smy > 0.0)) smy = 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        smx = pmax(smx, __shfl_xor_sync(ALL, smx, o));
        smy = pmax(smy, __shfl_xor_sync(ALL, smy, o));
    }
    if (lane == 0) { red[0][warp] = smx; red[1][warp] = smy; }
    __syncthreads();
    if (t == 0) {
        double mx = 0.0, my = 0.0;
#pragma unroll
        for (int q = 0; q < NW; q++) { mx = pmax(mx, red[0][q]); my = pmax(my, red[1][q]); }
        atomic_max_speed(a.smax + 2 * P.scen + 0, mx);
        atomic_max_speed(a.smax + 2 * P.scen + 1, my);
    }
}

template <int NW, bool GEO> __global__ void __launch_bounds__(NW * 32, NW >= 8 ? 1 : 12 / NW) step_tile_f64(StepArgs a)
{
    if (!launch_live(a)) return;
    tile64_item<NW, GEO>(a, blockIdx.x);
    step_tail<double, false>(a);
}

}  // namespace tsu
