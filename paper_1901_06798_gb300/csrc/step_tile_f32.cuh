// step_tile_f32.cuh -- the FP32 surface-perturbation split step (Sec. 2.2,
// x sweep then y sweep) of every patch of a level in one launch.
//
// A CTA takes a tile of up to 60 columns x h rows of one patch.  It copies the
// tile with its two ghost cells per side (64 columns x h + 4 rows of eta', hu,
// hv, B) into shared memory, sweeps it in x in place, and then in y from there
// to the output buffer:
//   * x: a warp takes a row, two adjacent columns per lane (lanes x, y of every
//     float2); neighbours' values move by warp shuffles.  Rows are independent,
//     so the row is the unit of work and Q* of the ghost rows comes with it;
//   * y: the rows of a tile are cut into a segment per warp; a lane takes two
//     adjacent columns and marches up the segment, a row per iteration, starting
//     two rows below its first.  The march's state (the row below, the edge below)
//     alternates between two register sets.
// Q* never leaves the SM: the step reads the state and B once and writes the
// state once.  Registers are those of one sweep at a time (the y sweep's 128),
// so four CTAs of four warps fit on an SM with tiles of up to 48 rows (12 warps of
// 168 registers: 143.1 against 141.3 us on 3000^2 developed cells).
//
// What bounds it is the issue of instructions: 61% of the issue slots on a developed
// sea (334 warp instructions for 32 cells), DRAM under a third of its rate.  Two
// kernels with Q* in DRAM between them, one-warp strips in x and row pairs in y, took
// 309 us for a step of the 4096^2 shelf some hundred steps after its uplift and 294 us
// for 2050 x 1537 developed cells in the caller's memory; with this kernel the steps
// take 222 and 94 us (the shelf's first 20 steps, most of the sea at rest: 174 us each).
// The y march over pairs of rows instead of pairs of columns: 237 against 149 us for
// 3000^2 cells.
//
// A row of a warp takes the cheapest of four forms, by warp votes; all give the
// bits of the general one:
//   * still water: every cell wet, momenta exactly zero and the surface exactly
//     level across the edges.  Every wave is then an exact zero and Q* = Q; only
//     the wave speeds of the CFL number are left to compute;
//   * dry: no cell wet.  No edge has waves; the cells are post-processed;
//   * ocean: every cell wet and every edge subsonic with no bounded bed step:
//     limit2_ocean;
//   * any other: the general solver and limiter.  In y a segment that meets such
//     an edge is marched again in general form, so that the ocean's march holds no
//     register for it.
// GEO: latitude-longitude grid in capacity form (Sec. 2.1 spherical
// coordinates): the x sweep of row j runs with dt / (kap_j dx) and reports
// speeds / kap_j; what a y-edge gives its cells is weighted by its relative
// length ced_e (its Courant number uses dt ced_e / (kbar_e dy), kbar_e the mean
// capacity of its two cells); the cell update divides by kap_j and adds
// (ced_{j+1} - ced_j) hv_j to the mass.
// BULK: one thread copies each field's row segment with a bulk copy
// (cp.async.bulk); all complete on one mbarrier, which every thread polls with a
// bounded budget.
#pragma once
#include <type_traits>
#include "step_f32x2.cuh"
#include "tile_rules.h"

namespace tsu {

constexpr int kTileCols = 60;        // columns a tile updates
constexpr int kTileRing = 64;        // columns it holds
constexpr int kTileRow = 4 * kTileRing;   // floats of one tile row: four fields

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}

template <int NW, bool GEO, bool BULK> __device__ __forceinline__ void tile_item(const StepArgs &a, int item)
{
    using namespace x2;
    constexpr unsigned ALL = 0xffffffffu;
    constexpr int NT = NW * 32;
    extern __shared__ __align__(128) float tile[];   // [row][field][column]
    __shared__ float red[2][NW];
    __shared__ __align__(8) unsigned long long bar[1];
    __shared__ int gave_up;
    __shared__ unsigned dry_rows[(kTileRowsMax + 4 + 31) / 32];   // bit k: tile row k has a dry cell

    StepItem it;
    if (a.items) it = a.items[item];
    else {   // one patch cut into tiles of a.tile_rows rows
        const int nsx = a.tile_nsx, sy = item / nsx, sx = item - sy * nsx;
        const PatchDesc &P0 = a.descs[0];
        it.patch = 0;
        it.x0 = sx * kTileCols; it.y0 = sy * a.tile_rows;
        it.w = min(kTileCols, P0.nx - it.x0); it.h = min(a.tile_rows, P0.ny - it.y0);
    }
    if (it.w > kTileCols || it.w < 1 || it.h < 1 || it.h > a.tile_rows) return;   // not an item of this launch
    const PatchDesc P = a.descs[it.patch];
    if (a.gate != nullptr && a.gate[P.scen] == 0) return;   // not retaken (uniform over the CTA)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int cur = a.cur, pitch = P.pitch;
    const long long fs = P.fs;
    float *base = reinterpret_cast<float *>(a.arena) + P.off;
    const float g = a.gf, drytol = a.drytolf, sqrtg = a.sqrtgf;
    const float dt1 = a.dt1f[P.scen];
    const int x0 = it.x0, y0 = it.y0, w = it.w, h = it.h;
    const int nrows = h + 4, ncols = w + 4;
    // tile row k, column c <-> patch row y0 - 2 + k, column x0 - 2 + c
    const float *src = base + (long long)(cur * 3) * fs + (long long)y0 * pitch + x0;
    const long long fB = (long long)(6 - cur * 3) * fs;

    if (t < (kTileRowsMax + 4 + 31) / 32) dry_rows[t] = 0u;   // visible after the barrier below
    // ---- the tile into shared memory
    const bool v16 = ((reinterpret_cast<uintptr_t>(src) & 15) == 0) && ((pitch & 3) == 0) && ((fs & 3) == 0);
    if (BULK) {
        if (!v16) {
            if (t == 0 && a.err) atomicOr(a.err, TSU_DEV_ERR_LAYOUT);   // uniform over the CTA
            return;
        }
        const unsigned nb = (unsigned)((ncols * 4 + 15) & ~15);   // stays inside the row: the pitch is a multiple of 16 bytes
        if (t == 0) {
            mbar_init(bar, 1);
            gave_up = 0;
            mbar_init_fence();
            mbar_expect_tx(bar, (unsigned)nrows * 4u * nb);
            for (int k = 0; k < nrows; k++)
                for (int f = 0; f < 4; f++)
                    bulk_g2s(tile + k * kTileRow + f * kTileRing, src + (f < 3 ? f * fs : fB) + (long long)k * pitch, nb, bar);
        }
        __syncthreads();
        if (!mbar_wait(bar, 0u, a.wait_polls)) *(volatile int *)&gave_up = 1;
        __syncthreads();
        if (gave_up) {
            // the copies in flight land before the CTA exits; then the launch
            // reports the timeout
            if (t == 0) {
                mbar_wait(bar, 0u, kDrainPolls);
                if (a.err) atomicOr(a.err, TSU_DEV_ERR_TIMEOUT);
            }
            return;
        }
    } else {
        if (v16) {
            const int nch = (ncols + 3) >> 2;   // 16-byte chunks of a row: the last one stays inside the pitch
            for (int e = t; e < nrows * 64; e += NT) {
                const int k = e >> 6, f = (e >> 4) & 3, c = e & 15;
                if (c < nch)
                    cp_async16(tile + k * kTileRow + f * kTileRing + 4 * c,
                               src + (f < 3 ? f * fs : fB) + (long long)k * pitch + 4 * c);
            }
        } else {
            for (int e = t; e < nrows * 256; e += NT) {
                const int k = e >> 8, f = (e >> 6) & 3, c = e & 63;
                if (c < ncols)
                    cp_async_elem(tile + k * kTileRow + f * kTileRing + c,
                                  src + (f < 3 ? f * fs : fB) + (long long)k * pitch + c, 4);
            }
        }
        cp_async_commit();
    }
    if (!BULK && a.gmap != nullptr && P.bcmask == 0) {
        // Ghost cells from the cells that hold them (16 level-3 steps between regrids
        // used to copy them to the patches' rings first: 94 us a step of 7000 patches,
        // bound by 8 bytes of every 32-byte sector).  The first ones of a thread are
        // on their way while the rows land.  Cells without such a source
        // (interpolated) are in the ring already.
        // (a strip or segment one cell short of the patch's edge has one ghost column or row)
        const int nb = max(0, 2 - y0), nt = max(0, y0 + h + 2 - P.ny), nl = max(0, 2 - x0), nr = max(0, x0 + w + 2 - P.nx);
        const int rows2 = nb + nt, cols2 = nl + nr, nrow = rows2 * ncols, total = nrow + (nrows - rows2) * cols2;
        const GhostSrc *gm = a.gmap + a.goff[it.patch];
        const float *ar = reinterpret_cast<const float *>(a.arena);
        // ghost cell e of the tile: its place in the tile and its source (null: none)
        auto find = [&](int e, float *&to, long long &sf) -> const float * {
            int k, c;
            if (e < nrow) {
                const int r = e / ncols;
                c = e - r * ncols;
                k = r < nb ? r : nrows - nt + (r - nb);
            } else {
                const int r = (e - nrow) / cols2, q = (e - nrow) - r * cols2;
                k = nb + r;
                c = q < nl ? q : ncols - nr + (q - nl);
            }
            const int i = x0 - 2 + c, j = y0 - 2 + k, Wr = P.nx + 4;
            const int gi = j < 0 ? (j + 2) * Wr + i + 2 : (j >= P.ny ? (2 + j - P.ny) * Wr + i + 2 : 4 * Wr + 4 * j + (i < 0 ? i + 2 : 2 + i - P.nx));
            const GhostSrc s = gm[gi];
            to = tile + k * kTileRow + c;
            sf = s.sfs;
            if (s.src == kGhostNone && a.err) atomicOr(a.err, 1);
            return s.src >= 0 ? ar + s.src + (long long)(cur * 3) * s.sfs : nullptr;
        };
        constexpr int HOLD = 4;
        float *to[HOLD];
        float v[HOLD][3];
#pragma unroll
        for (int q = 0; q < HOLD; q++) {
            const int e = t + q * NT;
            to[q] = nullptr;
            if (e < total) {
                float *p;
                long long sf;
                const float *s = find(e, p, sf);
                if (s != nullptr) {
                    to[q] = p;
                    v[q][0] = s[0]; v[q][1] = s[sf]; v[q][2] = s[2 * sf];
                }
            }
        }
        cp_async_wait<0>();
        __syncthreads();
#pragma unroll
        for (int q = 0; q < HOLD; q++)
            if (to[q] != nullptr) { to[q][0] = v[q][0]; to[q][kTileRing] = v[q][1]; to[q][2 * kTileRing] = v[q][2]; }
        for (int e = t + HOLD * NT; e < total; e += NT) {
            float *p;
            long long sf;
            const float *s = find(e, p, sf);
            if (s != nullptr) { p[0] = s[0]; p[kTileRing] = s[sf]; p[2 * kTileRing] = s[2 * sf]; }
        }
    } else {
        if (!BULK) cp_async_wait<0>();
    }
    __syncthreads();
    if (ncols < kTileRing) {   // columns past a narrow tile repeat its last: no waves between them
        const int nf = kTileRing - ncols;
        for (int e = t; e < nrows * 4 * nf; e += NT) {
            const int r = e / nf, c = ncols + (e - r * nf);
            tile[r * kTileRing + c] = tile[r * kTileRing + ncols - 1];
        }
        __syncthreads();
    }

    // ---- x sweep, a row per warp
    const float *rkapP = GEO ? a.rkapf + (P.j0 + 2) : nullptr;   // 1 / capacity of patch row j at rkapP[j]
    const float dtdx = dt1 * a.rdx;
    float smx = 0.0f;
    {
        float2 sp = f2(0.0f);   // largest speeds of this lane's edges c0 and c0 + 1
        const int c0 = 2 * lane;   // this lane's columns: c0, c0 + 1; its edges: the left ones of both
        const bool limx = c0 >= 2 && c0 <= w + 2, limy = c0 + 1 >= 2 && c0 + 1 <= w + 2;   // edges of updated columns
        const bool outx = c0 >= 2 && c0 < w + 2, outy = c0 + 1 >= 2 && c0 + 1 < w + 2;     // updated columns
        auto from_left = [](float v) { return __shfl_up_sync(ALL, v, 1); };      // lane 0: its own value
        auto from_right = [](float v) { return __shfl_down_sync(ALL, v, 1); };   // lane 31: its own value
#pragma unroll 1
        for (int k = warp; k < nrows; k += NW) {
            float *row = tile + k * kTileRow + c0;
            C2 z;
            z.q0 = ld2(row); z.hn = ld2(row + kTileRing); z.ht = ld2(row + 2 * kTileRing); z.B = ld2(row + 3 * kTileRing);
            const int j = y0 - 2 + k;
            const bool rowint = j >= 0 && j < P.ny;
            float rk = 1.0f;
            if (GEO) rk = rkapP[j];
            const float2 dtdxr = f2(GEO ? dtdx * rk : dtdx);
            z.h = sub(z.q0, z.B);
            W2 xw;
            float2 S[3], D[3];
            bool general = true;
            if (__all_sync(ALL, fminf(z.h.x, z.h.y) >= drytol)) {
                C2 L;
                L.q0 = make_float2(from_left(z.q0.y), z.q0.x);
                L.h = make_float2(from_left(z.h.y), z.h.x);
                const bool rest = z.q0.x == L.q0.x && z.q0.y == L.q0.y &&
                                  ((__float_as_uint(z.hn.x) | __float_as_uint(z.hn.y) | __float_as_uint(z.ht.x) |
                                    __float_as_uint(z.ht.y)) << 1) == 0u;
                if (__all_sync(ALL, rest)) {
                    // still water: the speeds are sqrt(g h) of the cells and of the edge's mean depth
                    if (rowint) {
                        const float2 c = mul(f2(sqrtg), sqrt2(z.h)), ch = sqrt2(mul(f2(0.5f * g), add(L.h, z.h)));
                        const float cl = from_left(c.y);
                        sp.x = fmaxf(sp.x, fmaxf(fmaxf(cl, c.x), ch.x) * rk);
                        sp.y = fmaxf(sp.y, fmaxf(fmaxf(c.x, c.y), ch.y) * rk);
                    }
                    continue;
                }
                derive_wet(z, sqrtg);
                L.hn = make_float2(from_left(z.hn.y), z.hn.x);
                L.u = make_float2(from_left(z.u.y), z.u.x); L.v = make_float2(from_left(z.v.y), z.v.x);
                L.sq = make_float2(from_left(z.sq.y), z.sq.x);
                L.c = mul(f2(sqrtg), L.sq);
                L.pn = mul(L.hn, L.u); L.pt = mul(L.hn, L.v);
                const float2 ok = riemann2_ocean(g, L, z, xw);
                if (__all_sync(ALL, fminf(ok.x, ok.y) > 0.0f)) {
                    const float2 d0 = dot3(make_float2(xw.y0m.y, from_right(xw.y0m.x)), make_float2(xw.y0n.y, from_right(xw.y0n.x)),
                                           make_float2(xw.y0t.y, from_right(xw.y0t.x)), xw.y0m, xw.y0n, xw.y0t);
                    const float2 d2 = dot3(make_float2(from_left(xw.z2m.y), xw.z2m.x), make_float2(from_left(xw.z2n.y), xw.z2n.x),
                                           make_float2(from_left(xw.z2t.y), xw.z2t.x), xw.z2m, xw.z2n, xw.z2t);
                    const float tl = from_left(xw.z1t.y), tr = from_right(xw.z1t.x);
                    const float2 t1 = make_float2(xw.s1.x >= 0.0f ? tl : xw.z1t.y, xw.s1.y >= 0.0f ? xw.z1t.x : tr);
                    const float2 mdt = f2(-dtdxr.x);
                    limit2_ocean(xw, d0, t1, third_factor(xw, d2, mdt), mdt, S, D);
                    general = false;
                }
            } else if (lane == 0) {
                atomicOr(&dry_rows[k >> 5], 1u << (k & 31));
            }
            if (general && !__any_sync(ALL, z.h.x >= drytol || z.h.y >= drytol)) {
                post2(z.q0, z.hn, z.ht, z.B, drytol);
                if (outx) { row[0] = z.q0.x; row[kTileRing] = z.hn.x; row[2 * kTileRing] = z.ht.x; }
                if (outy) { row[1] = z.q0.y; row[kTileRing + 1] = z.hn.y; row[2 * kTileRing + 1] = z.ht.y; }
                continue;
            }
            if (general) {
                derive(z, sqrtg, drytol);
                C2 L;
                L.q0 = make_float2(from_left(z.q0.y), z.q0.x);
                L.hn = make_float2(from_left(z.hn.y), z.hn.x);
                L.ht = make_float2(from_left(z.ht.y), z.ht.x);
                L.B = make_float2(from_left(z.B.y), z.B.x);
                L.u = make_float2(from_left(z.u.y), z.u.x); L.v = make_float2(from_left(z.v.y), z.v.x);
                L.c = make_float2(from_left(z.c.y), z.c.x); L.sq = make_float2(from_left(z.sq.y), z.sq.x);
                L.h = make_float2(from_left(z.h.y), z.h.x);
                L.pn = mul(L.hn, L.u); L.pt = mul(L.hn, L.v);
                L.wx = L.h.x >= drytol; L.wy = z.wx;
                riemann2(g, L, z, xw);
                // upwind of edge c0: the left lane's edge c0 - 1 or the own c0 + 1; of
                // edge c0 + 1: the own c0 or the right lane's c0 + 2
                const bool a0 = xw.n0.x <= 0.0f, a1 = xw.s1.x >= 0.0f, a2 = xw.s2.x >= 0.0f;
                const bool b0 = xw.n0.y <= 0.0f, b1 = xw.s1.y >= 0.0f, b2 = xw.s2.y >= 0.0f;
                auto up = [&](float2 zz, bool p, bool q) {
                    const float l = from_left(zz.y), r = from_right(zz.x);
                    return make_float2(p ? l : zz.y, q ? zz.x : r);
                };
                const float2 d0 = dot3(up(xw.y0m, a0, b0), up(xw.y0n, a0, b0), up(xw.y0t, a0, b0), xw.y0m, xw.y0n, xw.y0t);
                const float2 d2 = dot3(up(xw.z2m, a2, b2), up(xw.z2n, a2, b2), up(xw.z2t, a2, b2), xw.z2m, xw.z2n, xw.z2t);
                limit2(xw, d0, up(xw.z1t, a1, b1), d2, dtdxr, S, D);
            }
            if (rowint) {
                sp.x = fmaxf(sp.x, fmaxf(xw.n0.x, xw.s2.x) * rk);
                sp.y = fmaxf(sp.y, fmaxf(xw.n0.y, xw.s2.y) * rk);
            }
            float2 q0 = fnma(dtdxr, add(D[0], make_float2(S[0].y, from_right(S[0].x))), z.q0);
            float2 q1 = fnma(dtdxr, add(D[1], make_float2(S[1].y, from_right(S[1].x))), z.hn);
            float2 q2 = fnma(dtdxr, add(D[2], make_float2(S[2].y, from_right(S[2].x))), z.ht);
            {
                const float2 hq = sub(q0, z.B);
                if (!__all_sync(ALL, min_nan(hq.x, hq.y) >= drytol)) post2(q0, q1, q2, z.B, drytol);
            }
            // (past an odd last column the pair's other lane is a halo column, which nobody reads again)
            if (outx || outy) { st2(row, q0); st2(row + kTileRing, q1); st2(row + 2 * kTileRing, q2); }
        }
        smx = fmaxf(limx ? sp.x : 0.0f, limy ? sp.y : 0.0f);
    }
    __syncthreads();

    // ---- y sweep: a warp marches up its segment of rows, two adjacent columns per
    // lane.  Ring row k = 0 .. hs + 3 of the segment is tile row s0 + k; y-edge k
    // lies between ring rows k - 1 and k.  Iteration k solves edge k, limits edge
    // k - 1 and updates row k - 2 from D of edge k - 2 and S of edge k - 1.
    const int sl = (h + NW - 1) / NW;   // rows of a segment
    const int s0 = warp * sl, hs = min(sl, h - s0);
    const float dtdy = dt1 * a.rdy;
    const float *cedP = GEO ? a.cedf + (P.j0 + 2) : nullptr;    // relative length of the y-edge below patch row j
    const float *cratP = GEO ? a.cratf + (P.j0 + 2) : nullptr;  // the same over the mean capacity of its two cells
    float smy = 0.0f;
    if (hs > 0) {
        const int c0 = 2 * lane;
        const bool outx = c0 >= 2 && c0 < w + 2, outy = c0 + 1 >= 2 && c0 + 1 < w + 2;   // updated columns
        const float *cs = tile + s0 * kTileRow + c0;
        float *dst = base + (long long)((1 - cur) * 3) * fs + (long long)(y0 + s0) * pitch + (x0 + c0);   // ring row k at dst + k pitch
        // pairs of columns stored as one (uniform over the warp)
        const bool v8 = (w & 1) == 0 && ((reinterpret_cast<uintptr_t>(dst) & 7) == 0) && ((pitch & 1) == 0) && ((fs & 1) == 0);
        float2 sp = f2(0.0f);   // largest speeds of the y-edges of this lane's columns
        const int jr = y0 + s0 - 2;   // patch row of ring row 0
        const bool drag = a.manningf > 0.0f;

        auto load = [&](const float *r, C2 &c) {   // y roles: hn = hv, ht = hu
            c.q0 = ld2(r); c.ht = ld2(r + kTileRing); c.hn = ld2(r + 2 * kTileRing); c.B = ld2(r + 3 * kTileRing);
            c.h = sub(c.q0, c.B);
        };
        auto ratio = [&](int k) { return cratP[jr + k]; };   // GEO, edge k >= 1
        auto speed = [&](int k, float2 n0, float2 s2) {   // edge k bounds a row of the segment: 2 .. hs + 2
            const float cr = GEO ? ratio(k) : 1.0f;
            sp.x = fmaxf(sp.x, fmaxf(n0.x, s2.x) * cr);
            sp.y = fmaxf(sp.y, fmaxf(n0.y, s2.y) * cr);
        };
        auto store = [&](float *d, float2 n0, float2 nn, float2 nt) {
            if (v8) {
                if (outx) { st2(d, n0); st2(d + fs, nt); st2(d + 2 * fs, nn); }
            } else {
                if (outx) { d[0] = n0.x; d[fs] = nt.x; d[2 * fs] = nn.x; }
                if (outy) { d[1] = n0.y; d[fs + 1] = nt.y; d[2 * fs + 1] = nn.y; }
            }
        };
        // ring row k, at r in the tile, to d
        auto update = [&](int k, const float *r, float *d, const float2 (&Dl)[3], const float2 (&Su)[3]) {
            C2 c;
            load(r, c);
            float2 dtk = f2(dtdy), m0 = add(Dl[0], Su[0]);
            if (GEO) {
                dtk = f2(dtdy * rkapP[jr + k]);
                m0 = fma(f2(cedP[jr + k + 1] - cedP[jr + k]), c.hn, m0);   // divergence of the edge length
            }
            float2 n0 = fnma(dtk, m0, c.q0);
            float2 nn = fnma(dtk, add(Dl[1], Su[1]), c.hn);
            float2 nt = fnma(dtk, add(Dl[2], Su[2]), c.ht);
            const float2 hq = sub(n0, c.B);
            if (!__all_sync(ALL, min_nan(hq.x, hq.y) >= drytol && max_nan(hq.x, hq.y) < 1e30f)) {
                post2(n0, nn, nt, c.B, drytol);
                // a surface that is not a finite number reaches the host as an infinite speed
                if ((outx && !(fabsf(n0.x) < 1e30f)) || (outy && !(fabsf(n0.y) < 1e30f))) smy = INFINITY;
            }
            if (drag) friction2(n0, nt, nn, c.B, drytol, a.manningf, dt1 * a.rR);
            store(d, n0, nn, nt);
        };
        // what edge k gives its rows, weighted by its length (GEO)
        auto weigh = [&](int k, float2 (&S)[3], float2 (&D)[3]) {
            if (GEO) {
                const float2 ce = f2(cedP[jr + k]);
#pragma unroll
                for (int m = 0; m < 3; m++) { S[m] = mul(ce, S[m]); D[m] = mul(ce, D[m]); }
            }
        };

        // The march for still water and the ocean only; false as soon as an edge is
        // neither.  One iteration: cells p (row k - 1) and c, edges m (k - 1) and n
        // with the factors cm, cn of their third waves (kept in place of s2); um: the
        // contact wave of the edge below m; rm and rp: edges k - 1 and k - 2 are at
        // rest; pm: p's momenta, bits or'ed.  STEADY: 4 <= k; the ramp is k = 0 .. 3.
        // c, pn and pt of p are formed again: the registers they would take cost more.
        const float *rk = cs;   // ring row k
        float *dk = dst + pitch;   // where row k - 2 goes: advanced before row 2 is stored, at k = 4
        auto ocean = [&](auto steady, int k, C2 &p, C2 &c, const W2 &m, W2 &n, float2 um, float2 &un, bool rm, bool &rn,
                         bool &rp, unsigned pm, unsigned &cm, float2 (&Dp)[3]) -> bool {
            constexpr bool STEADY = decltype(steady)::value;
            load(rk, c);
            const float *r2 = rk - 2 * kTileRow;
            rk += kTileRow;
            if (STEADY) dk += pitch;
            bool wet = min_nan(c.h.x, c.h.y) >= drytol;
            cm = __float_as_uint(c.hn.x) | __float_as_uint(c.hn.y) | __float_as_uint(c.ht.x) | __float_as_uint(c.ht.y);
            if (!STEADY && k == 0) {
                derive_wet(c, sqrtg);
                rn = true;
                return __all_sync(ALL, wet);
            }
            const float2 d1 = sub(c.q0, p.q0);
            rn = __all_sync(ALL, wet && ((cm | pm | __float_as_uint(d1.x) | __float_as_uint(d1.y)) & 0x7fffffffu) == 0u);
            derive_wet(c, sqrtg);
            p.c = mul(f2(sqrtg), p.sq);
            un = m.z1t;
            if (rn) {   // the speeds are sqrt(g h) of the cells and of the edge's mean depth
                zero_waves(n);
                const float2 ch = sqrt2(mul(f2(0.5f * g), add(p.h, c.h)));
                if (STEADY ? k <= hs + 2 : k >= 2) speed(k, make_float2(fmaxf(p.c.x, ch.x), fmaxf(p.c.y, ch.y)), c.c);
            } else {
                p.pn = mul(p.hn, p.u); p.pt = mul(p.hn, p.v);
                const float2 ok = riemann2_ocean(g, p, c, n);
                if (!__all_sync(ALL, wet && fminf(ok.x, ok.y) > 0.0f)) return false;
                if (STEADY ? k <= hs + 2 : k >= 2) speed(k, n.n0, n.s2);
                n.s2 = third_factor(n, dot3(m.z2m, m.z2n, m.z2t, n.z2m, n.z2n, n.z2t), f2(GEO ? -dtdy * ratio(k) : -dtdy));
            }
            if (STEADY || k == 3) {
                if (rm) {
                    if (STEADY) {
                        if (rp) {   // nothing moves: the row as it is
                            C2 q;
                            load(r2, q);
                            store(dk, q.q0, q.hn, q.ht);
                        } else {
                            const float2 zero[3] = {f2(0.0f), f2(0.0f), f2(0.0f)};
                            update(k - 2, r2, dk, Dp, zero);
                        }
                    }
                    Dp[0] = Dp[1] = Dp[2] = f2(0.0f);
                } else {
                    float2 S[3], D[3];
                    const float2 d0 = dot3(n.y0m, n.y0n, n.y0t, m.y0m, m.y0n, m.y0t);
                    const float2 t1 = make_float2(m.s1.x >= 0.0f ? um.x : n.z1t.x, m.s1.y >= 0.0f ? um.y : n.z1t.y);
                    limit2_ocean(m, d0, t1, m.s2, f2(GEO ? -dtdy * ratio(k - 1) : -dtdy), S, D);
                    weigh(k - 1, S, D);
                    if (STEADY) update(k - 2, r2, dk, Dp, S);
#pragma unroll
                    for (int q = 0; q < 3; q++) Dp[q] = D[q];
                }
            }
            rp = rm;
            return true;
        };
        const int last = hs + 3;
        // a segment with a dry cell goes to the general march at once
        bool good = true;
        for (int q = s0 >> 5; q <= (s0 + last) >> 5; q++) {
            const int lo = max(s0 - 32 * q, 0), hi = min(s0 + last - 32 * q, 31);
            if (dry_rows[q] & ((0xffffffffu >> (31 - hi)) & (0xffffffffu << lo))) good = false;
        }
        if (good) {
            C2 ca, cb;
            W2 ea, eb;
            float2 ua = f2(0.0f), ub = f2(0.0f), Dp[3];
            bool ra = true, rb = true, rp = true;
            unsigned ma = 0u, mb = 0u;
#pragma unroll
            for (int q = 0; q < 3; q++) Dp[q] = f2(0.0f);
            zero_waves(eb);
            // the ramp, rolled: its state copied from one iteration to the next
#pragma unroll 1
            for (int k = 0; good && k < 4; k++) {
                good = ocean(std::false_type(), k, cb, ca, eb, ea, ub, ua, rb, ra, rp, mb, ma, Dp);
                cb = ca; eb = ea; ub = ua; rb = ra; mb = ma;
            }
#pragma unroll 1
            for (int k = 4; good && k <= last; k += 2) {   // the two cells and edges in flight swap roles
                good = ocean(std::true_type(), k, cb, ca, eb, ea, ub, ua, rb, ra, rp, mb, ma, Dp);
                if (!good || k == last) break;
                good = ocean(std::true_type(), k + 1, ca, cb, ea, eb, ua, ub, ra, rb, rp, ma, mb, Dp);
            }
        }
        if (!good) {
            // the general march, from the segment's first row (rows already written get
            // the same values again)
            C2 p, c;
            W2 wo, wm, wn;   // edges k - 2, k - 1, k
            float2 Dp[3];
            bool dm = true;   // edge k - 1 lies between dry cells
            zero_waves(wo); zero_waves(wm);
#pragma unroll
            for (int q = 0; q < 3; q++) Dp[q] = f2(0.0f);
#pragma unroll 1
            for (int k = 0; k <= last; k++) {
                load(cs + k * kTileRow, c);
                derive(c, sqrtg, drytol);
                if (k >= 1) {
                    const bool dn = !__any_sync(ALL, c.wx || c.wy || p.wx || p.wy);
                    if (dn) {
                        zero_waves(wn);
                    } else {
                        riemann2(g, p, c, wn);
                        if (k >= 2 && k <= hs + 2) speed(k, wn.n0, wn.s2);
                    }
                    if (k >= 3) {
                        float2 S[3], D[3];
                        if (dm) {
#pragma unroll
                            for (int q = 0; q < 3; q++) { S[q] = f2(0.0f); D[q] = f2(0.0f); }
                        } else {
                            // upwind of edge k - 1: edge k - 2 or k
                            const bool a0 = wm.n0.x <= 0.0f, a1 = wm.s1.x >= 0.0f, a2 = wm.s2.x >= 0.0f;
                            const bool b0 = wm.n0.y <= 0.0f, b1 = wm.s1.y >= 0.0f, b2 = wm.s2.y >= 0.0f;
                            auto up = [](float2 lo, float2 hi, bool x, bool y) { return make_float2(x ? lo.x : hi.x, y ? lo.y : hi.y); };
                            const float2 d0 = dot3(up(wo.y0m, wn.y0m, a0, b0), up(wo.y0n, wn.y0n, a0, b0),
                                                   up(wo.y0t, wn.y0t, a0, b0), wm.y0m, wm.y0n, wm.y0t);
                            const float2 d2 = dot3(up(wo.z2m, wn.z2m, a2, b2), up(wo.z2n, wn.z2n, a2, b2),
                                                   up(wo.z2t, wn.z2t, a2, b2), wm.z2m, wm.z2n, wm.z2t);
                            limit2(wm, d0, up(wo.z1t, wn.z1t, a1, b1), d2, f2(GEO ? dtdy * ratio(k - 1) : dtdy), S, D);
                            weigh(k - 1, S, D);
                        }
                        if (k >= 4) update(k - 2, cs + (k - 2) * kTileRow, dst + (long long)(k - 2) * pitch, Dp, S);
#pragma unroll
                        for (int q = 0; q < 3; q++) Dp[q] = D[q];
                    }
                    wo = wm; wm = wn;
                    dm = dn;
                }
                p = c;
            }
        }
        smy = fmaxf(smy, fmaxf(outx ? sp.x : 0.0f, outy ? sp.y : 0.0f));
    }

    // ---- the CTA's largest speeds
    if (!(smx > 0.0f)) smx = 0.0f;
    if (!(smy > 0.0f)) smy = 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        smx = fmaxf(smx, __shfl_xor_sync(ALL, smx, o));
        smy = fmaxf(smy, __shfl_xor_sync(ALL, smy, o));
    }
    if (lane == 0) { red[0][warp] = smx; red[1][warp] = smy; }
    __syncthreads();
    if (t == 0) {
        float mx = 0.0f, my = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; q++) { mx = fmaxf(mx, red[0][q]); my = fmaxf(my, red[1][q]); }
        atomic_max_speed(a.smax + 2 * P.scen + 0, (double)mx);
        atomic_max_speed(a.smax + 2 * P.scen + 1, (double)my);
    }
}

template <int NW, bool GEO, bool BULK>
__global__ void __launch_bounds__(NW * 32, 16 / NW) step_tile_f32(StepArgs a)
{
    if (!launch_live(a)) return;
    tile_item<NW, GEO, BULK>(a, blockIdx.x);
    step_tail<float, true>(a);
}

// The retake launch (a.gate set): a CTA slot's worth of CTAs, which leave at once
// unless a scenario is to be retaken and otherwise stride over the items.  With as
// many CTAs as items it cost 12 us on the 4096^2 grid to find nothing to do.
template <bool GEO> __global__ void __launch_bounds__(128, 4) retake_tile_f32(StepArgs a)
{
    if (!launch_live(a)) return;
    for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        tile_item<4, GEO, false>(a, item);
        __syncthreads();   // before the next tile overwrites this one
    }
    step_tail<float, true>(a);
}

}  // namespace tsu
