// Voxel-driven gather backprojection of the MAR-DEAM c-step (arXiv 2202.00116,
// Sec. 2.3): b~_i(x) = sum_y h(x,y) B~_i(y) and delta_i(x) = sum_y h(x,y) D_i(y)
// per voxel, fused with the log-ratio update c_i <- c_i - (1/Z) ln(b^_i / b~_i);
// the gradient b^ - b~; and the plain transpose A^T y of two-component ray data.
// h is Joseph's; the gather recomputes the forward kernel's sample positions bit for
// bit, so the weights are the forward's transposed (on single slices, and for heights
// just below slice 0, to half a unit in the last place of 1) and no atomics are needed.
#include <math.h>

#include "deam_internal.h"
#include "deam_pair.cuh"

namespace deam {

// Voxel-driven gather backprojection.  A thread owns one (ix, iy) column and the
// SLAB slices of one z-slab, whose sums it keeps in shared memory ([slot][thread]:
// conflict-free).  A warp owns an 8 x 4 patch of columns and takes the views that
// can reach its slab two at a time (STEP; one where they lie far apart): the channels
// whose rays tap a column come from the fan angles of the patch's corners, and then a
// row of the detector is one turn of the loop, which adds the samples of up to RAYS
// rays of each view (2.6 rays per view and column at 512^2 x 816 channels; four, or
// two and one on coarse fans).  These lie within a few
// hundredths of a slice of each other, so nearly always all between the same two
// slices, and one read and write of these two serves them all.  Sample positions
// are the forward kernel's, bit for bit (same in-plane table, same explicitly
// rounded t(p), omega_r and fz).
//
// What bounds it: issue (0.6 per cycle and scheduler) and the latency of the
// payload gathers with the 20 warps per SM that 96 registers allow, the L1 data
// path being 67-69 % busy.  The c-step's instances of four rays and two views spill
// 56 bytes of stores and 128 of loads at 96 registers, the adjoint's 8 (ptxas);
// 128 registers without spills at 4 blocks were as fast, 80 at 6 slower.  One ray at a time (two views abreast) cost twice the
// shared-memory traffic, half the loads in flight and 70 instead of 31
// instructions per (column, ray, row): 37.4 -> 23.3 ms on one rotation of the
// 512^2 x 64 scan, 20.5 -> 8.5 ms on one of the 256^2 x 32 scan.  Measured and
// slower: sums in registers with the slices unrolled (37.5 ms on the first),
// four views per turn (29-50 ms), first moments of the rays' heights instead of
// each ray's own weights (32.6 ms, and no longer the forward's weights).
constexpr int kBwdThreads = 128;

// A ray's data, or the sums of a voxel: (b~_1, b~_2) and, for the c-step, also
// (delta_1, delta_2).  The gradient carries the second pair alone, the plain
// adjoint its two components.
template <bool FOUR>
struct Sums {
    pair32 a, b;
};
template <>
struct Sums<false> {
    pair32 a;
};

template <int MODE>
__device__ __forceinline__ Sums<MODE == BWD_UPDATE> ray_data(const BwdArgs& A, long long i) {
    Sums<MODE == BWD_UPDATE> P;
    if constexpr (MODE == BWD_UPDATE)
        asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(P.a), "=l"(P.b) : "l"(A.payload + i));
    else if constexpr (MODE == BWD_GRADIENT)
        asm("ld.global.nc.u64 %0, [%1 + 8];" : "=l"(P.a) : "l"(A.payload + i));
    else
        asm("ld.global.nc.u64 %0, [%1];" : "=l"(P.a) : "l"(A.rays2 + i));
    return P;
}

// s + w P
template <bool FOUR>
__device__ __forceinline__ void add_scaled(Sums<FOUR>& s, pair32 w, const Sums<FOUR>& P) {
    s.a = fma2(w, P.a, s.a);
    if constexpr (FOUR) s.b = fma2(w, P.b, s.b);
}
template <bool FOUR>
__device__ __forceinline__ void add_to(Sums<FOUR>& s, const Sums<FOUR>& P) {
    s.a = add2(s.a, P.a);
    if constexpr (FOUR) s.b = add2(s.b, P.b);
}

// Fan angle of a direction (dot along the central ray, crs across it).  Within
// 31 degrees of the central ray (every fan of this scanner family) a degree-9
// odd polynomial, the Chebyshev interpolant of atan(x) / x in x^2 on [0, 0.36]
// (3e-7 rad); it only places the channel window, whose margin is larger by far.
__device__ __forceinline__ float fan_angle(float crs, float dot) {
    if (fabsf(crs) > 0.6f * dot) return atan2f(crs, dot);
    const float r = __fdividef(crs, dot), x = r * r;
    float s = 0.0578066558f;
    s = fmaf(s, x, -0.128525928f);
    s = fmaf(s, x, 0.198297724f);
    s = fmaf(s, x, -0.333260238f);
    s = fmaf(s, x, 0.999999464f);
    return s * r;
}

// What a view asks of the 8 x 4 columns of a warp, seen from one of their corner
// columns: the corner's channel coordinate u, the half width hw of a column's
// channel window around its own coordinate, and the rows [lo, hi] (real numbers)
// that can reach the slab.
struct CornerWindow {
    float u, hw, lo, hi;
};

template <int C>
__device__ __forceinline__ CornerWindow corner_window(const Geo& G, int v, float fix, float fiy, float zlo, float zhi) {
    constexpr float kDiag = 64.f * C * C + 32.f * (C - 1);  // over the patch's diagonal, squared
    CornerWindow W;
    const float4 vw = __ldg(&G.view4[v]);
    const float sz = __ldg(&G.view_z[v]);
    const float px = (fix - vw.x) * G.dx, py = (fiy - vw.y) * G.dy;
    const float dot = -fmaf(px, vw.z, py * vw.w);
    const float crs = fmaf(px, vw.w, -py * vw.z);
    const float d2 = fmaf(px, px, py * py);
    const float inv = rsqrtf(d2);
    const float dist = d2 * inv;
    const float rest = __fdividef(1.f, fmaxf(dist - G.vox_reach_mm, 1e-3f * dist));
    const float rho = G.vox_reach_mm * rest;  // a voxel edge as an angle, a little over
    // A ray taps a column if at the column's plane it passes within one voxel
    // edge e of its centre, across the dominant axis: e |cos| of perpendicular
    // distance, an angle below e |cos| / (dist - e).  Taking the larger of the
    // two axes covers rays of either dominance.  What varies over the patch is
    // covered by the corners up to second order in its angle (64 rho^2), and so is
    // the error of interpolating u between them ((7^2 + 3^2) / 8 rho^2 as |u''| is
    // at most 1 / (dist^2 dgamma)); 0.05 channel of margin covers the rounding.
    // (The bound e / (dist - e), without the cosine, lets through up to 40 % more
    // channels.)
    const float edge = fmaxf(fabsf(px) * G.dy, fabsf(py) * G.dx) * inv * 1.001f;
    const float bend = rho * rho;
    W.hw = fmaf(fmaf(edge * rest, fmaf(kDiag, bend, 1.f), 0.125f * kDiag * bend), G.inv_dgamma, 0.05f);
    W.u = fmaf(fan_angle(crs, dot), G.inv_dgamma, G.chan_c0);
    W.lo = 0.f;
    W.hi = (float)(G.R - 1);
    const float t = dist * G.inv_sdd, slope = t * G.domega;
    if (G.R > 1 && slope > 1e-20f) {
        // fz(r) = sigma_z + t (omega0 + r domega) with t = dist / sdd for a ray
        // through the column's centre; the rays that tap it pass within one voxel
        // edge, which moves t by at most rho of itself and the row of a height z by
        // the same share of (z - sigma_z) / (t domega)
        const float is = __fdividef(1.f, slope);
        const float off = G.omega0 * t * is;
        const float share = rho * fmaf(16.f, rho, 1.f);
        const float ulo = (zlo - sz) * is, uhi = (zhi - sz) * is;
        W.lo = ulo - off - fmaf(fabsf(ulo), share, 0.02f);
        W.hi = uhi - off + fmaf(fabsf(uhi), share, 0.02f);
    }
    if (rho * C > 0.1f) {  // voxels too large for these bounds: every channel and row
        W.u = 0.f;
        W.hw = 1e9f;
        W.lo = 0.f;
        W.hi = (float)(G.R - 1);
    }
    return W;
}

// The 8 x 4 columns of a warp: a lane's place in the patch, and what eight views
// ask of it (every lane looks at one view from one corner of the patch: done for
// each column, a window costs as much as a row of samples).
template <int C>
struct Patch {
    int ix, iy;       // the lane's first column
    float mx, my;     // its columns' centre in patch widths from the patch's (inside the image)
    float rx, ry;     // 1 / patch widths
    float cx, cy;     // the corner that the lane looks from
    float u, ux, uy;  // of the lane's view: channel coordinate at the patch's centre, and its change over the patch
    float hw;         // half width of the window of the columns of any lane
    int row0, row1;   // rows of the lane's view (STEP 2: of its pair 2 w, 2 w + 1) that can reach the slab

    __device__ __forceinline__ Patch(const Geo& G, int x0, int y0, int lane) {
        // lanes in 4 x 2 blocks of columns: the eight lanes of a 128-byte wavefront
        // read few distinct channels whatever the view's direction
        const int lx = (lane & 3) + ((lane >> 1) & 4), ly = ((lane >> 2) & 1) + ((lane >> 3) & 2);
        ix = x0 + C * lx;
        iy = y0 + C * ly;
        const int ex = min(8 * C - 1, max(G.nx - 1 - x0, 0)), ey = min(4 * C - 1, max(G.ny - 1 - y0, 0));
        constexpr float kHalf = 0.5f * (C - 1);
        rx = __fdividef(1.f, (float)max(ex, 1));
        ry = __fdividef(1.f, (float)max(ey, 1));
        mx = ((float)(C * lx) + kHalf) * rx - 0.5f;
        my = ((float)(C * ly) + kHalf) * ry - 0.5f;
        cx = (float)(x0 + ((lane & 1) ? ex : 0));
        cy = (float)(y0 + ((lane & 2) ? ey : 0));
    }
    // views vb .. vb + 7 (the last repeated beyond it): lane 4 w + c looks at view w
    template <int STEP>
    __device__ __forceinline__ void look(const Geo& G, int vb, int last, int lane, float zlo, float zhi) {
        const CornerWindow win = corner_window<C>(G, min(vb + (lane >> 2), last), cx, cy, zlo, zhi);
        float lo = win.lo, hi = win.hi;
        hw = win.hw;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            hw = fmaxf(hw, __shfl_xor_sync(0xffffffffu, hw, o));
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        // the plane through the corners' coordinates; what they are off it by, and
        // (several columns per lane) the way from the centre to any of them, widen
        // the window
        const float a = __shfl_sync(0xffffffffu, win.u, lane & ~3), b = __shfl_sync(0xffffffffu, win.u, lane & ~3 | 1);
        const float c = __shfl_sync(0xffffffffu, win.u, lane & ~3 | 2), d = __shfl_sync(0xffffffffu, win.u, lane | 3);
        u = 0.25f * ((a + b) + (c + d));
        ux = 0.5f * ((b - a) + (d - c));
        uy = 0.5f * ((c - a) + (d - b));
        hw += 0.25f * fabsf((b - a) - (d - c));
        if (C > 1) hw += 0.5f * (C - 1) * (fabsf(ux) * rx + fabsf(uy) * ry);
        if (STEP > 1) {  // both views of a pair
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, 4));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, 4));
        }
        row0 = max(0, __float2int_ru(fminf(lo, (float)G.R)));
        row1 = min(G.R - 1, __float2int_rd(fmaxf(fminf(hi, (float)G.R), -1.f)));
    }
    // channels [k0, k1] of view w whose rays can tap the lane's columns
    __device__ __forceinline__ void channels(const Geo& G, int w, int& k0, int& k1) const {
        const float h = __shfl_sync(0xffffffffu, hw, 4 * w);
        float at = __shfl_sync(0xffffffffu, u, 4 * w);
        at = fmaf(mx, __shfl_sync(0xffffffffu, ux, 4 * w), at);
        at = fmaf(my, __shfl_sync(0xffffffffu, uy, 4 * w), at);
        k0 = __float2int_ru(fmaxf(at - h, 0.f));
        k1 = __float2int_rd(fminf(at + h, (float)(G.K - 1)));
    }
};

// G neighbouring rays (v, k .. k + G - 1) at a column: Joseph length x in-plane
// weight (0: the ray does not tap the column) and ray parameter.
template <int G_>
struct Rays {
    float c[G_], t[G_];
};

// One ray's c (0: it does not tap the column) and t, from its table entry vk
__device__ __forceinline__ void tap_ray(const Geo& G, long long vk, float fix, float fiy, float& c, float& t) {
    const InPlane ip = inplane_at(__ldg(&G.ip4[vk]), __ldg(&G.ipL[vk]));
    const float pf = ip.axis ? fiy : fix, qf = ip.axis ? fix : fiy;
    const float fq = __fmaf_rn(pf, ip.bq, ip.aq);
    const float jq = floorf(fq);
    const float aq = fq - jq;
    float wq = 0.f;
    if (jq == qf) wq = 1.f - aq;
    else if (jq == qf - 1.f) wq = aq;
    c = ip.Lxy * wq;
    t = ray_t(ip, pf);
}

template <int G_>
__device__ __forceinline__ void load_rays(const Geo& G, Rays<G_>& y, int v, int k, int k1, float fix, float fiy,
                                          float& tmin, float& tmax) {
    const long long vk = (long long)v * G.K + k;
#pragma unroll
    for (int g = 0; g < G_; ++g) {
        y.c[g] = y.t[g] = 0.f;
        if (k + g <= k1 &&
            DEAM_IN_BOUNDS(G, k >= 0 && vk + g < (long long)G.V * G.K, SITE_BWD_TABLE, vk + g)) {
            tap_ray(G, vk + g, fix, fiy, y.c[g], y.t[g]);
            if (y.c[g] != 0.f) {
                tmin = fminf(tmin, y.t[g]);
                tmax = fmaxf(tmax, y.t[g]);
            }
        }
    }
}

template <int MODE, int G_>
__device__ __forceinline__ void fetch_rays(const Geo& G, const BwdArgs& A, const Rays<G_>& y, long long i,
                                           Sums<MODE == BWD_UPDATE> (&P)[G_]) {
#pragma unroll
    for (int g = 0; g < G_; ++g)
        if (y.c[g] != 0.f && DEAM_IN_BOUNDS(G, i + g < (long long)G.V * G.R * G.K, SITE_BWD_RAY, i + g))
            P[g] = ray_data<MODE>(A, i + g);
}

// A sample a above a slice (0 <= a < 1), times c: into that slice's sums lo and
// the next one's hi.
template <bool FOUR>
__device__ __forceinline__ void add_sample(Sums<FOUR>& lo, Sums<FOUR>& hi, float a, float c, const Sums<FOUR>& P) {
    const float w1 = c * a, w0 = c - w1;
    add_scaled<FOUR>(lo, dup2(w0), P);
    add_scaled<FOUR>(hi, dup2(w1), P);
}

// A voxel's sums a = (b~_1, b~_2, delta_1, delta_2), or the two of A^T y or the
// gradient, to their end: stored, or the c-step.  False: out of range (checked
// builds).
template <int MODE>
__device__ __forceinline__ bool finish_voxel(const Geo& G, const BwdArgs& A, long long vi, float4 a,
                                             unsigned long long& skipped) {
    if (!DEAM_IN_BOUNDS(G, vi < (long long)G.nx * G.ny * G.nz, SITE_BWD_IMAGE, vi)) return false;
    if (MODE != BWD_UPDATE) {  // A^T y, or the gradient delta_i
        A.img[vi] = make_float2(a.x, a.y);
        return true;
    }
    if (A.sums) {  // regularised c-step: reg_update_kernel finishes the update
        A.sums[vi] = a;
        return true;
    }
    float2 c = A.img[vi];
    // c-step: c_i <- c_i - (1/Z) ln(b^_i / b~_i) = c_i - (1/Z) log1p(delta_i / b~_i);
    // the ratio and its logarithm in FP64 (two per voxel and iteration)
    if (a.x > 0.f && a.z > -a.x) {
        c.x = (float)fma(-log1p((double)a.z / (double)a.x), A.invZ, (double)c.x);
        if (A.clamp_nonneg) c.x = fmaxf(c.x, 0.f);
    } else {
        ++skipped;
    }
    if (a.y > 0.f && a.w > -a.y) {
        c.y = (float)fma(-log1p((double)a.w / (double)a.y), A.invZ, (double)c.y);
        if (A.clamp_nonneg) c.y = fmaxf(c.y, 0.f);
    } else {
        ++skipped;
    }
    A.img[vi] = c;
    return true;
}

// One (column tile, z-slab) of the gather backprojection: the work of one block
// of VS groups of TX x TY threads.  Each group takes every VS-th eight views;
// their sums are added in a fixed order (deterministic).  A turn takes RAYS rays of
// STEP views.
template <int MODE, int SLAB, int TX, int TY, int VS, int STEP, int RAYS>
__device__ __forceinline__ void bwd_tile(const Geo& G, const BwdArgs& A, Sums<MODE == BWD_UPDATE>* smem, int bx, int by,
                                         int slab) {
    // MODE: BWD_ADJOINT (A^T of two-component ray data), BWD_UPDATE (payload ->
    // b~, delta -> c-step), BWD_GRADIENT (payload -> delta = b^ - b~ = dF/dc)
    constexpr bool FOUR = MODE == BWD_UPDATE;
    constexpr int NT = TX * TY;
    static_assert(TX % 8 == 0 && TY % 4 == 0, "warps own 8 x 4 columns");
    // a warp's 32 columns are an 8 x 4 patch: they see nearly the same ray
    // parameter, so their rows fall between the same slices at nearly the same turn
    const int tid = threadIdx.x % NT, group = threadIdx.x / NT;
    const int warp = tid >> 5, lane = tid & 31;
    Patch<1> patch(G, bx * TX + (warp % (TX / 8)) * 8, by * TY + (warp / (TX / 8)) * 4, lane);
    const int ix = patch.ix, iy = patch.iy;
    const bool inside = ix < G.nx && iy < G.ny;
    const int z0 = slab * SLAB;
    constexpr int G_ = RAYS;
    Sums<FOUR>* acc = smem + group * (SLAB + 2) * NT + tid;  // slot s (slice z0 - 1 + s) at acc[s * NT]
#pragma unroll
    for (int s = 0; s < SLAB + 2; ++s) acc[s * NT] = Sums<FOUR>{};
    // views that can reach this column tile's slab (host-computed per tile)
    const int2 vrange =
        __ldg(&A.slab_views[((long long)slab * ((G.ny + TY - 1) / TY) + by) * ((G.nx + TX - 1) / TX) + bx]);
    const float fix = (float)ix, fiy = (float)iy;
    const float zlo = (float)(z0 - 1), zhi = (float)(z0 + SLAB);
    for (int vb = vrange.x + 8 * group; vb <= vrange.y; vb += 8 * VS) {
        patch.template look<STEP>(G, vb, vrange.y, lane, zlo, zhi);
        // Views in pairs (STEP 2): their samples of a row lie within a few hundredths of a
        // slice of each other, so nearly always all between the same two slices
        // (one read and write of their sums serves the rays of both)
        const int nv = min(8, vrange.y - vb + 1);
        for (int w = 0; w < nv; w += STEP) {
            const int v = vb + w;
            const int r0 = __shfl_sync(0xffffffffu, patch.row0, 4 * w), r1 = __shfl_sync(0xffffffffu, patch.row1, 4 * w);
            int ka0, ka1, kb0, kb1;
            patch.channels(G, w, ka0, ka1);
            patch.channels(G, w + STEP - 1, kb0, kb1);
            if (r0 > r1) continue;  // no row of these views reaches the slab
            if (!inside) continue;
            const bool second = STEP > 1 && w + 1 < nv;
            if (!second) kb1 = kb0 - 1;
            const float sza = __ldg(&G.view_z[v]), szb = __ldg(&G.view_z[second ? v + 1 : v]);
            const int n = max(ka1 - ka0, kb1 - kb0);
            for (int j = 0; j <= n; j += G_) {
                Rays<G_> a, b;
                float ta0 = INFINITY, ta1 = 0.f, tb0 = INFINITY, tb1 = 0.f;
                load_rays<G_>(G, a, v, ka0 + j, ka1, fix, fiy, ta0, ta1);
                if (STEP > 1) load_rays<G_>(G, b, v + 1, kb0 + j, kb1, fix, fiy, tb0, tb1);
                if (ta1 == 0.f && tb1 == 0.f) continue;
                long long i = ((long long)v * G.R + r0) * G.K + j;
                const long long next_view = (long long)G.R * G.K;
                Sums<FOUR> P[G_], Q[G_];
#pragma unroll
                for (int g = 0; g < G_; ++g) P[g] = Q[g] = Sums<FOUR>{};
                float rf = (float)r0;
#pragma unroll 1
                for (int r = r0; r <= r1; ++r) {
                    fetch_rays<MODE, G_>(G, A, a, i + ka0, P);
                    if (STEP > 1) fetch_rays<MODE, G_>(G, A, b, i + next_view + kb0, Q);
                    const float om = __fmaf_rn(rf, G.domega, G.omega0);
                    const float rowf = MODE == BWD_ADJOINT ? __ldg(&G.row[r]).y : 1.f;
                    rf += 1.f;
                    i += G.K;
                    // lowest and highest sample of the row
                    const float za0 = row_fz(sza, om, ta0), za1 = row_fz(sza, om, ta1);
                    const float zb0 = row_fz(szb, om, tb0), zb1 = row_fz(szb, om, tb1);
                    float zmin = INFINITY, zmax = -INFINITY;
                    if (ta1 != 0.f) {
                        zmin = fminf(za0, za1);
                        zmax = fmaxf(za0, za1);
                    }
                    if (tb1 != 0.f) {
                        zmin = fminf(zmin, fminf(zb0, zb1));
                        zmax = fmaxf(zmax, fmaxf(zb0, zb1));
                    }
                    const float f = floorf(zmin);
                    const int slot = (int)f - (z0 - 1);
                    if (zmax < f + 1.f) {
                        if (slot < 0 || slot > SLAB) continue;
                        Sums<FOUR> lo = acc[slot * NT], hi = acc[(slot + 1) * NT];
#pragma unroll
                        for (int g = 0; g < G_; ++g) {
                            add_sample<FOUR>(lo, hi, row_fz(sza, om, a.t[g]) - f, a.c[g] * rowf, P[g]);
                            if (STEP > 1)
                                add_sample<FOUR>(lo, hi, row_fz(szb, om, b.t[g]) - f, b.c[g] * rowf, Q[g]);
                        }
                        acc[slot * NT] = lo;
                        acc[(slot + 1) * NT] = hi;
                    } else {
#pragma unroll 1
                        for (int s = max(slot, 0); s <= SLAB; ++s) {
                            const float fs = (float)(z0 - 1 + s);
                            if (zmax < fs) break;
                            Sums<FOUR> lo = acc[s * NT], hi = acc[(s + 1) * NT];
#pragma unroll
                            for (int g = 0; g < G_; ++g) {
                                // rounded down: a height just below slice 0 is less than 1 above
                                // slice -1 (all other differences are exact)
                                const float x = __fsub_rd(row_fz(sza, om, a.t[g]), fs);
                                const float y = __fsub_rd(row_fz(szb, om, b.t[g]), fs);
                                if (x >= 0.f && x < 1.f) add_sample<FOUR>(lo, hi, x, a.c[g] * rowf, P[g]);
                                if (STEP > 1 && y >= 0.f && y < 1.f)
                                    add_sample<FOUR>(lo, hi, y, b.c[g] * rowf, Q[g]);
                            }
                            acc[s * NT] = lo;
                            acc[(s + 1) * NT] = hi;
                        }
                    }
                }
            }
        }
        __syncwarp();
    }
    if constexpr (VS > 1) __syncthreads();
    if (!inside) return;
    unsigned long long skipped = 0;
#pragma unroll 1
    for (int s = group; s < SLAB; s += VS) {  // the groups share out the slices
        const int iz = z0 + s;
        if (iz >= G.nz) break;
        Sums<FOUR> sum = smem[(s + 1) * NT + tid];
#pragma unroll
        for (int g = 1; g < VS; ++g) add_to<FOUR>(sum, smem[(g * (SLAB + 2) + s + 1) * NT + tid]);
        const float2 lo = unpack2(sum.a);
        float4 a = make_float4(lo.x, lo.y, 0.f, 0.f);
        if constexpr (FOUR) {
            const float2 hi = unpack2(sum.b);
            a.z = hi.x;
            a.w = hi.y;
        }
        if (!finish_voxel<MODE>(G, A, ((long long)iz * G.ny + iy) * G.nx + ix, a, skipped)) break;
    }
    if (FOUR && skipped) atomicAdd(A.skipped, skipped);
}

// The sums of a thread's C x C columns (0, 0), (1, 0), (0, 1), (1, 1) over every
// VS-th eight views.  EXACT leaves out the rays whose weight is zero, else they are
// added with it.
template <int MODE, int C, int VS, bool FLAT, bool EXACT>
__device__ __forceinline__ void slice_sums(const Geo& G, const BwdArgs& A, Patch<C>& patch, bool inside, int group,
                                           int lane, Sums<MODE == BWD_UPDATE> (&acc)[C * C]) {
    constexpr bool FOUR = MODE == BWD_UPDATE;
    constexpr int NV = C > 1 ? 1 : 4;  // views abreast, a ray of each per turn
    const float fix = (float)patch.ix, fiy = (float)patch.iy;
#pragma unroll
    for (int j = 0; j < C * C; ++j) acc[j] = Sums<FOUR>{};
    for (int vb = 8 * group; vb < G.V; vb += 8 * VS) {
        patch.template look<2>(G, vb, G.V - 1, lane, -1.f, 1.f);
        const int nv = min(8, G.V - vb);
        for (int w = 0; w < nv; w += NV) {
            int k0[NV], k1[NV], n = -1;
#pragma unroll
            for (int u = 0; u < NV; ++u) {
                patch.channels(G, w + u, k0[u], k1[u]);
                if (NV > 1 && w + u >= nv) k1[u] = k0[u] - 1;
                n = max(n, k1[u] - k0[u]);
            }
            if (!inside) continue;
            const int v = vb + w;
#pragma unroll 1
            for (int j = 0; j <= n; ++j) {
                InPlane ip[NV];
                Sums<FOUR> P[NV];
                float sz[NV];
#pragma unroll
                for (int g = 0; g < NV; ++g) {
                    const int k = k0[g] + j;
                    const bool on = NV == 1 || k <= k1[g];
                    const long long i = on ? (long long)(v + g) * G.K + k : 0;
                    ip[g] = InPlane{};
                    P[g] = Sums<FOUR>{};
                    sz[g] = __ldg(&G.view_z[on ? v + g : 0]);
                    if (!DEAM_IN_BOUNDS(G, i >= 0 && i < (long long)G.V * G.K, SITE_BWD_TABLE, i)) continue;
                    P[g] = ray_data<MODE>(A, i);
                    ip[g] = inplane_at(__ldg(&G.ip4[i]), __ldg(&G.ipL[i]));
                    if (!on) ip[g].Lxy = 0.f;
                }
#pragma unroll
                for (int g = 0; g < NV; ++g) {
                    // planes p0 .. p0 + C - 1, at each of them the shares of q0 .. q0 + C - 1
                    const float p0 = ip[g].axis ? fiy : fix, q0 = ip[g].axis ? fix : fiy;
                    float c[C][C];
#pragma unroll
                    for (int p = 0; p < C; ++p) {
                        const float pf = p0 + (float)p;
                        const float d = __fmaf_rn(pf, ip[g].bq, ip[g].aq) - q0;
                        float L = ip[g].Lxy;
                        if (!FLAT) L *= __saturatef(1.f - fabsf(row_fz(sz[g], G.omega0, ray_t(ip[g], pf))));
#pragma unroll
                        for (int q = 0; q < C; ++q) c[p][q] = L * __saturatef(1.f - fabsf(d - (float)q));
                    }
#pragma unroll
                    for (int j = 0; j < C * C; ++j) {
                        const float x = ip[g].axis ? c[j / C][j % C] : c[j % C][j / C];
                        if (!EXACT || x != 0.f) add_scaled<FOUR>(acc[j], dup2(x), P[g]);
                    }
                }
            }
        }
        __syncwarp();
    }
}

// One slice seen by one detector row (fan-beam scans): no rows and no slices to
// walk, so a thread keeps the sums of its C x C columns in registers.  A block is one
// 8 C x 4 C patch of columns; its VS warps take every VS-th eight views.  FLAT: the
// rays lie in the slice (no cone, source at its height).
//
// What bounds it: issue (0.85 per cycle and scheduler).  2 x 2 columns share the
// window, the ray's table entry and its data, and a plane's position gives two
// weights: 5.5 rays instead of four times 3.5, 80 instead of 165 instructions per
// column and view, 1.61 -> 0.87 ms at 512^2 x 1160 views with one ray per turn (two,
// three, four: 0.91, 0.98, 1.18 ms).  Small images leave too few patches for that:
// one column per thread, and the rays of four views in flight per turn to cover the
// loads (128^2 x 360 views: 53 us; 58 with four rays of one view, 57 with 2 x 2
// columns).  Skipping the columns that a ray does not tap, instead of adding zeros
// and looking for infinities afterwards, was 1.15 against 0.98 ms.
template <int MODE, int C, int VS, bool FLAT>
__global__ void __launch_bounds__(32 * VS, 32 / VS) bwd_slice_kernel(const Geo G, const BwdArgs A) {
    constexpr bool FOUR = MODE == BWD_UPDATE;
    __shared__ Sums<FOUR> part[VS * 32];
    const int lane = threadIdx.x & 31, group = threadIdx.x >> 5;
    const int ntx = (G.nx + 8 * C - 1) / (8 * C);
    Patch<C> patch(G, (blockIdx.x % ntx) * 8 * C, (blockIdx.x / ntx) * 4 * C, lane);
    const bool inside = patch.ix < G.nx && patch.iy < G.ny;
    Sums<FOUR> acc[C * C];
    slice_sums<MODE, C, VS, FLAT, false>(G, A, patch, inside, group, lane, acc);
    // a weight of zero takes nothing from finite data; where a sum has met an
    // infinity or a NaN, the rays that tap the column decide
    float zero = 0.f;
#pragma unroll
    for (int j = 0; j < C * C; ++j) {
        const float2 lo = unpack2(acc[j].a);
        zero += 0.f * lo.x + 0.f * lo.y;
        if constexpr (FOUR) {
            const float2 hi = unpack2(acc[j].b);
            zero += 0.f * hi.x + 0.f * hi.y;
        }
    }
    if (__any_sync(0xffffffffu, zero != 0.f))
        slice_sums<MODE, C, VS, FLAT, true>(G, A, patch, inside, group, lane, acc);
    const float rowf = MODE == BWD_ADJOINT ? __ldg(&G.row[0]).y : 1.f;  // else the payload carries it
    unsigned long long skipped = 0;
#pragma unroll
    for (int j = 0; j < C * C; ++j) {
        if (j) __syncthreads();  // the previous column's sums are read
        part[threadIdx.x] = acc[j];
        __syncthreads();
        const int ix = patch.ix + j % C, iy = patch.iy + j / C;
        if (group != j % VS || ix >= G.nx || iy >= G.ny) continue;
        Sums<FOUR> sum = part[lane];
#pragma unroll
        for (int g = 1; g < VS; ++g) add_to<FOUR>(sum, part[32 * g + lane]);
        const float2 lo = unpack2(sum.a);
        float4 a = make_float4(lo.x * rowf, lo.y * rowf, 0.f, 0.f);
        if constexpr (FOUR) {
            const float2 hi = unpack2(sum.b);
            a.z = hi.x;
            a.w = hi.y;
        }
        finish_voxel<MODE>(G, A, (long long)iy * G.nx + ix, a, skipped);
    }
    if (FOUR && skipped) atomicAdd(A.skipped, skipped);
}

template <int C, int VS, bool FLAT>
static cudaError_t launch_slice(int mode, const Geo& G, const BwdArgs& A, cudaStream_t s) {
    const int blocks = ((G.nx + 8 * C - 1) / (8 * C)) * ((G.ny + 4 * C - 1) / (4 * C));
    if (mode == BWD_UPDATE) bwd_slice_kernel<BWD_UPDATE, C, VS, FLAT><<<blocks, 32 * VS, 0, s>>>(G, A);
    else if (mode == BWD_GRADIENT) bwd_slice_kernel<BWD_GRADIENT, C, VS, FLAT><<<blocks, 32 * VS, 0, s>>>(G, A);
    else bwd_slice_kernel<BWD_ADJOINT, C, VS, FLAT><<<blocks, 32 * VS, 0, s>>>(G, A);
    return cudaGetLastError();
}

// Column tile of a block of VS view groups
template <int VS>
struct BwdTile {
    static constexpr int X = bwd_tile_x(VS), Y = bwd_tile_y(VS);
    static_assert(X * Y * VS == kBwdThreads, "view groups x columns fill the block");
};

// Blocks per SM: with one view a turn 80 registers do (16 views at 256^2 x 32, two
// iterations 1.26 ms, 1.39 with five blocks; the c-step's FP64 logarithms weigh most
// there and want the warps).
constexpr int bwd_blocks(int step) { return step == 1 ? 6 : 5; }

template <int MODE, int SLAB, int VS, int STEP, int RAYS>
__global__ void __launch_bounds__(kBwdThreads, bwd_blocks(STEP)) bwd_kernel(const Geo G, const BwdArgs A) {
    constexpr int TX = BwdTile<VS>::X, TY = BwdTile<VS>::Y;
    __shared__ Sums<MODE == BWD_UPDATE> acc[(SLAB + 2) * kBwdThreads];
    const int ntx = (G.nx + TX - 1) / TX, nty = (G.ny + TY - 1) / TY;
    int b = blockIdx.x;
    const int bx = b % ntx;
    b /= ntx;
    const int by = b % nty;
    bwd_tile<MODE, SLAB, TX, TY, VS, STEP, RAYS>(G, A, acc, bx, by, b / nty);
}

// Batched scans: one launch takes the column tiles x slabs of every
// scan of a slab class; each work item finds its scan by binary search in the
// prefix sums of tile counts.
// (the scan's descriptors are held in registers, hence one block per SM less).  Rays per
// turn follow the scan: three scans of 256^2 x 32 and 360 views with 100 channels 6.69 ms
// an iteration with four always, 4.96 now, with 60 channels 6.19 / 4.58, with 100 and
// slices of 1.5 mm 6.69 / 4.78; of 672 channels 15.0 ms either way.
template <int SLAB, int TX, int TY>
__global__ void __launch_bounds__(TX* TY, 4) bwd_batch_kernel(const BatchDesc B) {
    __shared__ Sums<true> acc[(SLAB + 2) * TX * TY];
    const long long total = __ldg(&B.btile_off[B.n]);
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
        const int i = find_scan(B.btile_off, B.n, t);
        const Geo G = B.geos[i];
        const BwdArgs A = B.bargs[i];
        long long lt = t - __ldg(&B.btile_off[i]);
        const int ntx = (G.nx + TX - 1) / TX, nty = (G.ny + TY - 1) / TY;
        const int bx = (int)(lt % ntx);
        lt /= ntx;
        const int by = (int)(lt % nty);
        const int slab = (int)(lt / nty);
        if (G.bwd_rays == 1) bwd_tile<BWD_UPDATE, SLAB, TX, TY, 1, 2, 1>(G, A, acc, bx, by, slab);
        else if (G.bwd_rays == 2) bwd_tile<BWD_UPDATE, SLAB, TX, TY, 1, 2, 2>(G, A, acc, bx, by, slab);
        else bwd_tile<BWD_UPDATE, SLAB, TX, TY, 1, 2, kRaysPerView>(G, A, acc, bx, by, slab);
    }
}

template <int SLAB, int VS, int STEP, int RAYS>
static cudaError_t launch_bwd(int mode, const Geo& G, const BwdArgs& A, cudaStream_t s) {
    constexpr int TX = BwdTile<VS>::X, TY = BwdTile<VS>::Y;
    const int blocks = ((G.nx + TX - 1) / TX) * ((G.ny + TY - 1) / TY) * ((G.nz + SLAB - 1) / SLAB);
    if (mode == BWD_UPDATE) bwd_kernel<BWD_UPDATE, SLAB, VS, STEP, RAYS><<<blocks, kBwdThreads, 0, s>>>(G, A);
    else if (mode == BWD_GRADIENT) bwd_kernel<BWD_GRADIENT, SLAB, VS, STEP, RAYS><<<blocks, kBwdThreads, 0, s>>>(G, A);
    else bwd_kernel<BWD_ADJOINT, SLAB, VS, STEP, RAYS><<<blocks, kBwdThreads, 0, s>>>(G, A);
    return cudaGetLastError();
}

template <int SLAB, int VS>
static cudaError_t launch_slab(int mode, const BwdPlan& P, const Geo& G, const BwdArgs& A, cudaStream_t s) {
    return P.view_step == 1 ? launch_bwd<SLAB, VS, 1, kRaysPerView>(mode, G, A, s)
           : P.rays == 1    ? launch_bwd<SLAB, VS, 2, 1>(mode, G, A, s)
           : P.rays == 2    ? launch_bwd<SLAB, VS, 2, 2>(mode, G, A, s)
                            : launch_bwd<SLAB, VS, 2, kRaysPerView>(mode, G, A, s);
}

cudaError_t launch_backward(int mode, const BwdPlan& P, const Geo& G, const BwdArgs& A, cudaStream_t s) {
#define DEAM_BWD(SL, VS) \
    if (P.slab == SL && P.vs == VS) return launch_slab<SL, VS>(mode, P, G, A, s);
    if (P.slab == 1) {
        if (P.flat) return P.vs == 8 ? launch_slice<2, 8, true>(mode, G, A, s) : launch_slice<1, 16, true>(mode, G, A, s);
        return P.vs == 8 ? launch_slice<2, 8, false>(mode, G, A, s) : launch_slice<1, 16, false>(mode, G, A, s);
    }
    DEAM_BWD(2, 1)
    DEAM_BWD(2, 2)
    DEAM_BWD(2, 4)
    DEAM_BWD(kMidSlab, 1)
    DEAM_BWD(kMidSlab, 2)
    DEAM_BWD(kMidSlab, 4)
    DEAM_BWD(kDeepSlab, 1)
    DEAM_BWD(kDeepSlab, 2)
    DEAM_BWD(kDeepSlab, 4)
#undef DEAM_BWD
    return cudaErrorInvalidValue;
}

long long backward_tiles(int shape, const Geo& G) {
    const int slab = kBwdShapes[shape][0], tx = kBwdShapes[shape][1], ty = kBwdShapes[shape][2];
    return (long long)((G.nx + tx - 1) / tx) * ((G.ny + ty - 1) / ty) * ((G.nz + slab - 1) / slab);
}


#define DEAM_BWD_BATCH_SHAPES(X) \
    X(0, 2, 16, 8) X(1, 2, 32, 4) X(2, 8, 16, 8) X(3, 8, 32, 4) X(4, 16, 16, 8) X(5, 16, 32, 4)

cudaError_t launch_backward_batch(int shape, const BatchDesc& B, int grid, cudaStream_t s) {
#define X(I, SL, TX, TY) \
    if (shape == I) {    \
        bwd_batch_kernel<SL, TX, TY><<<grid, TX * TY, 0, s>>>(B); \
        return cudaGetLastError(); \
    }
    DEAM_BWD_BATCH_SHAPES(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace deam
