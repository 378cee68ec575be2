// Device helpers of the per-ray spectral epilogue (Eq. 8 energy sums and the
// Eq. 5 I-divergence term) and block reductions, shared by the kernels that
// compute them.
#pragma once

#include <math.h>

#include "deam_internal.h"

namespace deam {

// ex2.approx: the SFU's 2^x (documented max relative error 2^-22); the tables
// carry mu * log2(e) so that exp(-mu.l) = 2^(-mu'.l).
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Kahan/Neumaier-style compensated accumulation of a block partial.
__device__ __forceinline__ void kahan_add(float& sum, float& comp, float x) {
    const float y = x - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// (1 + u) ln(1 + u) - u, the I-divergence term d ln(d/g) - d + g divided by g
// with u = (d - g) / g.  For |u| < 1/4 the Taylor series
// sum_{n>=2} (-1)^n u^n / (n (n-1)) through u^12 (the first dropped term is
// below 3e-9 of the sum) avoids the cancellation of the closed form.  Beyond,
// the closed form with one rounding for (1 + u) ln(1 + u) - u (an FMA): the
// cancellation there amplifies log1pf's error by at most (1+u) ln(1+u) / phi,
// about 10 at |u| = 1/4 and falling with |u|, so each term is within ~2e-6
// (relative) of its exact value; the terms are summed in FP64.
__device__ __forceinline__ float idiv_phi(float u) {
    if (u <= -1.f) return 1.f;  // d = 0: the term is g
    if (fabsf(u) < 0.25f) {
        float s = 1.f / 132.f;
        s = fmaf(s, u, -1.f / 110.f);
        s = fmaf(s, u, 1.f / 90.f);
        s = fmaf(s, u, -1.f / 72.f);
        s = fmaf(s, u, 1.f / 56.f);
        s = fmaf(s, u, -1.f / 42.f);
        s = fmaf(s, u, 1.f / 30.f);
        s = fmaf(s, u, -1.f / 20.f);
        s = fmaf(s, u, 1.f / 12.f);
        s = fmaf(s, u, -1.f / 6.f);
        s = fmaf(s, u, 0.5f);
        return s * u * u;
    }
    return fmaf(1.f + u, log1pf(u), -u);
}

// Sum (or max) over a block of NT threads in a fixed order: warp shuffles,
// then thread 0 combines the warp results in warp order.
template <int NT, typename T>
__device__ __forceinline__ T block_reduce(T v, bool is_max) {
    __shared__ T red[NT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const T w = __shfl_down_sync(0xffffffffu, v, o);
        v = is_max ? (w > v ? w : v) : v + w;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        v = red[0];
        for (int i = 1; i < NT / 32; ++i) v = is_max ? (red[i] > v ? red[i] : v) : v + red[i];
    }
    return v;
}

// The six sums of one ray over the energy bins: g_j = sum_E I0_j q~ and S_ij =
// sum_E mu_i I0_j q~ (j = L, H), q~ = 2^(-mu'.l).
struct RaySums {
    float gl, gh, s1l, s2l, s1h, s2h;
};

template <bool NEED_S>
__device__ __forceinline__ void add_bin(RaySums& p, float ex, float mu1, float mu2, float i0l, float i0h) {
    p.gl = fmaf(i0l, ex, p.gl);
    p.gh = fmaf(i0h, ex, p.gh);
    if (NEED_S) {
        const float ql = __fmul_rn(i0l, ex), qh = __fmul_rn(i0h, ex);
        p.s1l = fmaf(mu1, ql, p.s1l);
        p.s2l = fmaf(mu2, ql, p.s2l);
        p.s1h = fmaf(mu1, qh, p.s1h);
        p.s2h = fmaf(mu2, qh, p.s2h);
    }
}

template <bool NEED_S>
__device__ __forceinline__ void kahan_add(RaySums& s, RaySums& c, const RaySums& p) {
    kahan_add(s.gl, c.gl, p.gl);
    kahan_add(s.gh, c.gh, p.gh);
    if (NEED_S) {
        kahan_add(s.s1l, c.s1l, p.s1l);
        kahan_add(s.s2l, c.s2l, p.s2l);
        kahan_add(s.s1h, c.s1h, p.s1h);
        kahan_add(s.s2h, c.s2h, p.s2h);
    }
}

// Spectral tables in shared memory, as the sums over many rays read them: active
// bin e at a[e] = (mu_1', mu_2', mu_1, mu_2), b[e] = (I0_L, I0_H).
struct SpecTable {
    float4 a[kMaxE];
    float2 b[kMaxE];
};
__device__ __forceinline__ void fill_table(SpecTable& T, const Spec& S) {
    for (int e = S.e_lo + threadIdx.x; e < S.e_hi; e += blockDim.x) {
        T.a[e - S.e_lo] = make_float4(S.mu1l2[e], S.mu2l2[e], S.mu1[e], S.mu2[e]);
        T.b[e - S.e_lo] = make_float2(S.i0l[e], S.i0h[e]);
    }
}

// Spectral sums of N rays for both spectra (bowtie applied by the caller).  Bins
// are summed in blocks of 8 in FP32, block partials are added with compensation.
// COMP = false: plain FP32 sums, bin after bin (the uncompensated variant).
// bin(e) gives the table entry of active bin e of n.
template <bool NEED_S, bool COMP, int N, typename Bin>
__device__ __forceinline__ void spectral_sums(int n, const float (&l1)[N], const float (&l2)[N], RaySums (&s)[N], Bin bin) {
    RaySums c[N], p[N];
#pragma unroll
    for (int i = 0; i < N; ++i) s[i] = c[i] = RaySums{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto one = [&](int e, RaySums(&to)[N]) {
        float4 a;
        float2 b;
        bin(e, a, b);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float ex = ex2_approx(-fmaf(a.x, l1[i], a.y * l2[i]));
            add_bin<NEED_S>(to[i], ex, a.z, a.w, b.x, b.y);
        }
    };
    if constexpr (!COMP) {
        for (int e = 0; e < n; ++e) one(e, s);
    } else {
        for (int e0 = 0; e0 < n; e0 += 8) {
#pragma unroll
            for (int i = 0; i < N; ++i) p[i] = RaySums{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (e0 + j < n) one(e0 + j, p);
#pragma unroll
            for (int i = 0; i < N; ++i) kahan_add<NEED_S>(s[i], c[i], p[i]);
        }
    }
}

// One ray, the tables read from the kernel's parameters.
template <bool NEED_S, bool COMP = true>
__device__ __forceinline__ RaySums spectral_sums(const Spec& S, float l1, float l2) {
    const float a[1] = {l1}, b[1] = {l2};
    RaySums s[1];
    spectral_sums<NEED_S, COMP, 1>(S.e_hi - S.e_lo, a, b, s, [&](int e, float4& x, float2& y) {
        const int i = S.e_lo + e;
        x = make_float4(S.mu1l2[i], S.mu2l2[i], S.mu1[i], S.mu2[i]);
        y = make_float2(S.i0l[i], S.i0h[i]);
    });
    return s[0];
}

}  // namespace deam
