// MAR initialisation (Sec. 2.2, Eq. 4): log sinograms, LI / NMAR completion of
// the metal trace, equiangular fan-beam / helical FDK-style filtered
// backprojection, the thresholded prior and the image-domain decomposition.
// These run once per scan, before the DEAM iterations; every step is a
// data-parallel kernel here (the prior's projection reuses the Joseph forward
// kernel).  Declarations and conventions: include/deam.h.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "deam.h"
#include "deam_ctx.h"
#include "deam_internal.h"
#include "deam_pair.cuh"

namespace {

int fail(int code, const std::string& m) { return deam::set_error(code, m.c_str()); }

const double kPi = 3.14159265358979323846;

#define CK(x)                                                                                  \
    do {                                                                                       \
        cudaError_t e_ = (x);                                                                  \
        if (e_ != cudaSuccess) {                                                               \
            ctx->failed = true;                                                                \
            return fail(e_ == cudaErrorMemoryAllocation ? DEAM_ERR_OOM : DEAM_ERR_CUDA,        \
                        std::string(#x) + ": " + cudaGetErrorString(e_));                      \
        }                                                                                      \
    } while (0)

#define CHECK_READY(ctx)                                                                   \
    do {                                                                                   \
        if (!(ctx)) return fail(DEAM_ERR_ARG, "null context");                             \
        if ((ctx)->failed) return fail(DEAM_ERR_STATE, "context failed earlier");          \
        if (!(ctx)->has_data) return fail(DEAM_ERR_STATE, "deam_set_data has not been called"); \
    } while (0)

struct DevGuard {
    int prev = -1;
    explicit DevGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DevGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// FBP constants (rounded once from double on the host).
struct FbpGeo {
    int nx, ny, nz, V, R, K;
    float x0, y0, z0, dx, dy, dz;  // voxel centres x0 + i dx (mm)
    float inv_da, kc, kmax;        // channel coordinate = gamma / a + kc, valid in [0, kmax]
    float sdd, inv_rp, rc;         // row coordinate = w / row_pitch + rc
    float dbeta;                   // 2 pi / views per rotation
};

// The ramp filter keeps a zero-padded row of both spectra in shared memory.
constexpr int kMaxFbpChannels = 3072;

int grid_for(long long n, int threads) {
    return (int)std::max<long long>(1, std::min<long long>((n + threads - 1) / threads, 152LL * 32));
}

// ---- kernels -----------------------------------------------------------------

// p_j(y) = ln(I0_j b(k) / max(d~_j(y), floor)), both spectra.
__global__ void log_kernel(const float* __restrict__ dt, const float* __restrict__ bowtie, float i0l, float i0h,
                           float floor_c, long long nrays, int K, float* __restrict__ p) {
    for (long long y = (long long)blockIdx.x * blockDim.x + threadIdx.x; y < nrays;
         y += (long long)gridDim.x * blockDim.x) {
        const float b = bowtie ? bowtie[y % K] : 1.f;
        const float dl = fmaxf(dt[y], floor_c), dh = fmaxf(dt[nrays + y], floor_c);
        p[y] = logf(__fdiv_rn(i0l * b, dl));
        p[nrays + y] = logf(__fdiv_rn(i0h * b, dh));
    }
}

// Linear interpolation across the trace along each (view, row); one block per
// row, the row's (normalised) values and trace flags staged in shared memory.
// In place (out == p) is safe: a thread writes only its own channels and reads
// neighbours from shared memory.
template <bool PRIOR>
__global__ void trace_kernel(const float* p, const float* __restrict__ prior, int pstride,
                             const uint8_t* __restrict__ mask, int bit, float eps, int K, long long nrows, float* out) {
    extern __shared__ float sm[];
    float* nv = sm;
    unsigned char* on = (unsigned char*)(sm + K);
    for (long long row = blockIdx.x; row < nrows; row += gridDim.x) {
        const long long base = row * K;
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            const float pk = p[base + k];
            on[k] = (mask[base + k] >> bit) & 1;
            nv[k] = PRIOR ? __fdiv_rn(pk, fmaxf(prior[(base + k) * pstride], eps)) : pk;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            if (!on[k]) {
                out[base + k] = p[base + k];
                continue;
            }
            int kl = k - 1, kr = k + 1;
            while (kl >= 0 && on[kl]) --kl;
            while (kr < K && on[kr]) ++kr;
            float val;
            if (kl >= 0 && kr < K)
                val = fmaf(nv[kr] - nv[kl], __fdiv_rn((float)(k - kl), (float)(kr - kl)), nv[kl]);
            else if (kl >= 0)
                val = nv[kl];
            else if (kr < K)
                val = nv[kr];
            else
                val = nv[k];
            out[base + k] = PRIOR ? val * fmaxf(prior[(base + k) * pstride], eps) : val;
        }
        __syncthreads();
    }
}

// One or two spectra at once: a float or a pair.
template <int NS>
struct Lane;
template <>
struct Lane<1> {
    typedef float T;
    static __device__ __forceinline__ T dup(float x) { return x; }
    static __device__ __forceinline__ T add(T a, T b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ T sub(T a, T b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ T mul(T a, float w) { return __fmul_rn(a, w); }
    static __device__ __forceinline__ T load(const float* p, long long, long long i) { return p[i]; }
    static __device__ __forceinline__ float at(T v, int) { return v; }
    static __device__ __forceinline__ void four(T (&to)[4], const T* from) {
        const float4 v = *(const float4*)from;
        to[0] = v.x;
        to[1] = v.y;
        to[2] = v.z;
        to[3] = v.w;
    }
};
template <>
struct Lane<2> {
    typedef deam::pair32 T;
    static __device__ __forceinline__ T dup(float x) { return deam::dup2(x); }
    static __device__ __forceinline__ T add(T a, T b) { return deam::add2(a, b); }
    static __device__ __forceinline__ T sub(T a, T b) { return deam::sub2(a, b); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return deam::fma2(a, b, c); }
    static __device__ __forceinline__ T mul(T a, float w) {
        const float2 v = deam::unpack2(a);
        return deam::pack2(__fmul_rn(v.x, w), __fmul_rn(v.y, w));
    }
    static __device__ __forceinline__ T load(const float* p, long long n, long long i) {
        return deam::pack2(p[i], p[n + i]);
    }
    static __device__ __forceinline__ float at(T v, int s) { return s ? deam::unpack2(v).y : deam::unpack2(v).x; }
    static __device__ __forceinline__ void four(T (&to)[4], const T* from) {
        const ulonglong2 a = ((const ulonglong2*)from)[0], b = ((const ulonglong2*)from)[1];
        to[0] = a.x;
        to[1] = a.y;
        to[2] = b.x;
        to[3] = b.y;
    }
};

// Equiangular ramp filtering of each (view, row): the pre-weighted row (fan
// weight SID cos(gamma_k), cone weight per row) between zero padding in shared
// memory, q(n) = sum_m ker(|m|) pw(n - m), ker(0) and the odd taps only (the
// even taps vanish), compensated FP32 sums (the taps cancel strongly).  In: NS
// sinograms [NS][nrays]; out: their values interleaved [nrays][NS].
//
// An even n takes odd channels only and an odd n even ones, so the row is kept as
// two arrays x[0][i] = pw(2 i + 1), x[1][i] = pw(2 i + 2), and both parities are
//   q(2 i + par) = ker(0) pw(2 i + par) + sum_j ker(2 j + 1) (x[par][i + j] + x[par][i - j - 1]).
// A thread computes four neighbouring i of one parity from two sliding windows of
// registers, four taps per pair of 16-byte loads: 5 operations and 0.5 shared
// words per tap and output, where one output per thread read three words (7.9 ms
// for two spectra of 55,680 rows x 672 channels, the shared-memory rate; 4.2 ms now,
// the FP32 pipe's packed rate bounding it at 2.5); taps beyond both ends of the row
// are left out.
template <int NS>
__global__ void __launch_bounds__(256) ramp_kernel(const float* p, long long nrays, const float* __restrict__ chanw,
                                                   const float* __restrict__ conew, const float* __restrict__ ker, int K,
                                                   int R, long long nrows, int per_block, float* out) {
    typedef Lane<NS> L;
    typedef typename L::T T;
    extern __shared__ __align__(16) unsigned char raw[];
    const int half = (K + 1) / 2;                // outputs of either parity (one less odd ones if K is odd)
    const int taps = (K / 2 + 3) / 4 * 4;        // odd taps 1, 3, ... < K, padded with zeros to fours
    const int pad = taps + 8, len = 2 * pad + (half + 3) / 4 * 4;
    T* kk = (T*)raw;                             // [taps] ker(2 j + 1)
    T* x = kk + taps;                            // [per_block][2][len], x[.][par][pad + i]
    const T zero = L::dup(0.f);
    for (int j = threadIdx.x; j < taps; j += blockDim.x) kk[j] = L::dup(2 * j + 1 < K ? ker[2 * j + 1] : 0.f);
    // the margins stay zero; the rows' values are replaced
    for (int i = threadIdx.x; i < per_block * 2 * len; i += blockDim.x) x[i] = zero;
    const float k0 = ker[0];
    const int quads = (half + 3) / 4;
    for (long long first = (long long)blockIdx.x * per_block; first < nrows; first += (long long)gridDim.x * per_block) {
        const int rows = (int)min((long long)per_block, nrows - first);
        __syncthreads();  // the previous rows' readers are done
        for (int row = 0; row < rows; ++row) {
            const long long ray = (first + row) * K;
            const float cw = conew[(first + row) % R];
            T* __restrict__ xr = x + row * 2 * len + pad;
            for (int c = threadIdx.x; c < K; c += blockDim.x)
                xr[(c & 1 ? 0 : len) + (c + 1) / 2 - 1] = L::mul(L::mul(L::load(p, nrays, ray + c), chanw[c]), cw);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < rows * 2 * quads; t += blockDim.x) {
            const int i0 = t % quads * 4, par = t / quads % 2, row = t / (2 * quads);
            const T* __restrict__ xr = x + (row * 2 + par) * len + pad + i0;
            T s[4], c[4], r[8], l[8];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                // pw(2 i + par): x[1][i - 1] for even, x[0][i] for odd outputs
                const T own = par ? x[(row * 2) * len + pad + i0 + a] : x[(row * 2 + 1) * len + pad + i0 + a - 1];
                s[a] = L::mul(own, k0);
                c[a] = zero;
            }
            // x[i0 + j .. i0 + j + 7] and x[i0 - j - 4 .. i0 - j + 3]
            T four[4];
            L::four(four, xr);
#pragma unroll
            for (int a = 0; a < 4; ++a) r[a] = l[4 + a] = four[a];
            // the last tap that reaches the row from either side
            const int end = min(taps, max(i0 + 4, half - i0) + 1);
#pragma unroll 1
            for (int j = 0; j < end; j += 4) {
                L::four(four, xr + j + 4);
#pragma unroll
                for (int a = 0; a < 4; ++a) r[4 + a] = four[a];
                L::four(four, xr - j - 4);
#pragma unroll
                for (int a = 0; a < 4; ++a) l[a] = four[a];
                T k[4];
                L::four(k, kk + j);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj)
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const T y = L::fma(k[jj], L::add(l[3 - jj + a], r[jj + a]), c[a]);
                        const T u = L::add(s[a], y);
                        c[a] = L::sub(y, L::sub(u, s[a]));
                        s[a] = u;
                    }
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    r[a] = r[4 + a];
                    l[4 + a] = l[a];
                }
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int n = 2 * (i0 + a) + par;
                if (n < K) ((T*)out)[(first + row) * K + n] = s[a];
            }
        }
    }
}

// Voxel-driven FBP backprojection of NS filtered sinograms q [nrays][NS]: a thread
// takes NZ neighbouring slices of one (ix, iy) column, a block row per iy, so that
// a slice's view window is uniform in the block; weight 1/L^2, bilinear in (row,
// channel), compensated FP32 sums.  What a view and a column have in common (the
// fan angle, its channel, the distance) is computed once for the slices whose
// windows hold the view: 3.4 ms at 256^2 x 32 x 1160 views and two spectra with two
// slices per thread, 4.0 ms with one, 4.3 ms with four (too few warps) and with one
// slice and scalar loads of planar sinograms.  Threads of one slice (small volumes,
// single slices) need no look at the window, detectors of one row (ROWS false) no
// height: 0.80 -> 0.67 ms at 512^2 x 720 views, 0.58 -> 0.39 at 64^2 x 16.
template <int NS, int NZ, bool ROWS>
__global__ void fbp_kernel(const float* __restrict__ q, const float4* __restrict__ vw, const float* __restrict__ vz,
                           const int2* __restrict__ win, const FbpGeo F, float* __restrict__ img) {
    typedef Lane<NS> L;
    typedef typename L::T T;
    const int ix = blockIdx.x * blockDim.x + threadIdx.x, iy = blockIdx.y, iz0 = blockIdx.z * NZ;
    if (ix >= F.nx) return;
    const T* __restrict__ qt = (const T*)q;
    const float X = fmaf((float)ix, F.dx, F.x0), Y = fmaf((float)iy, F.dy, F.y0);
    int2 w[NZ];
    float Z[NZ];
    T acc[NZ], cmp[NZ];
    int v0 = F.V, v1 = 0;
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
        w[z] = iz0 + z < F.nz ? win[iz0 + z] : make_int2(0, 0);
        Z[z] = fmaf((float)(iz0 + z), F.dz, F.z0);
        acc[z] = cmp[z] = L::dup(0.f);
        if (w[z].x < w[z].y) {
            v0 = min(v0, w[z].x);
            v1 = max(v1, w[z].y);
        }
    }
    for (int v = v0; v < v1; ++v) {
        const float4 sv = __ldg(&vw[v]);  // (s_x, s_y, cos beta, sin beta)
        const float ddx = X - sv.x, ddy = Y - sv.y;
        const float L2 = fmaf(ddx, ddx, ddy * ddy);
        // fan angle of the voxel: signed angle from the central ray -(cos, sin)
        const float dot = -fmaf(ddx, sv.z, ddy * sv.w);
        const float crs = fmaf(ddx, sv.w, -ddy * sv.z);
        const float kf = fmaf(atan2f(crs, dot), F.inv_da, F.kc);
        if (!(kf >= 0.f && kf <= F.kmax)) continue;
        const int k0 = min((int)kf, F.K - 2);
        const float ak = kf - (float)k0;
        const T ak2 = L::dup(ak);
        const float dist = ROWS ? sqrtf(L2) : 0.f;
        const float inv = __frcp_rn(L2);
        const float sz = ROWS ? __ldg(&vz[v]) : 0.f;
        const long long ev = (long long)v * F.R * F.K + k0;
#pragma unroll
        for (int z = 0; z < NZ; ++z) {
            if (NZ > 1 && (v < w[z].x || v >= w[z].y)) continue;
            long long e = ev;
            T val;
            if (ROWS) {
                const float wd = __fdiv_rn((Z[z] - sz) * F.sdd, dist);
                const float rf = fminf(fmaxf(fmaf(wd, F.inv_rp, F.rc), 0.f), (float)(F.R - 1));
                const int r0 = min((int)rf, F.R - 2);
                e += (long long)r0 * F.K;
                const T lo = __ldg(&qt[e]), hi = __ldg(&qt[e + F.K]);
                val = L::fma(ak2, L::sub(__ldg(&qt[e + 1]), lo), lo);
                const T up = L::fma(ak2, L::sub(__ldg(&qt[e + F.K + 1]), hi), hi);
                val = L::fma(L::dup(rf - (float)r0), L::sub(up, val), val);
            } else {
                const T lo = __ldg(&qt[e]);
                val = L::fma(ak2, L::sub(__ldg(&qt[e + 1]), lo), lo);
            }
            const T y = L::fma(val, L::dup(inv), L::sub(L::dup(0.f), cmp[z]));
            const T u = L::add(acc[z], y);
            cmp[z] = L::sub(L::sub(u, acc[z]), y);
            acc[z] = u;
        }
    }
    const long long nvox = (long long)F.nx * F.ny * F.nz;
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
        if (iz0 + z >= F.nz) break;
        const long long vi = ((long long)(iz0 + z) * F.ny + iy) * F.nx + ix;
#pragma unroll
        for (int s = 0; s < NS; ++s) img[s * nvox + vi] = L::at(acc[z], s) * F.dbeta;
    }
}

// One pass of the in-plane [1,2,1]/4 x [1,2,1]/4 smoothing (edges replicated).
__global__ void smooth_kernel(const float* __restrict__ f, int nx, int ny, long long n, float* __restrict__ out) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(i % nx), iy = (int)((i / nx) % ny);
        const long long base = i - ix - (long long)iy * nx;
        float acc = 0.f;
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            const int y = min(max(iy + b, 0), ny - 1);
            const float wy = b == 0 ? 0.5f : 0.25f;
#pragma unroll
            for (int a = -1; a <= 1; ++a) {
                const int x = min(max(ix + a, 0), nx - 1);
                const float wx = a == 0 ? 0.5f : 0.25f;
                acc = fmaf(wx * wy, f[base + (long long)y * nx + x], acc);
            }
        }
        out[i] = acc;
    }
}

__global__ void prior_kernel(const float* __restrict__ f, long long n, float t_air, float t_bone, float soft,
                             float* __restrict__ prior) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float x = f[i];
        prior[i] = x < t_air ? 0.f : (x < t_bone ? soft : x);
    }
}

// Eq. (4): (c_1, c_2) = M^-1 (mu_L, mu_H), M^-1 rounded once from double.
__global__ void decompose_kernel(const float* __restrict__ mu, long long n, float a, float b, float c, float d,
                                 float2* __restrict__ out) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float l = mu[i], h = mu[n + i];
        out[i] = make_float2(fmaf(a, l, b * h), fmaf(c, l, d * h));
    }
}

// ---- host helpers ------------------------------------------------------------

// prior (nullable): the prior's projection, element y at prior[y * pstride].
int complete(deam_ctx* ctx, const float* p, const float* prior, int pstride, int bit, float eps, float* out,
             cudaStream_t s) {
    const deam_geometry& g = ctx->geo;
    const long long nrows = (long long)g.n_views * g.n_rows;
    const int K = g.n_channels;
    if (!ctx->mask_set) {  // no trace: a copy
        if (out != p) CK(cudaMemcpyAsync(out, p, sizeof(float) * ctx->nrays, cudaMemcpyDeviceToDevice, s));
        return DEAM_OK;
    }
    const size_t sm = sizeof(float) * K + K;
    const int blocks = (int)std::min<long long>(nrows, 152LL * 16);
    if (prior)
        trace_kernel<true><<<blocks, 256, sm, s>>>(p, prior, pstride, ctx->mask, bit, eps, K, nrows, out);
    else
        trace_kernel<false><<<blocks, 256, sm, s>>>(p, nullptr, 1, ctx->mask, bit, eps, K, nrows, out);
    CK(cudaGetLastError());
    return DEAM_OK;
}

// Bytes of shared memory of ramp_kernel: the taps, and each row of K channels.
struct RampShared {
    size_t taps, row;
};
RampShared ramp_shared(int K, int ns) {
    const size_t cell = sizeof(float) * ns;
    const int half = (K + 1) / 2, taps = (K / 2 + 3) / 4 * 4, len = 2 * (taps + 8) + (half + 3) / 4 * 4;
    return {taps * cell, 2 * (size_t)len * cell};
}

template <int NS>
cudaError_t filter(deam_ctx* ctx, const float* p, const float* chanw, const float* conew, const float* ker, float* q,
                   cudaStream_t s) {
    const int K = ctx->geo.n_channels, R = ctx->geo.n_rows;
    const long long nrows = (long long)ctx->geo.n_views * R;
    const RampShared m = ramp_shared(K, NS);
    // rows per block: outputs (in fours) for half as many threads again, as far as
    // 48 KB hold their rows, so that the threads with short windows take a second one
    // (two rows of 672 channels; one row, 0.3 to 0.7 ms slower of 15.5 for the whole
    // initialisation); a long row may need more, by opt-in (3072 channels of two
    // spectra: 86 KB).  Few rows are spread over four blocks per SM first (360 rows of
    // 256 channels: 16 us six to a block, 10 us one)
    const int fours = 2 * (((K + 1) / 2 + 3) / 4);
    const size_t room = 48 * 1024 > m.taps + m.row ? 48 * 1024 - m.taps : m.row;
    const long long spread = std::max(1LL, nrows / (152 * 4));
    const int per = (int)std::min<size_t>(std::min<long long>(std::max(1, 384 / fours), spread), room / m.row);
    const size_t sm = m.taps + per * m.row;
    if (sm > 48 * 1024) {
        // the limit is the kernel's, not this call's: always the longest row's, so that
        // calls of several threads do not lower it for one another
        const RampShared most = ramp_shared(kMaxFbpChannels, NS);
        const cudaError_t e = cudaFuncSetAttribute(ramp_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(most.taps + most.row));
        if (e != cudaSuccess) return e;
    }
    const int blocks = (int)std::min<long long>((nrows + per - 1) / per, 1LL << 20);
    ramp_kernel<NS><<<blocks, 256, sm, s>>>(p, ctx->nrays, chanw, conew, ker, K, R, nrows, per, q);
    return cudaGetLastError();
}

// FBP of n sinograms p [n][V][R][K] into img [n][nz][ny][nx]; q is scratch of
// the same size as p (n = 1: may equal p when p may be overwritten).
int fbp(deam_ctx* ctx, const float* p, int n, float* q, float* img, cudaStream_t s) {
    const deam_geometry& g = ctx->geo;
    const int K = g.n_channels, R = g.n_rows, V = g.n_views, N = g.views_per_rotation;
    // host tables in double, rounded once
    std::vector<float> ker(K), chanw(K), conew(R), vz(V);
    std::vector<float4> vw(V);
    std::vector<int2> win(g.nz);
    const double a = g.channel_pitch;
    for (int m = 0; m < K; ++m) {
        double v;
        if (m == 0) v = 1.0 / (8.0 * a * a);
        else if (m % 2 == 0) v = 0.0;
        else {
            const double sn = sin(m * a);
            v = -1.0 / (2.0 * kPi * kPi * sn * sn);
        }
        ker[m] = (float)(a * v);
    }
    for (int k = 0; k < K; ++k)
        chanw[k] = (float)(g.sid * cos((k - (K - 1) / 2.0 + g.channel_offset) * a));
    for (int r = 0; r < R; ++r) {
        const double w = (r - (R - 1) / 2.0 + g.row_offset) * g.row_pitch;
        conew[r] = (float)(g.sdd / sqrt(g.sdd * g.sdd + w * w));
    }
    for (int v = 0; v < V; ++v) {
        const double beta = g.start_angle + 2.0 * kPi * v / N;
        vw[v] = make_float4((float)(g.sid * cos(beta)), (float)(g.sid * sin(beta)), (float)cos(beta),
                            (float)sin(beta));
        vz[v] = (float)(g.z_start + g.feed * (double)v / N);
    }
    const double Z0 = g.cz - (g.nz - 1) / 2.0 * g.dz;
    for (int iz = 0; iz < g.nz; ++iz) {
        long lo = 0, hi = V < N ? V : N;
        if (g.feed != 0.0 && R > 1) {
            const double vc = (Z0 + iz * g.dz - g.z_start) * (double)N / g.feed;
            lo = (long)ceil(vc - N / 2.0);
            hi = lo + N;
        }
        lo = std::max<long>(lo, 0);
        hi = std::min<long>(hi, V);
        win[iz] = make_int2((int)lo, (int)std::max(lo, hi));
    }
    FbpGeo F;
    F.nx = g.nx; F.ny = g.ny; F.nz = g.nz; F.V = V; F.R = R; F.K = K;
    F.x0 = (float)(g.cx - (g.nx - 1) / 2.0 * g.dx);
    F.y0 = (float)(g.cy - (g.ny - 1) / 2.0 * g.dy);
    F.z0 = (float)Z0;
    F.dx = (float)g.dx; F.dy = (float)g.dy; F.dz = (float)g.dz;
    F.inv_da = (float)(1.0 / a);
    F.kc = (float)((K - 1) / 2.0 - g.channel_offset);
    F.kmax = (float)(K - 1);
    F.sdd = (float)g.sdd;
    F.inv_rp = (float)(1.0 / g.row_pitch);
    F.rc = (float)((R - 1) / 2.0 - g.row_offset);
    F.dbeta = (float)(2.0 * kPi / N);

    // one scratch block for the tables
    const size_t off_ker = 0, off_chw = off_ker + K, off_cone = off_chw + K, off_vz = off_cone + R;
    const size_t nfl = off_vz + V;
    const size_t bytes_fl = ((nfl * sizeof(float) + 15) / 16) * 16;
    const size_t bytes = bytes_fl + sizeof(float4) * V + sizeof(int2) * g.nz;
    char* tab = nullptr;
    CK(cudaMallocAsync((void**)&tab, bytes, s));
    std::vector<char> host(bytes);
    memcpy(host.data() + off_ker * 4, ker.data(), 4 * K);
    memcpy(host.data() + off_chw * 4, chanw.data(), 4 * K);
    memcpy(host.data() + off_cone * 4, conew.data(), 4 * R);
    memcpy(host.data() + off_vz * 4, vz.data(), 4 * V);
    memcpy(host.data() + bytes_fl, vw.data(), sizeof(float4) * V);
    memcpy(host.data() + bytes_fl + sizeof(float4) * V, win.data(), sizeof(int2) * g.nz);
    cudaError_t e = cudaMemcpyAsync(tab, host.data(), bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host staging buffer goes out of scope
    const float* d_ker = (const float*)tab + off_ker;
    const float* d_chw = (const float*)tab + off_chw;
    const float* d_cone = (const float*)tab + off_cone;
    const float* d_vz = (const float*)tab + off_vz;
    const float4* d_vw = (const float4*)(tab + bytes_fl);
    const int2* d_win = (const int2*)(tab + bytes_fl + sizeof(float4) * V);
    if (e == cudaSuccess)
        e = n == 2 ? filter<2>(ctx, p, d_chw, d_cone, d_ker, q, s) : filter<1>(ctx, p, d_chw, d_cone, d_ker, q, s);
    if (e == cudaSuccess) {
        // two slices per thread where that leaves 16 warps per SM with views to add
        // (slices' windows, in rotations: 128^2 x 24 voxels, a rotation past 13 slices,
        // 3277 warps 0.15 ms against 0.16 with one; 96^2 x 96, as far, 1843 warps 0.29 against
        // 0.25; 128^2 x 8 1365 warps 0.28 against 0.20)
        double seen = 0.0;
        for (const int2& w : win) seen += w.y - w.x;
        const double warps = (g.nx + 31) / 32 * (double)g.ny * seen / std::min(V, N) / 2.0;
        auto run = [&](auto rows) {
            const bool two = g.nz > 1 && warps >= 152.0 * 16.0;
            const dim3 grid((g.nx + 127) / 128, g.ny, two ? (g.nz + 1) / 2 : g.nz);
            constexpr bool ROWS = decltype(rows)::value;
            if (n == 2 && two) fbp_kernel<2, 2, ROWS><<<grid, 128, 0, s>>>(q, d_vw, d_vz, d_win, F, img);
            else if (n == 2) fbp_kernel<2, 1, ROWS><<<grid, 128, 0, s>>>(q, d_vw, d_vz, d_win, F, img);
            else if (two) fbp_kernel<1, 2, ROWS><<<grid, 128, 0, s>>>(q, d_vw, d_vz, d_win, F, img);
            else fbp_kernel<1, 1, ROWS><<<grid, 128, 0, s>>>(q, d_vw, d_vz, d_win, F, img);
        };
        if (R > 1) run(std::true_type{});
        else run(std::false_type{});
        e = cudaGetLastError();
    }
    cudaError_t e2 = cudaFreeAsync(tab, s);
    CK(e);
    CK(e2);
    return DEAM_OK;
}

bool is_dev(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" {

int deam_log_sinogram(deam_ctx* ctx, double count_floor, float* p, void* stream) {
    CHECK_READY(ctx);
    if (!p || !is_dev(p)) return fail(DEAM_ERR_ARG, "p must be a device pointer");
    if (!(isfinite(count_floor) && count_floor > 0.0)) return fail(DEAM_ERR_ARG, "count_floor must be > 0");
    DevGuard dg(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    log_kernel<<<grid_for(ctx->nrays, 256), 256, 0, s>>>(ctx->dt, ctx->bowtie, (float)ctx->i0tot[0],
                                                         (float)ctx->i0tot[1], (float)count_floor, ctx->nrays,
                                                         ctx->geo.n_channels, p);
    CK(cudaGetLastError());
    return DEAM_OK;
}

int deam_complete_trace(deam_ctx* ctx, const float* p, const float* prior_proj, int spectrum, double eps, float* out,
                        void* stream) {
    CHECK_READY(ctx);
    if (!p || !out || !is_dev(p) || !is_dev(out)) return fail(DEAM_ERR_ARG, "p and out must be device pointers");
    if (prior_proj && !is_dev(prior_proj)) return fail(DEAM_ERR_ARG, "prior_proj must be a device pointer");
    if (spectrum != 0 && spectrum != 1) return fail(DEAM_ERR_ARG, "spectrum must be 0 (L) or 1 (H)");
    if (!(isfinite(eps) && eps > 0.0)) return fail(DEAM_ERR_ARG, "eps must be > 0");
    DevGuard dg(ctx->device);
    return complete(ctx, p, prior_proj, 1, spectrum, (float)eps, out, (cudaStream_t)stream);
}

int deam_fbp(deam_ctx* ctx, const float* p, int n, float* img, void* stream) {
    CHECK_READY(ctx);
    if (n != 1 && n != 2) return fail(DEAM_ERR_ARG, "n must be 1 or 2");
    if (!p || !img || !is_dev(p) || !is_dev(img)) return fail(DEAM_ERR_ARG, "p and img must be device pointers");
    if (ctx->geo.n_channels < 2 || ctx->geo.n_channels > kMaxFbpChannels)
        return fail(DEAM_ERR_ARG, "FBP needs 2 to 3072 channels (the ramp filter stages a row in shared memory)");
    DevGuard dg(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    float* q = nullptr;
    CK(cudaMallocAsync((void**)&q, sizeof(float) * ctx->nrays * n, s));
    const int rc = fbp(ctx, p, n, q, img, s);
    cudaFreeAsync(q, s);
    return rc;
}

int deam_mar_init(deam_ctx* ctx, const deam_mar_params* P, const float* prior_in, float* c, float* prior_out,
                  float* mu_out, void* stream) {
    CHECK_READY(ctx);
    if (!P || !c || !is_dev(c)) return fail(DEAM_ERR_ARG, "params and a device c are required");
    if ((prior_in && !is_dev(prior_in)) || (prior_out && !is_dev(prior_out)) || (mu_out && !is_dev(mu_out)))
        return fail(DEAM_ERR_ARG, "prior_in, prior_out and mu_out must be device pointers (or NULL)");
    for (double x : {P->calib[0], P->calib[1], P->calib[2], P->calib[3], P->t_air, P->t_bone, P->soft_value})
        if (!isfinite(x)) return fail(DEAM_ERR_ARG, "MAR parameters must be finite");
    const double det = P->calib[0] * P->calib[3] - P->calib[1] * P->calib[2];
    const double scale = std::max(std::fabs(P->calib[0] * P->calib[3]), std::fabs(P->calib[1] * P->calib[2]));
    if (!(std::fabs(det) > 1e-12 * scale)) return fail(DEAM_ERR_ARG, "calibration matrix is singular");
    if (!(isfinite(P->count_floor) && P->count_floor > 0.0)) return fail(DEAM_ERR_ARG, "count_floor must be > 0");
    if (!(isfinite(P->eps) && P->eps > 0.0)) return fail(DEAM_ERR_ARG, "eps must be > 0");
    if (P->prior_spectrum != 0 && P->prior_spectrum != 1) return fail(DEAM_ERR_ARG, "prior_spectrum must be 0 or 1");
    if (P->prior_smooth < 0 || P->prior_smooth > 16) return fail(DEAM_ERR_ARG, "prior_smooth must be 0..16");
    if (ctx->geo.n_channels < 2 || ctx->geo.n_channels > kMaxFbpChannels)
        return fail(DEAM_ERR_ARG, "FBP needs 2 to 3072 channels (the ramp filter stages a row in shared memory)");
    DevGuard dg(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    const long long nr = ctx->nrays, nv = ctx->nvox;
    float *p = nullptr, *t = nullptr, *img = nullptr;
    float2* l = nullptr;
    // p: both sinograms, then the filtered ones; t: completed sinograms;
    // img: f | prior | mu_L | mu_H | smoothing scratch
    CK(cudaMallocAsync((void**)&p, sizeof(float) * 2 * nr, s));
    cudaError_t e = cudaMallocAsync((void**)&t, sizeof(float) * 2 * nr, s);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&img, sizeof(float) * 5 * nv, s);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&l, sizeof(float2) * nr, s);
    auto release = [&]() {
        if (p) cudaFreeAsync(p, s);
        if (t) cudaFreeAsync(t, s);
        if (img) cudaFreeAsync(img, s);
        if (l) cudaFreeAsync(l, s);
    };
    auto run = [&]() -> int {
        CK(e);
        float* f = img;
        float* prior = img + nv;
        float* mu = img + 2 * nv;
        log_kernel<<<grid_for(nr, 256), 256, 0, s>>>(ctx->dt, ctx->bowtie, (float)ctx->i0tot[0],
                                                     (float)ctx->i0tot[1], (float)P->count_floor, nr,
                                                     ctx->geo.n_channels, p);
        CK(cudaGetLastError());
        if (prior_in) {
            CK(cudaMemcpyAsync(prior, prior_in, sizeof(float) * nv, cudaMemcpyDeviceToDevice, s));
        } else {
            // single-energy FBP of the chosen spectrum with the trace linearly
            // interpolated, thresholded into the prior
            const int j = P->prior_spectrum;
            int rc = complete(ctx, p + (size_t)j * nr, nullptr, 1, j, (float)P->eps, t, s);
            if (rc != DEAM_OK) return rc;
            rc = fbp(ctx, t, 1, t, f, s);
            if (rc != DEAM_OK) return rc;
            // filtering: passes ping-pong between f and the scratch image
            float* a = f;
            float* b = img + 4 * nv;  // smoothing scratch
            for (int pass = 0; pass < P->prior_smooth; ++pass) {
                smooth_kernel<<<grid_for(nv, 256), 256, 0, s>>>(a, ctx->geo.nx, ctx->geo.ny, nv, b);
                CK(cudaGetLastError());
                std::swap(a, b);
            }
            prior_kernel<<<grid_for(nv, 256), 256, 0, s>>>(a, nv, (float)P->t_air, (float)P->t_bone,
                                                           (float)P->soft_value, prior);
            CK(cudaGetLastError());
        }
        // the prior's projection: Joseph forward projection of (prior, 0) into
        // l (float2 per ray; NMAR reads its first component).  Only the rays in or
        // next to a trace are projected, the others stay unset and have no use
        // (256^2 x 32, 37.4 M rays, two rods: 7.2 ms for all of them, 1.7 for these)
        if (ctx->mask_set) {
            const int rc = deam::build_layouts(ctx, nullptr, prior, 0, s);
            if (rc != DEAM_OK) return rc;
            deam::FwdArgs A = deam::fwd_args(ctx);
            A.l_out = l;
            A.mask = ctx->mask;
            CK(deam::launch_forward(deam::FWD_LINE, ctx->G, ctx->S, A, ctx->n_fwd_blocks, s));
        }
        for (int j = 0; j < 2; ++j) {
            const int rc = complete(ctx, p + (size_t)j * nr, (const float*)l, 2, j, (float)P->eps, t + (size_t)j * nr, s);
            if (rc != DEAM_OK) return rc;
        }
        const int rc = fbp(ctx, t, 2, p, mu, s);  // both spectra (the sinograms p are done with)
        if (rc != DEAM_OK) return rc;
        const double ia = P->calib[3] / det, ib = -P->calib[1] / det, ic = -P->calib[2] / det, id = P->calib[0] / det;
        decompose_kernel<<<grid_for(nv, 256), 256, 0, s>>>(mu, nv, (float)ia, (float)ib, (float)ic, (float)id,
                                                           (float2*)c);
        CK(cudaGetLastError());
        if (prior_out) CK(cudaMemcpyAsync(prior_out, prior, sizeof(float) * nv, cudaMemcpyDeviceToDevice, s));
        if (mu_out) CK(cudaMemcpyAsync(mu_out, mu, sizeof(float) * 2 * nv, cudaMemcpyDeviceToDevice, s));
        return DEAM_OK;
    };
    int rc = run();
    release();
    return rc;
}

}  // extern "C"
