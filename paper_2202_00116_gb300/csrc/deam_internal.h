// Internal declarations shared by the kernels (deam_kernels.cu) and the C ABI
// (deam_api.cu) of the sm_103a MAR-DEAM library.  Not installed.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "deam.h"

namespace deam {

constexpr int kMaxE = 256;        // energy bins carried in the kernel-parameter tables
constexpr int kFwdThreads = 256;  // threads per forward block

// Geometry in voxel-index units, as read by both projector directions.  Every
// per-ray quantity is derived from these tables by ray_inplane()/row terms with
// explicitly rounded FP32 operations, so the forward and the gather-backward
// kernels compute bit-identical sample positions and weights.
struct Geo {
    int nx, ny, nz, V, R, K;
    int fwd_rows;            // rows a forward thread projects at once (forward_rows; host)
    int fwd_narrow;          // forward blocks of four warps (forward_narrow; host)
    int bwd_rays;            // rays of a view that a turn of the batched backprojection takes (turn_rays)
    float dx, dy;            // voxel edge lengths (mm)
    float dx_sdd, dy_sdd;    // dx / sdd, dy / sdd
    float dx_dy, dy_dx;      // dx / dy, dy / dx
    const float4* view4;     // [V] (sigma_x, sigma_y, cos beta, sin beta); sigma = source in index units
    const float* view_z;     // [V] sigma_z = (s_z - Z0) / dz
    const float2* chan;      // [K] (cos gamma_k, sin gamma_k)
    const float2* row;       // [R] (w_r / dz, sqrt(1 + (w_r/sdd)^2)): .y is the row length factor
    const float4* ip4;       // [V][K] (aq, bq, tau0, kappa) of ray_inplane, built once by build_inplane_table
    const float* ipL;        // [V][K] Lxy, negated for y-dominant rays
    float omega0, domega;    // omega_r = omega0 + r domega (row_omega)
    float chan_c0, inv_dgamma;  // channel coordinate = gamma / dgamma + chan_c0
    float vox_reach_mm;      // max(dx, dy): reach of a voxel's bilinear footprint in-plane
    float inv_sdd;           // 1 / sdd: in-plane distance from the source -> ray parameter t
    unsigned int* fault;     // [2] bounds-checked builds: first failing site and index (else unused)
};

// Bounds-checked builds (-DDEAM_BOUNDS_CHECK): every guarded access tests its
// index first; a failing test records (site, index) in the context's fault
// words -- the first one only -- and the access is skipped, so the kernel
// finishes and the entry point reports DEAM_ERR_ARG on return.  Never traps.
enum BoundsSite : unsigned {
    SITE_FWD_LAYOUT = 1,   // forward: paired-layout gather
    SITE_FWD_RAY = 2,      // forward: per-ray data (d~, mask, payload, outputs)
    SITE_BWD_RAY = 3,      // backprojection: ray data / payload gather
    SITE_BWD_TABLE = 4,    // backprojection: in-plane ray table
    SITE_BWD_IMAGE = 5,    // backprojection: image / sums
    SITE_INJECTED = 99     // written from the host by deam_bounds_inject
};
#ifdef DEAM_BOUNDS_CHECK
__device__ __forceinline__ bool in_bounds(unsigned int* fault, bool ok, unsigned site, long long idx) {
    if (!ok && fault && atomicCAS(fault, 0u, site) == 0u) fault[1] = (unsigned)(idx < 0 ? 0xffffffffu : idx);
    return ok;
}
#define DEAM_IN_BOUNDS(G, cond, site, idx) ::deam::in_bounds((G).fault, (cond), (site), (long long)(idx))
#else
#define DEAM_IN_BOUNDS(G, cond, site, idx) true
#endif

// Spectral model tables (kernel parameters: they live in the constant bank).
struct Spec {
    int e_lo, e_hi;                  // active bins [e_lo, e_hi)
    float mu1l2[kMaxE], mu2l2[kMaxE];  // mu_i(E) * log2(e), 1/mm
    float mu1[kMaxE], mu2[kMaxE];      // mu_i(E), 1/mm
    float i0l[kMaxE], i0h[kMaxE];      // I0_j(E), counts
};

struct InPlane {
    int axis;      // 0: x-dominant (planes ix), 1: y-dominant (planes iy)
    float aq, bq;  // fq(p) = aq + p bq: intercept with plane p on the other transaxial axis (index units)
    float tau0, kappa;  // ray parameter t(p) = tau0 + p kappa (fraction of u)
    float Lxy;     // (plane spacing) / |d_dominant|; times the row factor gives Joseph's L
};

// In-plane ray parameters of (view, channel).  Explicitly rounded operations
// (no contraction freedom) make the result identical wherever it is inlined.
__device__ __forceinline__ InPlane ray_inplane(const Geo& G, float4 vw, float2 ch) {
    // d_k = -(cos(beta + gamma), sin(beta + gamma)) by the angle-sum identities
    const float dxk = __fmaf_rn(vw.w, ch.y, -__fmul_rn(vw.z, ch.x));
    const float dyk = -__fmaf_rn(vw.w, ch.x, __fmul_rn(vw.z, ch.y));
    InPlane r;
    if (fabsf(dxk) >= fabsf(dyk)) {
        r.axis = 0;
        const float m = __fmul_rn(__fdiv_rn(dyk, dxk), G.dx_dy);
        r.aq = __fmaf_rn(-vw.x, m, vw.y);
        r.bq = m;
        r.kappa = __fdiv_rn(G.dx_sdd, dxk);
        r.tau0 = __fmul_rn(-vw.x, r.kappa);
        r.Lxy = __fdiv_rn(G.dx, fabsf(dxk));
    } else {
        r.axis = 1;
        const float m = __fmul_rn(__fdiv_rn(dxk, dyk), G.dy_dx);
        r.aq = __fmaf_rn(-vw.y, m, vw.x);
        r.bq = m;
        r.kappa = __fdiv_rn(G.dy_sdd, dyk);
        r.tau0 = __fmul_rn(-vw.y, r.kappa);
        r.Lxy = __fdiv_rn(G.dy, fabsf(dyk));
    }
    return r;
}

// In-plane parameters of (view, channel) read back from the table that
// build_inplane_table filled with ray_inplane(): the forward and backward
// projectors both read it, so their sample positions are identical by construction.
__device__ __forceinline__ InPlane inplane_at(float4 a, float lsigned) {
    InPlane r;
    r.axis = lsigned < 0.f ? 1 : 0;
    r.aq = a.x;
    r.bq = a.y;
    r.tau0 = a.z;
    r.kappa = a.w;
    r.Lxy = fabsf(lsigned);
    return r;
}

// Row height omega_r = w_r / dz of detector row r, in slices: omega0 + r domega,
// one explicitly rounded FMA wherever either projector direction needs it.
__device__ __forceinline__ float row_omega(const Geo& G, int r) { return __fmaf_rn((float)r, G.domega, G.omega0); }

// Ray parameter at plane p (fraction of u from the source): t(p) = tau0 + p kappa.
__device__ __forceinline__ float ray_t(const InPlane& ip, float p) { return __fmaf_rn(p, ip.kappa, ip.tau0); }

// z-intercept (index units) of the ray of row r at ray parameter t:
// fz = sigma_z + omega_r t.  Both projector directions evaluate exactly this
// expression (t from ray_t), so they select the same taps.
__device__ __forceinline__ float row_fz(float sigma_z, float omega, float t) { return __fmaf_rn(omega, t, sigma_z); }

// ---------------------------------------------------------------------------
// kernel launchers (deam_kernels.cu)
// ---------------------------------------------------------------------------
enum BwdMode { BWD_ADJOINT = 0, BWD_UPDATE = 1, BWD_GRADIENT = 2 };
// FWD_DEAM_F32: FWD_DEAM with plain FP32 spectral sums and FP32 objective
// accumulation (the uncompensated variant, for comparison)
enum FwdMode { FWD_LINE = 0, FWD_LINE_G = 1, FWD_DEAM = 2, FWD_MASK = 3, FWD_MAX = 4, FWD_COUNT = 5, FWD_DEAM_F32 = 6 };

struct FwdArgs {
    const float4* volX;   // [nx][nz+2][ny+1] q-paired layout for x-dominant rays
    const float4* volY;   // [ny][nz+2][nx+1] q-paired layout for y-dominant rays
    float2* l_out;        // FWD_LINE(_G): [V][R][K] line integrals (nullable in LINE_G)
    float* g_out;         // FWD_LINE_G: [2][V][R][K] expected counts
    const float* dt;      // FWD_DEAM: d~ [2][V][R][K]
    const uint8_t* mask;  // FWD_DEAM: [V][R][K] metal traces, bit j = spectrum j (nullable: none);
                          // FWD_LINE: project only the rays in or next to a trace (nullable: all)
    const float* bowtie;  // [K] (nullable: 1)
    float4* payload;      // FWD_DEAM: [V][R][K] (B~1, B~2, D1, D2)
    double* partial;      // FWD_DEAM: per-block objective; FWD_MAX: per-block max; FWD_COUNT: samples
    double* total;        // FWD_DEAM with fwd_rows 1: the objective (nullable: the partials alone)
    unsigned* ticket;     // with total: counts finished blocks; 0 between launches
    unsigned long long* clear;  // with total: set to 0 (nullable)
    uint8_t* mask_out;    // FWD_MASK
    float threshold;      // FWD_MASK
    int fold_rowfac;      // FWD_DEAM: 1 stores the payload times the row length factor (the
                          // backprojector's input form); 0: the payload as defined (deam_ray_terms)
};

struct BwdArgs {
    const float2* rays2;    // BWD_ADJOINT input [V][R][K][2]
    const float4* payload;  // BWD_UPDATE / BWD_GRADIENT input [V][R][K][4]
    float2* img;            // adjoint or gradient output / update in-out c [nz][ny][nx]
    const int2* slab_views; // [n_slabs][tiles y][tiles x] view range [lo, hi] per z-slab and column tile
    double invZ;            // 1 / Z of the c-step
    int clamp_nonneg;
    unsigned long long* skipped;  // update: count of unchanged (voxel, component) pairs
    // regularised c-step (Eqs. 6-7), lambda > 0: the backprojection stores its
    // per-voxel sums in `sums` and reg_update_kernel solves; neighbours' c^k are
    // read from the projector layout volX, which holds c^k while the update runs
    float4* sums;                 // [nvox] (b~_1, b~_2, delta_1, delta_2); nullptr: plain c-step
    float lambda, delta, Z;
    float pdx, pdy, pdz;          // voxel edges (mm) for the 1/distance weights
    const float4* volX;
};

// Batched launch over many scans (deam_batch_*): per-scan descriptors in
// device memory and prefix sums of each scan's work items.
struct BatchDesc {
    int n;                      // scans
    const Geo* geos;            // [n]
    const Spec* specs;          // [n]
    const FwdArgs* fargs;       // [n]
    const BwdArgs* bargs;       // [n] (slab views for the chosen slab depth)
    const long long* ftile_off; // [n+1] prefix sums of forward ray tiles
    const long long* btile_off; // [n+1] prefix sums of backprojection tiles
    double* partial;            // [ftile_off[n]] objective per forward tile
};
// Scan of batch work item t: the last i with off[i] <= t (prefix sums of the
// scans' work items).
__device__ __forceinline__ int find_scan(const long long* off, int n, long long t) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(&off[mid]) <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Forward ray-tile and backprojection-tile shapes an autotuner may choose from.
constexpr int kFwdShapes[3][2] = {{8, 1}, {4, 2}, {2, 4}};             // (rows, views) x 32 channels
constexpr int kNumBwdShapes = 6;
constexpr int kBwdShapes[kNumBwdShapes][3] = {{2, 16, 8}, {2, 32, 4}, {8, 16, 8},
                                              {8, 32, 4}, {16, 16, 8}, {16, 32, 4}};  // (slab, tx, ty)
// Slab class of the gather backprojection for a scan: 2 for one or two
// slices, 8 when a detector row covers at most 2/3 of a slice (several rows
// per slice), else 16.  The batched launches use the class as their
// slab depth; a single-scan context runs its own plan (bwd_plan).
inline int pick_slab(int nz, int n_rows, double dz, double row_pitch, double sid, double sdd) {
    if (nz <= 2) return 2;
    return (n_rows == 1 || dz >= 1.5 * row_pitch * sid / sdd) ? 8 : 16;
}
// Rays of a view that one turn of the row loop takes (more rays: more turns).
// Four at 5 blocks of 128 threads per SM; three at 6 blocks are as fast at 2.6
// rays per view and 8 % slower at 3.5 (384^2 x 48 on 816 channels).  Two where a
// column is tapped by fewer than 1.9 rays of a view, one below 0.7 (turn_rays), as a
// turn costs its rays whether they tap or not: 360 views, 4 / 2 / 1 rays per turn at
// 512^2 x 16 and 64 channels (0.2 rays) 3.18 / 2.30 / 2.08 ms, 200 (0.7) 3.54 / 2.50 /
// 2.50, 300 (1.0) 3.60 / 2.59 / 3.28, 500 (1.7) 3.71 / 3.27; at 256^2 x 32 and 100
// channels (0.7) 1.30 / 0.95 / 0.86, 200 (1.4) 1.37 / 1.02 / 1.45, 300 (2.1) 1.42 / 1.46,
// 400 (2.7) 1.48 / 1.80.
constexpr int kRaysPerView = 4;
// How a single-scan context backprojects: z-slabs of `slab` slices, and the views
// of a column shared out over `vs` warps (whose sums are added at the end).
//   slab: a deep slab costs less set-up per sample (a slab is visited by the views
//   of slab + rows covered), a shallow one leaves more of the 256 KB to L1.  16
//   against 13 slices, deep class: 18.7 / 19.8 ms at 384^2 x 48, 11.5 / 12.5 ms at
//   256^2 x 16 x 1440 views, 22.9 / 23.1 ms on a rotation of 512^2 x 64.  With
//   rows of 2/3 of a slice or less 11 against 16: 8.5 / 9.8 ms on a rotation of
//   256^2 x 32 x 672 channels; 11, 8 and 13 slices: there 8.6 / 9.3 / 9.0, 384^2 x 48
//   12.0 / 12.4 / 11.3, 384^2 x 24 11.5 / 12.0 / 11.1, 512^2 x 64 10.6 / 11.2 / 10.6,
//   192^2 x 40 2.76 / 2.79 / 2.61, 320^2 x 33 with one row 1.60 / 1.55 / 1.61 (the
//   slices that the last slab leaves empty weigh as much as the depth).
//   vs: 5 blocks of 4 warps run on an SM; below 8 rounds of the GPU the views are
//   split so that the last, part-filled round weighs less: 4 warps against 1
//   11.8 -> 9.9 ms (256^2 x 16: 2048 warps of columns), 11.7 -> 8.5 ms (256^2 x 32);
//   2 against 1 19.4 -> 18.8 ms (384^2 x 48: 13,824); at 512^2 x 64 (32,768) 1 is
//   as fast as 2 and 3 % faster than 4.  Warps that get no eight views of their own
//   are idle, and where the columns alone fill the GPU each should have two eights, or
//   setting up and adding the sums costs more than is gained: 256^2 x 32 with 1 / 2 / 4
//   warps 8 views 92 / 122 / 206 us, 36 views 233 / 209 / 232, 90 views 469 / 417 / 430;
//   96^2 x 8 (288 warps) 8 views 101 / 104 / 107, 24 views 194 / 149 / 105.
//   view_step: two views a turn, but one where their samples lie in different slices:
//   a source that moves by 0.4 slices or more from view to view (256^2 x 32, 0.1 / 0.3 /
//   0.6 / 2 slices: two 1.48 / 0.63 / 0.36 / 0.26 ms, one 1.57 / 0.58 / 0.27 / 0.14),
//   or fewer than 16 views per rotation (0.1 slices apart, 12 / 24 / 60 views: two 1.64 /
//   1.51 / 1.48 ms, one 1.51 / 1.52 / 1.57).
//   single slices (slab 1): with four 16 x 8 patches per SM, 2 x 2 columns per thread
//   and 8 warps of views (4, 8, 16: 0.89, 0.85, 0.90 ms at 512^2); below, one column
//   per thread and 16 (8: 55 us against 53 at 128^2).
struct BwdPlan {
    int slab = 2, vs = 4;
    int view_step = 2;  // views a turn of the row loop takes (slabs)
    int rays = kRaysPerView;  // rays of each that it takes
    bool flat = false;  // slab 1: all rays lie in the slice
};
constexpr int kMidSlab = 11, kDeepSlab = 16;
constexpr int bwd_tile_x(int vs) { return vs == 1 ? 16 : 8; }
constexpr int bwd_tile_y(int vs) { return vs == 4 ? 4 : 8; }
long long forward_tiles(int shape, const Geo& G);
long long backward_tiles(int shape, const Geo& G);
cudaError_t launch_forward_batch(int shape, const BatchDesc& B, int grid, cudaStream_t s);
cudaError_t launch_backward_batch(int shape, const BatchDesc& B, int grid, cudaStream_t s);
// out[i * stride + *counter] = sum of partial[off[i] .. off[i+1]) (fixed order)
cudaError_t launch_sum_ranges(const double* partial, const long long* off, int n, double* out, const int* counter,
                              int stride, cudaStream_t s);
cudaError_t launch_counter_inc(int* counter, cudaStream_t s);

cudaError_t launch_inplane_table(const Geo& G, float4* ip4, float* ipL, cudaStream_t s);
cudaError_t launch_layout(const float2* c, const float* m, int ones, float4* volX, float4* volY,
                          int nx, int ny, int nz, cudaStream_t s);
// Detector rows that a thread of the forward kernel projects at once: 1, 4 or 8.
int forward_rows(const deam_geometry& g, int sms);
// Blocks of four warps instead of eight: scans of one row per thread whose blocks of
// eight are all resident at once, where whole blocks leave some SMs with a third more
// work than others (128^2 x 360 views, 360 blocks of eight: 33 us, of four 29, of two
// 29 and longer to add up).
bool forward_narrow(const Geo& G, int sms);
// Blocks of the forward grid: one per ray tile.
int forward_blocks(const Geo& G);
cudaError_t launch_forward(int mode, const Geo& G, const Spec& S, const FwdArgs& A, int n_blocks,
                           cudaStream_t s);
cudaError_t launch_backward(int mode, const BwdPlan& P, const Geo& G, const BwdArgs& A, cudaStream_t s);
cudaError_t launch_sum_partials(const double* partial, int n, double* out, int do_max, cudaStream_t s);
cudaError_t launch_clamp_copy(const float* d, float* dt, long long n, cudaStream_t s);
cudaError_t launch_mask_bits(uint8_t* m, long long n, int per_spectrum, cudaStream_t s);
cudaError_t launch_reg_update(const Geo& G, const BwdArgs& A, cudaStream_t s);
cudaError_t launch_penalty(const float2* c, int nx, int ny, int nz, float dx, float dy, float dz, float lambda,
                           float delta, double* partial, int n_blocks, cudaStream_t s);
// Measured shared-memory (L1 data path) load throughput of this device, bytes/s.
cudaError_t l1_probe(double* bytes_per_s, cudaStream_t s);
cudaError_t launch_combine(const float2* c, long long nvox, const float2* ab, int n, float* out, cudaStream_t s);

// Record an error message for deam_last_error() and return code (deam_api.cu).
int set_error(int code, const char* msg);
// Validate a scan description on the host: "" if deam_init would accept it,
// else the reason (deam_api.cu).
std::string validate_scan(const deam_geometry* g, const deam_spectra* s, const deam_basis* b);

}  // namespace deam
