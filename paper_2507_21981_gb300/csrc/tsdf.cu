// Depth -> TSDF fusion (Sec. III-B: a Gaussian node is turned back into a mesh by rendering
// multi-view depth maps and fusing them into a truncated signed distance field; the decimation
// that follows is not part of this library).
//
// A pre-pass writes every pixel's normalised depth d = D / A (NaN where A < min_alpha) into a
// packed array.  Then each voxel, x fastest (coalesced field reads and writes),
// takes the views in order: project the voxel centre, read d at the pixel holding
// the projection, sdf = d - z, skip when sdf < -trunc, f = min(1, sdf / trunc),
// F <- (W F + f) / (W + 1), W <- min(W + 1, max_weight).
// The field is read and written once per call whatever the number of views, so a call with
// many views is bound by the per-view arithmetic and the depth gathers (served by L2).
#include <algorithm>

#include "dgs_internal.cuh"

namespace dgs {
namespace {

constexpr int kTsdfThreads = 256;

// The view table: by value as a kernel parameter for up to kTsdfParamViews views, whose fields are
// then constant-bank operands (from shared memory their broadcasts were half of the data path),
// else from device memory.
template <bool BY_VALUE>
__device__ __forceinline__ const TsdfView& view_of(const TsdfViews& by_value, const TsdfView* __restrict__ table, int v) {
    if constexpr (BY_VALUE) return by_value.v[v];
    else return table[v];
}

constexpr int kDepthItems = 4;       // pixels per thread of the pre-pass

// Pre-pass: the normalised depth D / A of every pixel of every view into a packed array (NaN
// where A < min_alpha), so that the fusion makes one gather per (voxel, view) and no division.
// A block takes the next 1024 packed pixels, whatever views they belong to, so that views of very
// different sizes leave no blocks idle (one of 2048^2 among 399 of 64^2, 64^3 voxels, whole call: 0.31 ms,
// 1.62 with a grid of the largest view's blocks for every view).
template <bool BY_VALUE>
__global__ void __launch_bounds__(kTsdfThreads) k_tsdf_depth(const __grid_constant__ TsdfViews set,
                                                             const TsdfView* __restrict__ table, int V, int64_t n_pix,
                                                             float min_alpha, const float* __restrict__ depth,
                                                             const float* __restrict__ alpha, float* __restrict__ dn) {
    const int64_t first = (int64_t)blockIdx.x * (kTsdfThreads * kDepthItems);
    int lo = 0, hi = V - 1;                             // the view of the block's first pixel
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (view_of<BY_VALUE>(set, table, mid).q0 <= first) lo = mid; else hi = mid - 1;
    }
    float a[kDepthItems], d[kDepthItems];               // loads in flight together
#pragma unroll
    for (int m = 0; m < kDepthItems; ++m) {
        const int64_t q = first + m * kTsdfThreads + threadIdx.x;
        while (lo + 1 < V && view_of<BY_VALUE>(set, table, lo + 1).q0 <= q) ++lo;
        const TsdfView& cv = view_of<BY_VALUE>(set, table, lo);
        const int64_t p = cv.pix_off + (q - cv.q0);
        a[m] = q < n_pix ? alpha[p] : 0.f;
        d[m] = q < n_pix ? depth[p] : 0.f;
    }
#pragma unroll
    for (int m = 0; m < kDepthItems; ++m) {
        const int64_t q = first + m * kTsdfThreads + threadIdx.x;
        if (q < n_pix) dn[q] = a[m] >= min_alpha ? __fdividef(d[m], a[m]) : __int_as_float(0x7fc00000);
    }
}

// A voxel's centre along x: px + m voxel, m exact.  Rows of a multiple of four voxels step from
// the first voxel of an aligned group of four (m = 0..3); other rows take each voxel's own centre
// (m = 0).  Both kernels below round the same way.
__device__ __forceinline__ void voxel_x(int i, int nx, const TsdfParams& TP, float& px, float& m) {
    const int q = nx % 4 == 0 ? i & ~3 : i;
    px = fmaf((float)q + 0.5f, TP.voxel, TP.ox);
    m = (float)(i - q);
}

// Non-negative floats order like their bit patterns, negative ones and NaN lie above them: one
// integer comparison for 0 <= u < W (u is never -0: cx and cy are not).
__device__ __forceinline__ bool in_range(float u, float W) { return __float_as_uint(u) < __float_as_uint(W); }

// 1 / x for normal x: the approximate division below without its range handling (a pixel's z and
// a weight plus one are normal; a z that is not gives no pixel).
__device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// floor(u) for 0 <= u < 2^23, exactly: u + 2^23 rounded down holds it in its low bits (an addition
// in place of a conversion, which goes through the quarter-rate unit that rcp needs too).
__device__ __forceinline__ uint32_t floor_bits(float u) { return __float_as_uint(__fadd_rd(u, 8388608.f)); }
constexpr uint32_t kFloorBias = 0x4B000000u;            // bits of 2^23

// Packed pixel of (u, v) in a view of width W, both in range.
__device__ __forceinline__ uint32_t pixel_of(float u, float v, uint32_t W) {
    return floor_bits(v) * W + floor_bits(u) - kFloorBias * (W + 1u);
}

// One view's sample into a voxel's running average.
__device__ __forceinline__ void fuse(float d, float z, bool ok, const TsdfParams& TP, float& f, float& w) {
    const float sdf = d - z;
    if (!ok || !(sdf >= -TP.trunc)) return;             // also a pixel without coverage (NaN)
    const float fv = fminf(1.f, sdf * TP.inv_trunc);
    f = fmaf(w, f, fv) * rcp(w + 1.f);
    w = fminf(w + 1.f, TP.max_weight);
}

// Rows of fewer than 32 voxels: one thread per voxel in storage order.
template <bool BY_VALUE>
__global__ void __launch_bounds__(kTsdfThreads) k_tsdf(float* __restrict__ F, float* __restrict__ Wt, int nx, int ny,
                                                       int64_t n_vox, TsdfParams TP,
                                                       const __grid_constant__ TsdfViews set,
                                                       const TsdfView* __restrict__ table, int V,
                                                       const float* __restrict__ dn) {
    const int64_t idx = (int64_t)blockIdx.x * kTsdfThreads + threadIdx.x;
    if (idx >= n_vox) return;
    const int i = (int)(idx % nx);
    const int64_t r = idx / nx;
    const int j = (int)(r % ny), k = (int)(r / ny);
    float px, m;
    voxel_x(i, nx, TP, px, m);
    const float py = fmaf((float)j + 0.5f, TP.voxel, TP.oy), pz = fmaf((float)k + 0.5f, TP.voxel, TP.oz);
    float f = F[idx], w = Wt[idx];
    for (int v = 0; v < V; ++v) {
        const TsdfView& cv = view_of<BY_VALUE>(set, table, v);
        const float z0 = fmaf(cv.R[6], px, fmaf(cv.R[7], py, fmaf(cv.R[8], pz, cv.t[2])));
        const float x0 = fmaf(cv.R[0], px, fmaf(cv.R[1], py, fmaf(cv.R[2], pz, cv.t[0])));
        const float y0 = fmaf(cv.R[3], px, fmaf(cv.R[4], py, fmaf(cv.R[5], pz, cv.t[1])));
        const float z = fmaf(m, cv.R[6] * TP.voxel, z0);
        const float x = fmaf(m, cv.R[0] * TP.voxel, x0), y = fmaf(m, cv.R[3] * TP.voxel, y0);
        const float iz = rcp(z);
        const float u = fmaf(cv.fx * x, iz, cv.cx), vv = fmaf(cv.fy * y, iz, cv.cy);
        const bool ok = z > 0.f && in_range(u, cv.Wf) && in_range(vv, cv.Hf);
        const float d = ok ? __ldg(dn + cv.q0 + pixel_of(u, vv, (uint32_t)cv.W)) : 0.f;
        fuse(d, z, ok, TP, f, w);
    }
    F[idx] = f;
    Wt[idx] = w;
}

// Warp = NR x 32 consecutive voxels of one row, lane + 32 m the m-th of a lane: neighbouring lanes
// hold neighbouring voxels, whose projections share the 32-byte sectors of the depth image, the
// NR projections are made before the NR gathers, which are then in flight together, and the
// row's part of the camera transform is shared.  Each voxel takes the views in order.
// Bound by issue slots (90 % active, 49 instructions per voxel and view).  256^3 voxels and 32
// views of 640x480, with the pre-pass: 0.766 ms; four adjacent voxels per thread with the view
// table in shared memory took 1.115 ms (gathers of neighbouring lanes 4 voxels apart, conversions on
// the quarter-rate unit), this mapping with the table in shared memory 0.871.  Rows below 32 voxels
// would leave most lanes idle and take k_tsdf.
template <int NR, bool BY_VALUE>
__global__ void __launch_bounds__(kTsdfThreads) k_tsdf_rows(float* __restrict__ F, float* __restrict__ Wt, int nx, int ny,
                                                            int64_t n_seg, int segs, TsdfParams TP,
                                                            const __grid_constant__ TsdfViews set,
                                                            const TsdfView* __restrict__ table, int V,
                                                            const float* __restrict__ dn) {
    const int64_t seg = (int64_t)blockIdx.x * (kTsdfThreads / 32) + (threadIdx.x >> 5);
    if (seg >= n_seg) return;
    const int64_t row = seg / segs;
    const int i0 = (int)(seg - row * segs) * (32 * NR) + (int)lane_id();
    const int j = (int)(row % ny), k = (int)(row / ny);
    const float py = fmaf((float)j + 0.5f, TP.voxel, TP.oy), pz = fmaf((float)k + 0.5f, TP.voxel, TP.oz);
    float px[NR], ms[NR], f[NR], w[NR];
#pragma unroll
    for (int m = 0; m < NR; ++m) {
        const int i = i0 + 32 * m;
        voxel_x(i, nx, TP, px[m], ms[m]);
        if (i >= nx) px[m] = __int_as_float(0x7fc00000);    // no view sees it
        f[m] = i < nx ? F[row * nx + i] : 0.f;
        w[m] = i < nx ? Wt[row * nx + i] : 0.f;
    }
    for (int v = 0; v < V; ++v) {
        const TsdfView& cv = view_of<BY_VALUE>(set, table, v);
        const float rz = fmaf(cv.R[7], py, fmaf(cv.R[8], pz, cv.t[2]));
        const float rx = fmaf(cv.R[1], py, fmaf(cv.R[2], pz, cv.t[0]));
        const float ry = fmaf(cv.R[4], py, fmaf(cv.R[5], pz, cv.t[1]));
        const float sx = cv.R[0] * TP.voxel, sy = cv.R[3] * TP.voxel, sz = cv.R[6] * TP.voxel;
        const float cx = cv.cx, cy = cv.cy, Wf = cv.Wf, Hf = cv.Hf;
        const uint32_t W = (uint32_t)cv.W;
        const float* __restrict__ dv = dn + cv.q0;
        float zm[NR], d[NR];
        uint32_t pix[NR];
        bool ok[NR];
#pragma unroll
        for (int m = 0; m < NR; ++m) {
            const float z = fmaf(ms[m], sz, fmaf(cv.R[6], px[m], rz));
            const float x = fmaf(ms[m], sx, fmaf(cv.R[0], px[m], rx)), y = fmaf(ms[m], sy, fmaf(cv.R[3], px[m], ry));
            const float iz = rcp(z);
            const float u = fmaf(cv.fx * x, iz, cx), vv = fmaf(cv.fy * y, iz, cy);
            ok[m] = z > 0.f && in_range(u, Wf) && in_range(vv, Hf);
            pix[m] = pixel_of(u, vv, W);                // (below 2^30 where it is used)
            zm[m] = z;
        }
#pragma unroll
        for (int m = 0; m < NR; ++m) d[m] = ok[m] ? __ldg(dv + pix[m]) : 0.f;
#pragma unroll
        for (int m = 0; m < NR; ++m) fuse(d[m], zm[m], ok[m], TP, f[m], w[m]);
    }
#pragma unroll
    for (int m = 0; m < NR; ++m) {
        const int i = i0 + 32 * m;
        if (i < nx) {
            F[row * nx + i] = f[m];
            Wt[row * nx + i] = w[m];
        }
    }
}

}  // namespace

template <bool BY_VALUE>
static void tsdf_launch(const Launch& L, float* F, float* W, int nx, int ny, int64_t n_vox, const TsdfParams& TP,
                        const TsdfViews& set, const TsdfView* table, int V, int64_t n_pix, const float* depth,
                        const float* alpha, float* dn) {
    constexpr int kDepthPix = kTsdfThreads * kDepthItems;
    k_tsdf_depth<BY_VALUE><<<(unsigned)((n_pix + kDepthPix - 1) / kDepthPix), kTsdfThreads, 0, L.stream>>>(
        set, table, V, n_pix, TP.min_alpha, depth, alpha, dn);
    if (nx < 32) {
        k_tsdf<BY_VALUE><<<(unsigned)((n_vox + kTsdfThreads - 1) / kTsdfThreads), kTsdfThreads, 0, L.stream>>>(
            F, W, nx, ny, n_vox, TP, set, table, V, dn);
    } else {
        // the widest segment that leaves at most a fifth more lanes idle than single rounds do (128 x 128
        // rows, 16 views, against the four-voxel kernel: rows of 33 voxels 59 -> 50 us, 36 53 -> 49, 50 74 ->
        // 49, 98 114 -> 72, 130 141 -> 102, 250 232 -> 117; of 24, by k_tsdf, 49 -> 39)
        const int rounds = (nx + 31) / 32;
        const int NR = (rounds + 3) / 4 * 4 * 5 <= rounds * 6 ? 4 : (rounds + 1) / 2 * 2 * 5 <= rounds * 6 ? 2 : 1;
        const int segs = (rounds + NR - 1) / NR;
        const int64_t n_seg = n_vox / nx * segs;
        auto* kern = NR == 4 ? k_tsdf_rows<4, BY_VALUE> : NR == 2 ? k_tsdf_rows<2, BY_VALUE> : k_tsdf_rows<1, BY_VALUE>;
        kern<<<(unsigned)((n_seg + kTsdfThreads / 32 - 1) / (kTsdfThreads / 32)), kTsdfThreads, 0, L.stream>>>(
            F, W, nx, ny, n_seg, segs, TP, set, table, V, dn);
    }
    *L.launches += 2;
}

void launch_tsdf(const Launch& L, float* F, float* W, int nx, int ny, int64_t n_vox, const TsdfParams& TP,
                 const TsdfView* host_views, const TsdfView* table, int V, const float* depth, const float* alpha,
                 float* dn) {
    if (n_vox <= 0 || V <= 0) return;
    const int64_t n_pix = host_views[V - 1].q0 + (int64_t)host_views[V - 1].W * host_views[V - 1].H;
    TsdfViews set{};
    if (V <= kTsdfParamViews) {
        std::copy(host_views, host_views + V, set.v);
        tsdf_launch<true>(L, F, W, nx, ny, n_vox, TP, set, nullptr, V, n_pix, depth, alpha, dn);
    } else {
        tsdf_launch<false>(L, F, W, nx, ny, n_vox, TP, set, table, V, n_pix, depth, alpha, dn);
    }
}

}  // namespace dgs
