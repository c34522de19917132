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
constexpr int kLaneVox = 4;          // voxels per lane of the fusion kernels

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
    // most blocks lie inside one view
    const bool whole = lo + 1 >= V || view_of<BY_VALUE>(set, table, lo + 1).q0 >= first + kTsdfThreads * kDepthItems;
    int64_t shift = view_of<BY_VALUE>(set, table, lo).pix_off - view_of<BY_VALUE>(set, table, lo).q0;
    float a[kDepthItems], d[kDepthItems];               // loads in flight together
#pragma unroll
    for (int m = 0; m < kDepthItems; ++m) {
        const int64_t q = first + m * kTsdfThreads + threadIdx.x;
        if (!whole) {
            while (lo + 1 < V && view_of<BY_VALUE>(set, table, lo + 1).q0 <= q) ++lo;
            shift = view_of<BY_VALUE>(set, table, lo).pix_off - view_of<BY_VALUE>(set, table, lo).q0;
        }
        const int64_t p = q + shift;
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
// integer comparison for 0 <= u < W (u = -0 is a product that underflowed below zero: cx and cy are not -0).
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

// Warp = 32 kLaneVox consecutive voxels in storage order, lane + 32 m the m-th of a lane, whatever rows
// they belong to: for rows that k_tsdf_rows would pad with idle lanes.  The view's fields are read once
// for a lane's voxels, as there; nothing is shared along a row.  256 x 256 rows, 32 views of 640x480,
// a voxel of 1.2 px, with the pre-pass, against four adjacent voxels per thread with the view table in
// shared memory (one per thread where the row length is no multiple of four), and against segments
// of one row with one or two voxels per lane: rows of 28 voxels 190 / 199 -> 126 us, 33 248 / 235 -> 142, 64
// 330 / 240 -> 236, 80 396 / 406 -> 285, 129 751 / 635 -> 442.
template <bool BY_VALUE>
__global__ void __launch_bounds__(kTsdfThreads) k_tsdf(float* __restrict__ F, float* __restrict__ Wt, int nx, int ny,
                                                       int64_t n_vox, TsdfParams TP,
                                                       const __grid_constant__ TsdfViews set,
                                                       const TsdfView* __restrict__ table, int V,
                                                       const float* __restrict__ dn) {
    // (fewer than 2^31 voxels: 32-bit indices)
    const uint32_t idx0 = (blockIdx.x * (kTsdfThreads / 32u) + (threadIdx.x >> 5)) * (32u * kLaneVox) + lane_id();
    const uint32_t n = (uint32_t)n_vox;
    float px[kLaneVox], py[kLaneVox], pz[kLaneVox], ms[kLaneVox], f[kLaneVox], w[kLaneVox];
#pragma unroll
    for (int m = 0; m < kLaneVox; ++m) {
        const uint32_t idx = idx0 + 32u * m, r = idx / (uint32_t)nx, k = r / (uint32_t)ny;
        voxel_x((int)(idx - r * (uint32_t)nx), nx, TP, px[m], ms[m]);
        if (idx >= n) px[m] = __int_as_float(0x7fc00000);   // no view sees it
        py[m] = fmaf((float)(int)(r - k * (uint32_t)ny) + 0.5f, TP.voxel, TP.oy);
        pz[m] = fmaf((float)(int)k + 0.5f, TP.voxel, TP.oz);
        f[m] = idx < n ? F[idx] : 0.f;
        w[m] = idx < n ? Wt[idx] : 0.f;
    }
    for (int v = 0; v < V; ++v) {
        const TsdfView& cv = view_of<BY_VALUE>(set, table, v);
        const float sx = cv.R[0] * TP.voxel, sy = cv.R[3] * TP.voxel, sz = cv.R[6] * TP.voxel;
        const float cx = cv.cx, cy = cv.cy, Wf = cv.Wf, Hf = cv.Hf;
        const uint32_t W = (uint32_t)cv.W;
        const float* __restrict__ dv = dn + cv.q0;
        float zm[kLaneVox], d[kLaneVox];
        uint32_t pix[kLaneVox];
        bool ok[kLaneVox];
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) {
            const float z0 = fmaf(cv.R[6], px[m], fmaf(cv.R[7], py[m], fmaf(cv.R[8], pz[m], cv.t[2])));
            const float x0 = fmaf(cv.R[0], px[m], fmaf(cv.R[1], py[m], fmaf(cv.R[2], pz[m], cv.t[0])));
            const float y0 = fmaf(cv.R[3], px[m], fmaf(cv.R[4], py[m], fmaf(cv.R[5], pz[m], cv.t[1])));
            const float z = fmaf(ms[m], sz, z0);
            const float x = fmaf(ms[m], sx, x0), y = fmaf(ms[m], sy, y0);
            const float iz = rcp(z);
            const float u = fmaf(cv.fx * x, iz, cx), vv = fmaf(cv.fy * y, iz, cy);
            ok[m] = z > 0.f && in_range(u, Wf) && in_range(vv, Hf);
            pix[m] = pixel_of(u, vv, W);                // (below 2^30 where it is used)
            zm[m] = z;
        }
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) d[m] = ok[m] ? __ldg(dv + pix[m]) : 0.f;
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) fuse(d[m], zm[m], ok[m], TP, f[m], w[m]);
    }
#pragma unroll
    for (int m = 0; m < kLaneVox; ++m) {
        const uint32_t idx = idx0 + 32u * m;
        if (idx < n) {
            F[idx] = f[m];
            Wt[idx] = w[m];
        }
    }
}

// Warp = kLaneVox x 32 consecutive voxels of one row, lane + 32 m the m-th of a lane: neighbouring lanes
// hold neighbouring voxels, whose projections share the 32-byte sectors of the depth image, the
// kLaneVox projections are made before the gathers, which are then in flight together, and the
// row's part of the camera transform is shared.  Each voxel takes the views in order.
// Bound by issue slots.  256^3 voxels and 32 views of 640x480, with the pre-pass: 0.77 ms; four adjacent
// voxels per thread with the view table in shared memory took 1.12 ms (gathers of neighbouring lanes 4
// voxels apart, conversions on the quarter-rate unit), this mapping with the table in shared memory 0.87.
template <bool BY_VALUE>
__global__ void __launch_bounds__(kTsdfThreads) k_tsdf_rows(float* __restrict__ F, float* __restrict__ Wt, int nx, int ny,
                                                            int64_t n_seg, int segs, TsdfParams TP,
                                                            const __grid_constant__ TsdfViews set,
                                                            const TsdfView* __restrict__ table, int V,
                                                            const float* __restrict__ dn) {
    const int64_t seg = (int64_t)blockIdx.x * (kTsdfThreads / 32) + (threadIdx.x >> 5);
    if (seg >= n_seg) return;
    const int64_t row = seg / segs;
    const int i0 = (int)(seg - row * segs) * (32 * kLaneVox) + (int)lane_id();
    const int j = (int)(row % ny), k = (int)(row / ny);
    const float py = fmaf((float)j + 0.5f, TP.voxel, TP.oy), pz = fmaf((float)k + 0.5f, TP.voxel, TP.oz);
    float px[kLaneVox], ms[kLaneVox], f[kLaneVox], w[kLaneVox];
#pragma unroll
    for (int m = 0; m < kLaneVox; ++m) {
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
        float zm[kLaneVox], d[kLaneVox];
        uint32_t pix[kLaneVox];
        bool ok[kLaneVox];
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) {
            const float z = fmaf(ms[m], sz, fmaf(cv.R[6], px[m], rz));
            const float x = fmaf(ms[m], sx, fmaf(cv.R[0], px[m], rx)), y = fmaf(ms[m], sy, fmaf(cv.R[3], px[m], ry));
            const float iz = rcp(z);
            const float u = fmaf(cv.fx * x, iz, cx), vv = fmaf(cv.fy * y, iz, cy);
            ok[m] = z > 0.f && in_range(u, Wf) && in_range(vv, Hf);
            pix[m] = pixel_of(u, vv, W);                // (below 2^30 where it is used)
            zm[m] = z;
        }
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) d[m] = ok[m] ? __ldg(dv + pix[m]) : 0.f;
#pragma unroll
        for (int m = 0; m < kLaneVox; ++m) fuse(d[m], zm[m], ok[m], TP, f[m], w[m]);
    }
#pragma unroll
    for (int m = 0; m < kLaneVox; ++m) {
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
    // rows whose last segment leaves at most a sixteenth of the lanes idle are the faster form where
    // a voxel is about a pixel or less (rows of 128, as above: 404 against 436 us; at 5 px 404 against 381,
    // of 256 756 against 701), longer idle tails are not (112: 403 against 387; 160: 639 against 528)
    const int segs = (nx + 32 * kLaneVox - 1) / (32 * kLaneVox);
    if ((int64_t)segs * 32 * kLaneVox * 16 <= (int64_t)nx * 17) {
        const int64_t n_seg = n_vox / nx * segs;
        constexpr int kWarps = kTsdfThreads / 32;
        k_tsdf_rows<BY_VALUE><<<(unsigned)((n_seg + kWarps - 1) / kWarps), kTsdfThreads, 0, L.stream>>>(
            F, W, nx, ny, n_seg, segs, TP, set, table, V, dn);
    } else {
        constexpr int kVox = kTsdfThreads * kLaneVox;
        k_tsdf<BY_VALUE><<<(unsigned)((n_vox + kVox - 1) / kVox), kTsdfThreads, 0, L.stream>>>(F, W, nx, ny, n_vox, TP,
                                                                                               set, table, V, dn);
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
