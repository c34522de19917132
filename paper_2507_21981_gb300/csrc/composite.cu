// Tile ranges (K4) and front-to-back compositing of RGB + depth (K5).
//
// Sec. III-A: after sorting, every screen tile owns a contiguous run of depth-ordered
// Gaussians and each pixel alpha-blends them front to back.  Sec. III-C: the depth image is
// produced the same way, by alpha-compositing the camera-space z of the Gaussians.
//
// Two warps per block (two 8x4 sub-tiles of one tile), one thread per pixel.  A pixel stops at the
// first Gaussian that would drive its transmittance below t_min (that Gaussian is not
// composited); a warp stops once all of its pixels have.
#include <algorithm>

#include "dgs_internal.cuh"

namespace dgs {
namespace {

// Thread = 4 consecutive sorted keys at a time (one 16-byte load), grid-stride over the live
// keys (the grid is sized for the capacity, at most a few waves); a run starts where the key's
// tile differs from the one before and ends where it differs from the one after.  A key names
// (view in group, tile in view); its tile in the group is the view's first tile + tile in view.
__global__ void k_ranges(const uint32_t* __restrict__ keys, uint32_t n, const uint32_t* __restrict__ d_n,
                         uint2* __restrict__ ranges, int n_tiles, const ViewDesc* __restrict__ views, int v0, int nv,
                         int tile0, int tbits) {
    if (d_n) n = min(n, *d_n);
    const uint32_t stride = gridDim.x * blockDim.x * 4u;
    for (uint32_t i4 = (blockIdx.x * blockDim.x + threadIdx.x) * 4u; i4 < n; i4 += stride) {
    uint32_t k[6];                                  // k[0] = key before, k[5] = key after
    if (i4 + 4 <= n) {
        const uint4 q = *reinterpret_cast<const uint4*>(keys + i4);
        k[1] = q.x; k[2] = q.y; k[3] = q.z; k[4] = q.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) k[1 + j] = i4 + j < n ? keys[i4 + j] : 0u;
    }
    k[0] = i4 > 0 ? keys[i4 - 1] : 0u;
    k[5] = i4 + 4 < n ? keys[i4 + 4] : 0u;
#pragma unroll
    for (int j = 0; j < 6; ++j) k[j] &= kTileMask;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t i = i4 + j;
        if (i >= n) break;
        const uint32_t t = k[1 + j];
        const bool first = i == 0 || k[j] != t, last = i + 1 == n || k[2 + j] != t;
        if (!first && !last) continue;              // the view is decoded at run ends only
        const uint32_t vg = t >> tbits;
        if (vg >= (uint32_t)nv) continue;           // dead pairs sort past every real tile
        const uint32_t gt = (uint32_t)(views[v0 + vg].tile_base - tile0) + (t & ((1u << tbits) - 1u));
        if (gt >= (uint32_t)n_tiles) continue;      // (only keys of a sort that gave up waiting)
        if (first) ranges[gt].x = i;
        if (last) ranges[gt].y = i + 1;
    }
    }
}

// Heaviest tiles first (the longest-processing-time rule of list scheduling): a view group with
// few waves of tiles is otherwise finished by the blocks of its longest lists while most SMs
// idle, so the compositors take their tiles in descending order of list length, bucketed at 8
// steps per octave of length.  One block; within a bucket the order is arbitrary.
__device__ __forceinline__ uint32_t length_bucket(uint2 r) {
    const uint32_t c = r.y - r.x + 1u;              // >= 1
    const uint32_t oct = 31u - (uint32_t)__clz(c);  // floor(log2 c), 0..31
    const uint32_t frac = oct >= 3 ? (c >> (oct - 3)) & 7u : (c << (3 - oct)) & 7u;
    return 255u - min(255u, oct * 8u + frac);       // heaviest first
}

__global__ void __launch_bounds__(1024) k_tile_order(const uint2* __restrict__ ranges, int n_tiles, uint32_t* order) {
    __shared__ uint32_t cnt[256];
    if (threadIdx.x < 256) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < n_tiles; t += blockDim.x) atomicAdd(&cnt[length_bucket(ranges[t])], 1u);
    __syncthreads();
    if (threadIdx.x < 32) {                         // exclusive scan of the 256 counts, 8 per lane
        const int lane = threadIdx.x;
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { v[j] = cnt[lane * 8 + j]; sum += v[j]; }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t run = incl - sum;
#pragma unroll
        for (int j = 0; j < 8; ++j) { cnt[lane * 8 + j] = run; run += v[j]; }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n_tiles; t += blockDim.x) order[atomicAdd(&cnt[length_bucket(ranges[t])], 1u)] = t;
}

// The same order for more than kOrderOneBlock tiles, over many blocks: bucket counts, which the last
// block to finish turns into the buckets' first places, then the placement (28,800 tiles: 16 us,
// one block takes 26).
__global__ void __launch_bounds__(256) k_order_count(const uint2* __restrict__ ranges, int n_tiles, uint32_t* cnt, uint32_t* done) {
    __shared__ uint32_t s_cnt[256];
    __shared__ bool s_last;
    __shared__ uint32_t s_w[8];
    s_cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int t = blockIdx.x * 256 + threadIdx.x; t < n_tiles; t += gridDim.x * 256) atomicAdd(&s_cnt[length_bucket(ranges[t])], 1u);
    __syncthreads();
    if (s_cnt[threadIdx.x]) atomicAdd(cnt + threadIdx.x, s_cnt[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t v = __ldcg(cnt + threadIdx.x);
    uint32_t y = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y += t;
    }
    if (lane == 31) s_w[warp] = y;
    __syncthreads();
    uint32_t pre = y - v;
    for (int w = 0; w < warp; ++w) pre += s_w[w];
    cnt[threadIdx.x] = pre;
}

__global__ void __launch_bounds__(256) k_order_place(const uint2* __restrict__ ranges, int n_tiles, uint32_t* cnt,
                                                     uint32_t* __restrict__ order) {
    __shared__ uint32_t s_cnt[256], s_base[256];
    s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int t = blockIdx.x * 256 + threadIdx.x;
    const uint32_t b = t < n_tiles ? length_bucket(ranges[t]) : 0u;
    const uint32_t rank = t < n_tiles ? atomicAdd(&s_cnt[b], 1u) : 0u;
    __syncthreads();
    const uint32_t c = s_cnt[threadIdx.x];          // one global addition per bucket and block
    if (c) s_base[threadIdx.x] = atomicAdd(cnt + threadIdx.x, c);
    __syncthreads();
    if (t < n_tiles) order[s_base[b] + rank] = (uint32_t)t;
}

// One block: every tile's first checkpoint slot (an exclusive scan of its segments after the
// first, in tile order), then the (tile, segment) jobs of the adjoint in descending order of
// their length, bucketed as above; *n_jobs = their number.
__global__ void __launch_bounds__(1024) k_segment_jobs(const uint2* __restrict__ ranges, int n_tiles, Checkpoints ck) {
    __shared__ uint32_t cnt[256];
    __shared__ uint32_t s_w[32];
    __shared__ uint32_t s_carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto n_seg = [&](int t) { const uint2 r = ranges[t]; return (r.y - r.x + kSegEntries - 1) / kSegEntries; };
    if (tid < 256) cnt[tid] = 0;
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int t0 = 0; t0 < n_tiles; t0 += blockDim.x) {
        const int t = t0 + tid;
        const uint32_t v = t < n_tiles ? max(n_seg(t), 1u) - 1u : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        uint32_t pre = s_carry, all = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
            if (q < warp) pre += s_w[q];
            all += s_w[q];
        }
        if (t < n_tiles) ck.off[t] = pre + x - v;
        __syncthreads();
        if (tid == 0) s_carry += all;
        __syncthreads();
    }
    for (int t = tid; t < n_tiles; t += blockDim.x) {
        const uint2 r = ranges[t];
        const uint32_t ns = n_seg(t);
        for (uint32_t sg = 0; sg < ns; ++sg) {
            const uint32_t a = r.x + sg * kSegEntries;
            atomicAdd(&cnt[length_bucket(make_uint2(a, min(r.y, a + kSegEntries) - 1u))], 1u);
        }
    }
    __syncthreads();
    if (tid < 32) {
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { v[j] = cnt[tid * 8 + j]; sum += v[j]; }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (tid >= o) incl += y;
        }
        uint32_t run = incl - sum;
#pragma unroll
        for (int j = 0; j < 8; ++j) { cnt[tid * 8 + j] = run; run += v[j]; }
        if (tid == 31) *ck.n_jobs = run;
    }
    __syncthreads();
    for (int t = tid; t < n_tiles; t += blockDim.x) {
        const uint2 r = ranges[t];
        const uint32_t ns = n_seg(t);
        for (uint32_t sg = 0; sg < ns; ++sg) {
            const uint32_t a = r.x + sg * kSegEntries;
            const uint32_t b = length_bucket(make_uint2(a, min(r.y, a + kSegEntries) - 1u));
            ck.jobs[atomicAdd(&cnt[b], 1u)] = make_uint2((uint32_t)t, sg);
        }
    }
}

// Block = kCompWarps sub-tiles of one tile, warp = one 8x4 sub-tile, lane = one pixel; warps are
// independent (no block barrier).  A warp scans the tile's list 128 entries per step, keeps those
// whose sub-tile mask (written by binning: the ellipse reaches a pixel centre of the sub-tile,
// exact test with the binning margin) holds its bit, and queues their instance numbers; 32 queued
// entries make a batch, whose records are gathered one per lane while the batch before is
// composited, and staged in shared memory.  The blend takes kBlend records at a time: their
// alphas first (independent of each other), then the pixel's transmittance through them in order.
// It stops once the warp's 32 pixels have terminated.
//
// What bounds it: on views of few tiles the longest lists, each a serial chain of one warp, so the
// latency per record; on large batches the shared-memory data path (three 16-byte broadcasts per
// record move 512 B each to registers: 12 cycles an SM; 88 % busy, 72 % issue).  Measured, one view
// group, against staging each 32-entry chunk by itself and blending record by record: 64x2
// 640x480 views 4.15 -> 3.91 ms; 46 ragged views 2.76 -> 1.73; two views 0.145 -> 0.072.  The
// packed multiply-adds are 5-10 % of that, marking an ended pixel by its sign bit with an OR
// 1-2 %; kBlend 2 or 8, or 18 blocks (which spill), are slower on the batch.
//
// AUG: the view's image randomisation is applied to the RGB before it is stored.  CK: the
// per-pixel state is checkpointed at every segment start for the adjoint (see Checkpoints);
// batches then end at segment ends.
constexpr int kScan = 4;                        // list entries per lane and scan step
constexpr int kQueue = 256;                     // ring of queued entries: at most 31 + 32 kScan are held
constexpr int kBlend = 4;
static_assert(kSegEntries % (32 * kScan) == 0, "a scan step must not cross a segment");
static_assert(kQueue >= 31 + 32 * kScan && (kQueue & (kQueue - 1)) == 0, "ring size");

template <bool COUNT, bool AUG, bool CK, int BLOCKS>
__global__ void __launch_bounds__(kCompWarps * 32, BLOCKS) k_composite(const ViewDesc* __restrict__ views, int v0, int nv,
                                                   const uint2* __restrict__ ranges, const uint32_t* __restrict__ keys,
                                                   const uint32_t* __restrict__ vals,
                                                   const Record* __restrict__ rec, Params P, float* __restrict__ out_rgb,
                                                   float* __restrict__ out_depth, float* __restrict__ out_alpha,
                                                   unsigned long long* __restrict__ work,
                                                   const uint32_t* __restrict__ tile_order, Checkpoints ck) {
    __shared__ float4 s_rec[kCompWarps][3][32];
    __shared__ uint32_t s_queue[kCompWarps][kQueue];
    if (sort_failed(P.err)) return;            // the lists are not valid: nothing to composite
    // kCompWarps sub-tiles of one tile per block: a block frees its slot as soon as its own
    // warps end, not when the tile's slowest sub-tile does
    const int bpt = (P.tile_w * P.tile_h) / (32 * kCompWarps);   // blocks per tile
    const int tb = (int)blockIdx.x / bpt;
    const int gt = tile_order ? (int)tile_order[tb] : tb;        // tile within the group
    const int ga = gt + P.tile0;               // tile within the call
    // view of this tile: last view of the group whose tile_base <= ga
    int lo = v0, hi = v0 + nv - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (views[mid].tile_base <= ga) lo = mid; else hi = mid - 1;
    }
    const ViewDesc& vd = views[lo];
    const int tile = ga - vd.tile_base;
    const int tx = tile % vd.tiles_x, ty = tile / vd.tiles_x;
    const int lane = threadIdx.x & 31, bw = threadIdx.x >> 5;
    const int w = ((int)blockIdx.x - tb * bpt) * kCompWarps + bw;   // sub-tile within the tile
    const int sub_cols = P.tile_w >> 3;        // 8-pixel-wide sub-tiles per tile row
    const int wx0 = tx * P.tile_w + (w % sub_cols) * 8, wy0 = ty * P.tile_h + (w / sub_cols) * 4;
    const int wx1 = min(wx0 + 7, vd.W - 1), wy1 = min(wy0 + 3, vd.H - 1);
    if (wx0 > wx1 || wy0 > wy1) return;        // sub-tile outside the image
    const int px = wx0 + (lane & 7), py = wy0 + (lane >> 3);
    const bool inside = px < vd.W && py < vd.H;
    const float2 f = make_float2((float)px + 0.5f, (float)py + 0.5f);
    const uint2 range = ranges[gt];
    // T < 0 marks a pixel that has ended; its transmittance is then -T
    float T = inside ? 1.f : -1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f, D = 0.f;
    // compared as integers: an ended pixel's negative value (-0 too) is below every t_min >= 0
    const int tmin = __float_as_int(P.t_min + 0.f);
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t wbit = 1u << (kTileBits + w);
    float4* const sr0 = s_rec[bw][0];
    float4* const sr1 = s_rec[bw][1];
    float4* const sr2 = s_rec[bw][2];
    uint32_t* const queue = s_queue[bw];
    uint32_t n_eval = 0, n_reach = 0, n_comp = 0;

    // the next scan step's keys and instance numbers, loaded one step ahead
    uint32_t base = range.x, kk[kScan], vv[kScan];
    auto prefetch = [&]() {
#pragma unroll
        for (int j = 0; j < kScan; ++j) {
            const uint32_t i = base + 32u * j + lane;
            kk[j] = 0u;
            vv[j] = 0u;
            if (i < range.y) { kk[j] = __ldg(keys + i); vv[j] = __ldg(vals + i); }
        }
    };
    prefetch();
    uint32_t head = 0, tail = 0, seg = 0;       // queue ends; list segment being scanned
    // scans the list until a batch of 32 selected entries is queued, or the segment (CK) or list
    // ends; returns the size of the next batch (0: the list is done)
    auto next_batch = [&]() -> int {
        for (;;) {
            const uint32_t limit = CK ? min(range.y, range.x + (seg + 1) * kSegEntries) : range.y;
            while (tail - head < 32u && base < limit) {
#pragma unroll
                for (int j = 0; j < kScan; ++j) {
                    // (debug builds check every entry of the range, whichever sub-tiles it reaches)
                    const bool ok = !kDebugChecks || base + 32u * j + lane >= range.y ||
                                    in_bounds(vv[j], P.n_rec, P.err, kSiteCompositeRecord);
                    const bool rel = (kk[j] & wbit) && ok;
                    const uint32_t m = __ballot_sync(0xffffffffu, rel);
                    if (rel) queue[(tail + __popc(m & lt)) & (kQueue - 1)] = vv[j];
                    tail += __popc(m);
                }
                base += 32u * kScan;
                prefetch();
            }
            if (tail != head) break;
            if (base >= range.y) return 0;
            ++seg;                              // CK only: an empty segment
        }
        __syncwarp();
        return (int)min(tail - head, 32u);
    };
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), q = a, col = a;
    auto gather = [&](int n) {                  // lane k: record of the batch's k-th entry
        if (lane < n) {
            const Record* r = rec + queue[(head + lane) & (kQueue - 1)];
            a = r->r0; q = r->r1; col = r->r2;
        }
        head += n;
    };
    int n = next_batch();
    uint32_t bseg = seg, cseg = 0;              // segment of the batch; last segment with a checkpoint
    if (n) gather(n);
    while (n) {
        // stage the gathered batch, padded to 32 with records that reach no pixel
        __syncwarp();
        const bool live = lane < n;
        sr0[lane] = live ? make_float4(-a.x, -a.y, kHalfLog2e * q.x, kHalfLog2e * q.z) : make_float4(0.f, 0.f, 0.f, 0.f);
        sr1[lane] = live ? make_float4(q.y, reach_threshold(P, a.z), a.z, 0.f) : make_float4(0.f, INFINITY, 0.f, 0.f);
        sr2[lane] = live ? make_float4(col.x, col.y, col.z, a.w) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (CK && bseg != cseg) {               // checkpoints of the segments entered since
            const int n_sub = P.tile_w * P.tile_h / 32;
            for (uint32_t sg = cseg + 1; sg <= bseg; ++sg)
                ck.st[((size_t)(ck.off[gt] + sg - 1) * n_sub + w) * 32 + lane] =
                    CkState{fabsf(T), C0, C1, C2, D, T < 0.f ? 1.f : 0.f};
            cseg = bseg;
        }
        __syncwarp();
        const int nc = n;
        n = next_batch();
        bseg = seg;
        if (n) gather(n);
        if (COUNT) n_eval += T < 0.f ? 0u : (uint32_t)nc;
        for (int k = 0; k < nc; k += kBlend) {
            float al[kBlend];
            bool reach[kBlend];                 // COUNT: inside the 3-sigma ellipse
#pragma unroll
            for (int u = 0; u < kBlend; ++u) {
                const float4 g0 = sr0[k + u], g1 = sr1[k + u];
                const float2 d = add2(f, make_float2(g0.x, g0.y));
                const float t = fmaf(g1.x, d.y, d.x);
                const float2 m = mul2(make_float2(g0.z, g0.w), make_float2(t, d.y));
                const float pe = fmaf(m.x, t, m.y * d.y);
                if (COUNT) reach[u] = pe >= P.p_min;
                al[u] = pe >= g1.y ? fminf(P.alpha_max, g1.z * fast_exp2(pe)) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < kBlend; ++u) {
                const float4 g2 = sr2[k + u];
                const float Tn = fmaf(-al[u], T, T);    // T (1 - alpha), one rounding
                const float wgt = al[u] * T;
                const bool go = __float_as_int(Tn) >= tmin;
                if (COUNT && reach[u] && T >= 0.f) ++n_reach;
                if (COUNT && go && al[u] > 0.f) ++n_comp;
                if (go) {
                    const float2 c01 = fma2(make_float2(wgt, wgt), make_float2(g2.x, g2.y), make_float2(C0, C1));
                    const float2 c2d = fma2(make_float2(wgt, wgt), make_float2(g2.z, g2.w), make_float2(C2, D));
                    C0 = c01.x; C1 = c01.y; C2 = c2d.x; D = c2d.y;
                }
                T = go ? Tn : __int_as_float(__float_as_int(T) | 0x80000000);   // (-|T|)
            }
            if (__all_sync(0xffffffffu, T < 0.f)) { n = 0; break; }
        }
    }
    if (CK && lane == 0) ck.last[(size_t)gt * (P.tile_w * P.tile_h / 32) + w] = cseg + 1;
    T = fabsf(T);
    if (COUNT) {
        const uint32_t a = __reduce_add_sync(0xffffffffu, n_eval), b = __reduce_add_sync(0xffffffffu, n_reach),
                       cc = __reduce_add_sync(0xffffffffu, n_comp);
        if (lane == 0) { atomicAdd(work + 0, a); atomicAdd(work + 1, b); atomicAdd(work + 2, cc); }
    }
    if (inside) {
        const int64_t p = vd.pix_off + (int64_t)py * vd.W + px;
        float r = fmaf(P.bg0, T, C0), g = fmaf(P.bg1, T, C1), b = fmaf(P.bg2, T, C2);
        if (AUG) {
            const dgs_augment& a = P.aug[lo];
            augment_pixel(a, a.overlay_beta != 0.f ? overlay_pixel(P.overlay, P.ov_w, P.ov_h, a, px, py) : nullptr,
                          r, g, b);
        }
        out_rgb[p * 3 + 0] = r;
        out_rgb[p * 3 + 1] = g;
        out_rgb[p * 3 + 2] = b;
        out_depth[p] = D;
        if (out_alpha) out_alpha[p] = 1.f - T;
    }
}

}  // namespace

void launch_ranges(const Launch& L, const uint32_t* keys, uint32_t n, uint2* ranges, int n_tiles,
                   const uint32_t* d_n, const ViewDesc* views, int nv, const Params& P) {
    if (n == 0) return;
    const uint32_t threads = (n + 3) / 4;
    const uint32_t blocks = std::min<uint32_t>((threads + 255) / 256, sm_count() * 8u);
    k_ranges<<<blocks, 256, 0, L.stream>>>(keys, n, d_n, ranges, n_tiles, views, (int)P.view0, nv,
                                                          P.tile0, P.tbits);
    ++*L.launches;
}

void launch_tile_order(const Launch& L, const uint2* ranges, int n_tiles, uint32_t* order, uint32_t* scratch) {
    if (n_tiles == 0) return;
    if (n_tiles <= kOrderOneBlock) {
        k_tile_order<<<1, 1024, 0, L.stream>>>(ranges, n_tiles, order);
        ++*L.launches;
        return;
    }
    const unsigned blocks = (unsigned)((n_tiles + 255) / 256);
    k_order_count<<<blocks, 256, 0, L.stream>>>(ranges, n_tiles, scratch, scratch + 256);
    k_order_place<<<blocks, 256, 0, L.stream>>>(ranges, n_tiles, scratch, order);
    *L.launches += 2;
}

void launch_segment_jobs(const Launch& L, const uint2* ranges, int n_tiles, const Checkpoints& ck) {
    if (n_tiles == 0) {
        cudaMemsetAsync(ck.n_jobs, 0, sizeof(uint32_t), L.stream);
        return;
    }
    k_segment_jobs<<<1, 1024, 0, L.stream>>>(ranges, n_tiles, ck);
    ++*L.launches;
}

void launch_composite(const Launch& L, const ViewDesc* views, int v0, int n_group_views, int n_tiles,
                      const uint2* ranges, const uint32_t* keys, const uint32_t* vals, const Record* records,
                      const Params& P, float* out_rgb, float* out_depth, float* out_alpha, unsigned long long* work,
                      const uint32_t* tile_order, const Checkpoints& ck) {
    if (n_tiles == 0) return;
    // checkpoints are for the adjoint, which never runs on randomised outputs
    const bool with_ck = ck.st != nullptr && !P.aug;
    // few waves: fewer resident blocks with more registers shorten the longest lists' chains; many waves:
    // the most blocks that fit.  The lines are in blocks (four to a 16x16 tile, one to an 8x8).  One-group
    // times with 14 against 16 blocks an SM, us: 28,800 blocks 123 / 129, 38,400 145 / 141, 76,800 289 / 281 (tiles of
    // 8x8: 19,200 98 / 107, 38,400 172 / 176, 57,600 256 / 254); with randomisation 38,400 152 / 168, 57,600 229 / 227;
    // with checkpoints (60 bytes of spills at 16) 38,400 147 / 178, 76,800 295 / 305, 153,600 625 / 614.
    const int bpt = (P.tile_w * P.tile_h) / (32 * kCompWarps);
    const bool few = (int64_t)n_tiles * bpt <= (with_ck ? 98304 : P.aug ? 49152 : 32768);
    auto* kern = with_ck ? (work ? k_composite<true, false, true, 16> : few ? k_composite<false, false, true, 14>
                                                                           : k_composite<false, false, true, 16>)
                 : work  ? (P.aug ? k_composite<true, true, false, 16> : k_composite<true, false, false, 16>)
                 : few   ? (P.aug ? k_composite<false, true, false, 14> : k_composite<false, false, false, 14>)
                         : (P.aug ? k_composite<false, true, false, 16> : k_composite<false, false, false, 16>);
    kern<<<n_tiles * bpt, kCompWarps * 32, 0, L.stream>>>(views, v0, n_group_views, ranges, keys, vals, records, P,
                                                          out_rgb, out_depth, out_alpha, work, tile_order, ck);
    ++*L.launches;
}

}  // namespace dgs
