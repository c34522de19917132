// LiDAR by Gaussian ray tracing through a per-node BVH (Sec. III-C: LiDAR is simulated by
// native ray tracing of the scene's Gaussians, accelerated by a BVH).
//
// Per ray o + t d (|d| = 1) and Gaussian (mean mu, whitening M = diag(1/s) R^T in its node's
// frame): o' = M (o_n - mu), d' = M d_n; the response peaks at t* = -(o'.d')/(d'.d') with
// Mahalanobis distance q* = |o' x d'|^2 / (d'.d').  A hit needs q* <= q_max and
// r_min <= t* <= r_max; alpha = min(alpha_max, opacity exp(-q*/2)), skipped below alpha_min.
// Hits composite front to back in (t*, global id) order with the camera's termination rule;
// D = sum T alpha t*, A = 1 - T.
//
// Acceleration structure, per node (built once from the node's attributes, in its frame): a
// 64-byte record per Gaussian (mu, opacity, M) and an implicit complete binary tree over
// leaves of 8 consecutive Gaussians in storage order (heap numbering: root 1, children 2k and
// 2k+1, leaves P..2P-1), each node holding the box of the 3-sigma ellipsoids below it.  The
// tree's quality follows the storage order: Z-ordered nodes (dgs_spatial_order) give compact
// leaves.  Trees are never refitted per env: rays are moved into each node's frame instead.
//
// Tracing: one warp per ray, its lanes testing 32 boxes or 32 Gaussians at a time (k_lidar_trace); in
// dense beam patterns one warp per packet of 32 neighbouring rays (k_lidar_packets).
#include <algorithm>

#include "dgs_internal.cuh"

namespace dgs {
namespace {

constexpr int kLeaf = 8;             // Gaussians per leaf

__device__ __forceinline__ float sigmoidf(float x) { return 1.f / (1.f + __expf(-x)); }

// Records and leaf boxes of one node: thread i = Gaussian i (threads past n give empty boxes),
// lanes 8j..8j+7 of a warp reduce the box of leaf j.
template <int DT>
__global__ void k_lidar_records(NodeDesc nd, float sq, float4* __restrict__ rec, float4* __restrict__ box,
                                int64_t P) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (i < nd.n) {
        const float mx = nd.mean[3 * i], my = nd.mean[3 * i + 1], mz = nd.mean[3 * i + 2];
        float qw = ld_attr<DT>(nd.quat, 4 * i), qx = ld_attr<DT>(nd.quat, 4 * i + 1),
              qy = ld_attr<DT>(nd.quat, 4 * i + 2), qz = ld_attr<DT>(nd.quat, 4 * i + 3);
        const float qn = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
        qw *= qn; qx *= qn; qy *= qn; qz *= qn;
        const float R[3][3] = {{1.f - 2.f * (qy * qy + qz * qz), 2.f * (qx * qy - qw * qz), 2.f * (qx * qz + qw * qy)},
                               {2.f * (qx * qy + qw * qz), 1.f - 2.f * (qx * qx + qz * qz), 2.f * (qy * qz - qw * qx)},
                               {2.f * (qx * qz - qw * qy), 2.f * (qy * qz + qw * qx), 1.f - 2.f * (qx * qx + qy * qy)}};
        float s[3], is[3];
        for (int a = 0; a < 3; ++a) {
            const float l = ld_attr<DT>(nd.log_scale, 3 * i + a);
            s[a] = expf(l);
            is[a] = expf(-l);
        }
        float M[3][3];
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) M[a][b] = R[b][a] * is[a];
        const float op = sigmoidf(nd.opac[i]);
        rec[4 * i + 0] = make_float4(mx, my, mz, op);
        rec[4 * i + 1] = make_float4(M[0][0], M[0][1], M[0][2], M[1][0]);
        rec[4 * i + 2] = make_float4(M[1][1], M[1][2], M[2][0], M[2][1]);
        // squared radius of the sphere holding the q_max ellipsoid: a ray farther from the mean
        // than that cannot hit (cheap test before the exact one)
        const float smax = fmaxf(fmaxf(s[0], s[1]), s[2]);
        rec[4 * i + 3] = make_float4(M[2][2], sq * sq * smax * smax * 1.002f, 0.f, 0.f);
        const float m[3] = {mx, my, mz};
        for (int a = 0; a < 3; ++a) {
            // half extent of the ellipsoid q <= q_max along axis a, widened slightly so that
            // rounding never drops a hit the exact test keeps
            const float h = sq * sqrtf(R[a][0] * R[a][0] * s[0] * s[0] + R[a][1] * R[a][1] * s[1] * s[1] +
                                       R[a][2] * R[a][2] * s[2] * s[2]);
            const float hw = fmaf(h, 1.001f, 1e-6f + 1e-6f * fabsf(m[a]));
            lo[a] = m[a] - hw;
            hi[a] = m[a] + hw;
        }
    }
#pragma unroll
    for (int o = 1; o < kLeaf; o <<= 1) {
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    }
    const int64_t leaf = i / kLeaf;
    if ((i & (kLeaf - 1)) == 0 && leaf < P) {
        box[2 * (P + leaf)] = make_float4(lo[0], lo[1], lo[2], 0.f);
        box[2 * (P + leaf) + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
}

// One tree level of every tree that has it: node k in [h, 2h) = union of its children.
struct LevelJob {
    float4* box;
    int64_t first;           // first thread of this tree in the launch
};

__global__ void k_lidar_level(const LevelJob* __restrict__ jobs, int n_jobs, int64_t h, int64_t total) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].first <= t) lo = mid; else hi = mid - 1;
    }
    float4* box = jobs[lo].box;
    const int64_t k = h + (t - jobs[lo].first);
    const float4 a0 = box[4 * k], a1 = box[4 * k + 1], b0 = box[4 * k + 2], b1 = box[4 * k + 3];
    box[2 * k] = make_float4(fminf(a0.x, b0.x), fminf(a0.y, b0.y), fminf(a0.z, b0.z), 0.f);
    box[2 * k + 1] = make_float4(fmaxf(a1.x, b1.x), fmaxf(a1.y, b1.y), fmaxf(a1.z, b1.z), 0.f);
}

// A sensor's beam j: its unit direction.
__device__ __forceinline__ void sensor_ray(const float* __restrict__ dirs, int64_t j, float (&ds)[3]) {
    ds[0] = dirs[3 * j]; ds[1] = dirs[3 * j + 1]; ds[2] = dirs[3 * j + 2];
    const float r = rsqrtf(ds[0] * ds[0] + ds[1] * ds[1] + ds[2] * ds[2]);
    ds[0] *= r; ds[1] *= r; ds[2] *= r;
}

// The packets of 32 rays, one per warp of the block: those whose directions lie within `cone` of their mean
// are listed to be traced together (k_lidar_packets), the others to be left to k_lidar_trace; counts =
// their numbers, to which a block adds once.
__device__ __forceinline__ void list_packets(uint32_t block, const float* __restrict__ dirs, int n_dirs,
                                             int64_t n_rays, const LidarPackets& L) {
    __shared__ uint32_t s_near[32], s_first[2];
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, full = 0xffffffffu;
    const int64_t ray0 = ((int64_t)block * 32 + warp) * 32, j0 = ray0 % n_dirs;
    bool near = ray0 + 32 <= n_rays && j0 + 32 <= n_dirs;            // 32 rays of one sensor
    if (near) {
        float ds[3], m[3];
        sensor_ray(dirs, j0 + lane, ds);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            m[a] = ds[a];
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) m[a] += __shfl_xor_sync(full, m[a], o);
        }
        const float r = rsqrtf(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
        const float e0 = ds[0] - m[0] * r, e1 = ds[1] - m[1] * r, e2 = ds[2] - m[2] * r;
        near = __all_sync(full, fmaf(e0, e0, fmaf(e1, e1, e2 * e2)) <= L.cone * L.cone);
    }
    if (lane == 0) s_near[warp] = near;
    __syncthreads();
    if (warp != 0) return;
    const uint32_t pk = block * 32u + lane;
    const bool in = pk < L.n && s_near[lane], out = pk < L.n && !in;
    const uint32_t m_in = __ballot_sync(full, in), m_out = __ballot_sync(full, out);
    if (lane < 2) {
        const uint32_t n = __popc(lane ? m_out : m_in);
        s_first[lane] = n ? atomicAdd(L.counts + lane, n) : 0u;
    }
    __syncwarp();
    const uint32_t below = (1u << lane) - 1u;
    if (in) L.together[s_first[0] + __popc(m_in & below)] = pk;
    if (out) L.left[s_first[1] + __popc(m_out & below)] = pk;
}

// Per (sensor, slot): the sensor's rotation and origin expressed in the node's frame.  The blocks from
// setup_blocks on list the packets.
constexpr int kSetupThreads = 1024;
__global__ void __launch_bounds__(kSetupThreads) k_lidar_setup(const LidarSensorDev* __restrict__ sensors, int S,
                                                               const int32_t* __restrict__ slot_node, int K,
                                                               const float* __restrict__ node_poses,
                                                               LidarSlot* __restrict__ out, uint32_t* __restrict__ err,
                                                               unsigned setup_blocks, const float* __restrict__ dirs,
                                                               int n_dirs, int64_t n_rays, LidarPackets packets) {
    if (blockIdx.x >= setup_blocks) {
        list_packets(blockIdx.x - setup_blocks, dirs, n_dirs, n_rays, packets);
        return;
    }
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= S * K) return;
    const int s = idx / K, j = idx % K;
    const LidarSensorDev& sd = sensors[s];
    LidarSlot o;
    o.node = slot_node[sd.env * K + j];
    if (o.node >= 0) {
        const float* W = node_poses + ((int64_t)sd.env * K + j) * 12;
        float Wm[12];
        bool ok = true;
        for (int a = 0; a < 12; ++a) {
            Wm[a] = W[a];
            ok &= isfinite(Wm[a]);
        }
        for (int a = 0; a < 3 && ok; ++a)
            for (int b = 0; b < 3; ++b) {
                const float d = Wm[a] * Wm[b] + Wm[4 + a] * Wm[4 + b] + Wm[8 + a] * Wm[8 + b];
                ok &= fabsf(d - (a == b ? 1.f : 0.f)) <= 1e-4f;
            }
        if (!ok) {
            atomicOr(err, kErrPose);
            o.node = -1;
        } else {
            // node_from_sensor = (world_from_node)^-1 world_from_sensor
            const float* P = sd.pose;
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b)
                    o.R[3 * a + b] = Wm[a] * P[b] + Wm[4 + a] * P[4 + b] + Wm[8 + a] * P[8 + b];
            const float v0 = P[3] - Wm[3], v1 = P[7] - Wm[7], v2 = P[11] - Wm[11];
            for (int a = 0; a < 3; ++a) o.o[a] = Wm[a] * v0 + Wm[4 + a] * v1 + Wm[8 + a] * v2;
        }
    }
    out[idx] = o;
}

__device__ __forceinline__ bool slab(const float4 lo, const float4 hi, const float o[3], const float id[3], float t_lo,
                                     float t_hi) {
    if (lo.x > hi.x) return false;                   // empty box
    const float x0 = (lo.x - o[0]) * id[0], x1 = (hi.x - o[0]) * id[0];
    const float y0 = (lo.y - o[1]) * id[1], y1 = (hi.y - o[1]) * id[1];
    const float z0 = (lo.z - o[2]) * id[2], z1 = (hi.z - o[2]) * id[2];
    // fminf/fmaxf drop the NaN of 0 * inf (ray parallel to a slab through its origin)
    const float enter = fmaxf(fmaxf(fminf(x0, x1), fminf(y0, y1)), fmaxf(fminf(z0, z1), t_lo));
    const float exit = fminf(fminf(fmaxf(x0, x1), fmaxf(y0, y1)), fminf(fmaxf(z0, z1), t_hi));
    return enter <= exit;
}

__device__ __forceinline__ float slab_enter(const float4 lo, const float4 hi, const float o[3], const float id[3]) {
    const float x0 = (lo.x - o[0]) * id[0], x1 = (hi.x - o[0]) * id[0];
    const float y0 = (lo.y - o[1]) * id[1], y1 = (hi.y - o[1]) * id[1];
    const float z0 = (lo.z - o[2]) * id[2], z1 = (hi.z - o[2]) * id[2];
    return fmaxf(fmaxf(fminf(x0, x1), fminf(y0, y1)), fminf(z0, z1));
}

// Per-warp state in shared memory: the traversal stack (heap index, slot and entry distance of
// every node still to visit) and the pending hits (bits of t*, global id, alpha), unsorted.
constexpr int kRayWarps = 4;         // warps (rays in flight) per block
constexpr int kStack = 256;          // 32 roots + 31 per expansion, at most 7 expansions deep: 249
constexpr int kPend = 128;           // pending hits
constexpr int kPendRegs = kPend / 32;
constexpr int kKeep = 64;            // hits kept when the pending buffer is cut
struct RayWarp {
    uint32_t node[kStack], slot[kStack];
    float enter[kStack];
    uint32_t t[kPend], g[kPend];
    float a[kPend];
};

// A ray in a slot's node frame.
struct NodeRay {
    float o[3], d[3], id[3];
};

__device__ __forceinline__ NodeRay node_ray(const LidarSlot& S, const float (&ds)[3]) {
    NodeRay r;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        r.o[a] = S.o[a];
        r.d[a] = S.R[3 * a] * ds[0] + S.R[3 * a + 1] * ds[1] + S.R[3 * a + 2] * ds[2];
        r.id[a] = 1.f / r.d[a];
    }
    return r;
}

// A ray against the Gaussian of record (r0, r1, r2, r3): whether its peak lies within q_max and the
// range window, with its distance t and Mahalanobis distance q.
__device__ __forceinline__ bool peak(const float4 r0, const float4 r1, const float4 r2, const float4 r3, const NodeRay& R,
                                     const LidarParams& LP, float& t, float& q) {
    const float v0 = R.o[0] - r0.x, v1 = R.o[1] - r0.y, v2 = R.o[2] - r0.z;
    const float x0 = fmaf(v1, R.d[2], -v2 * R.d[1]), x1 = fmaf(v2, R.d[0], -v0 * R.d[2]),
                x2 = fmaf(v0, R.d[1], -v1 * R.d[0]);
    if (fmaf(x0, x0, fmaf(x1, x1, x2 * x2)) > r3.y) return false;   // |d| = 1 up to rounding
    const float op0 = fmaf(r1.x, v0, fmaf(r1.y, v1, r1.z * v2));
    const float op1 = fmaf(r1.w, v0, fmaf(r2.x, v1, r2.y * v2));
    const float op2 = fmaf(r2.z, v0, fmaf(r2.w, v1, r3.x * v2));
    const float dp0 = fmaf(r1.x, R.d[0], fmaf(r1.y, R.d[1], r1.z * R.d[2]));
    const float dp1 = fmaf(r1.w, R.d[0], fmaf(r2.x, R.d[1], r2.y * R.d[2]));
    const float dp2 = fmaf(r2.z, R.d[0], fmaf(r2.w, R.d[1], r3.x * R.d[2]));
    const float dd = fmaf(dp0, dp0, fmaf(dp1, dp1, dp2 * dp2));
    const float od = fmaf(op0, dp0, fmaf(op1, dp1, op2 * dp2));
    const float c0 = fmaf(op1, dp2, -op2 * dp1), c1 = fmaf(op2, dp0, -op0 * dp2), c2 = fmaf(op0, dp1, -op1 * dp0);
    const float idd = 1.f / dd;
    t = fmaf(-od, idd, 0.f);           // never -0, whose bits would order it last
    q = fmaf(c0, c0, fmaf(c1, c1, c2 * c2)) * idd;
    return q <= LP.q_max && t >= LP.r_min && t <= LP.r_max;
}

__device__ __forceinline__ float hit_alpha(float opacity, float q, const LidarParams& LP) {
    return fminf(LP.alpha_max, opacity * fast_exp2(kHalfLog2e * q));
}

// Pushes the lanes with `in` set onto the stack, nearest entry on top (ties by lane).
__device__ __forceinline__ void push_sorted(RayWarp& W, int& sp, bool in, float enter, uint32_t node, uint32_t slot, int lane) {
    const unsigned m = __ballot_sync(0xffffffffu, in);
    int rank = 0;
    for (unsigned rest = m; rest; rest &= rest - 1) {
        const int src = __ffs(rest) - 1;
        const float e = __shfl_sync(0xffffffffu, enter, src);
        rank += e < enter || (e == enter && src < lane);
    }
    const int n = __popc(m);
    if (in) {
        const int at = sp + n - 1 - rank;
        W.node[at] = node;
        W.slot[at] = slot;
        W.enter[at] = enter;
    }
    sp += n;
    __syncwarp();
}

// The pending hits in registers, entry 32 q + lane in slot q (key ~0: none), and back.
__device__ __forceinline__ void load_pending(const RayWarp& W, int cnt, int lane, uint64_t (&key)[kPendRegs], float (&al)[kPendRegs]) {
#pragma unroll
    for (int q = 0; q < kPendRegs; ++q) {
        const int i = 32 * q + lane;
        key[q] = i < cnt ? ((uint64_t)W.t[i] << 32) | W.g[i] : ~0ull;
        al[q] = i < cnt ? W.a[i] : 0.f;
    }
    __syncwarp();
}

__device__ __forceinline__ int store_pending(RayWarp& W, int lane, const uint64_t (&key)[kPendRegs], const float (&al)[kPendRegs]) {
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < kPendRegs; ++q) {
        const bool live = key[q] != ~0ull;
        const unsigned m = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int at = cnt + __popc(m & ((1u << lane) - 1u));
            W.t[at] = (uint32_t)(key[q] >> 32);
            W.g[at] = (uint32_t)key[q];
            W.a[at] = al[q];
        }
        cnt += __popc(m);
    }
    __syncwarp();
    return cnt;
}

// Composites the pending hits with t* < bound in (t*, id) order, one warp-wide minimum per hit,
// and keeps the others.  Returns true when the transmittance ends the ray.
__device__ __forceinline__ bool composite_pending(RayWarp& W, int& cnt, float bound, float t_min, int lane, float& T, float& D) {
    uint64_t key[kPendRegs];
    float al[kPendRegs];
    load_pending(W, cnt, lane, key, al);
    bool done = false;
    for (;;) {
        uint64_t mine = key[0];
        float a = al[0];
#pragma unroll
        for (int q = 1; q < kPendRegs; ++q)
            if (key[q] < mine) { mine = key[q]; a = al[q]; }
        const uint32_t tb = __reduce_min_sync(0xffffffffu, (uint32_t)(mine >> 32));
        if (tb == ~0u || !(__uint_as_float(tb) < bound)) break;
        const uint32_t gb = __reduce_min_sync(0xffffffffu, (uint32_t)(mine >> 32) == tb ? (uint32_t)mine : ~0u);
        const uint64_t best = ((uint64_t)tb << 32) | gb;
        a = __shfl_sync(0xffffffffu, a, __ffs(__ballot_sync(0xffffffffu, mine == best)) - 1);
        const float Tn = fmaf(-a, T, T);
        if (Tn < t_min) { done = true; break; }
        D = fmaf(a * T, __uint_as_float(tb), D);
        T = Tn;
#pragma unroll
        for (int q = 0; q < kPendRegs; ++q)
            if (key[q] == best) key[q] = ~0ull;
    }
    cnt = done ? 0 : store_pending(W, lane, key, al);
    return done;
}

// Keeps the kKeep nearest of more pending hits; returns the key of the farthest kept (the kKeep-th
// smallest, found bit by bit: the largest x with fewer than kKeep keys below it).
__device__ __forceinline__ uint64_t cut_pending(RayWarp& W, int& cnt, int lane) {
    uint64_t key[kPendRegs];
    float al[kPendRegs];
    load_pending(W, cnt, lane, key, al);
    uint64_t x = 0;
    for (int b = 63; b >= 0; --b) {
        const uint64_t c = x | (1ull << b);
        int below = 0;
#pragma unroll
        for (int q = 0; q < kPendRegs; ++q) below += __popc(__ballot_sync(0xffffffffu, key[q] < c));
        if (below < kKeep) x = c;
    }
#pragma unroll
    for (int q = 0; q < kPendRegs; ++q)
        if (key[q] > x) key[q] = ~0ull;
    cnt = store_pending(W, lane, key, al);
    return x;
}

// Whether the packets listed as together (counts[0]) are traced so: half of all at least.  Fewer leave
// both kernels too little to do, one after the other.
__device__ __forceinline__ bool packets_taken(const uint32_t* counts, int64_t n_rays) {
    return 64ll * counts[0] >= n_rays;
}

// Warp = one ray at a time; persistent warps take the next ray from a counter.  Beams of a
// sensor are farther apart, at the distances where they hit, than the Gaussians are wide, so
// neighbouring rays share few leaves: the 32 lanes work on one ray instead, 32 boxes or 32
// Gaussians per step.
//   expand   the 2^s (s <= 4) descendants of a node s levels down are consecutive in heap
//            numbering: one box per lane, one coalesced load; those the ray's interval meets (two
//            on average) are pushed nearest on top.  Two nodes of a tree on top of the stack are
//            expanded together, 16 lanes each.  The first expansion of a tree takes the levels
//            that do not divide by four, so that the last ones before the leaves are full.
//   leaves   up to four leaves on top of the stack, 8 lanes each: one Gaussian per lane; hits go
//            to the pending buffer.
//   flush    a hit is final once its t* lies before the entry of every node still on the stack;
//            final hits are composited in (t*, id) order, so one traversal composites the whole
//            ray and ends as soon as the transmittance does.
// When the pending buffer fills with hits that are not final, the nearest kKeep stay, nodes and
// hits beyond them are skipped, and another round resumes after them.  The trees of up to 32
// slots share one stack; with more, a slot batch is traversed after the other and hits are
// final at the end of the round only.
// Bound by latency (boxes and records come from L2, one dependent load per step); 64 registers keep 32
// warps an SM.  Same outputs bit for bit: one sensor of 32 x 1024 beams through 380k Gaussians and 16
// sensors through 580k took 9-15 and 20-33 ms (by scene) with a packet of 32 rays per warp, where the
// slowest packet is the time; one ray per warp, one node of five levels per expansion, 72 registers
// 0.592 and 5.59 ms; two nodes 0.588 and 5.51; with 64 registers 0.555 and 5.04.
//
// LISTED: the rays are those of the packets that are not traced together, or that k_lidar_packets left.
template <bool LISTED>
__global__ void __launch_bounds__(kRayWarps * 32, 8) k_lidar_trace(const LidarTreeDev* __restrict__ trees,
                                                                const LidarSlot* __restrict__ slots, int K,
                                                                const float* __restrict__ dirs, int n_dirs,
                                                                int64_t n_rays, LidarParams LP,
                                                                float* __restrict__ out_d, float* __restrict__ out_a,
                                                                uint32_t* __restrict__ err,
                                                                unsigned long long* __restrict__ next_ray,
                                                                const uint32_t* __restrict__ left,
                                                                const uint32_t* __restrict__ counts) {
    __shared__ RayWarp s_warp[kRayWarps];
    const int lane = threadIdx.x & 31;
    RayWarp& W = s_warp[threadIdx.x >> 5];
    const bool some = LISTED && packets_taken(counts, n_rays);   // (else all rays, in order)
    for (;;) {
        unsigned long long ray = 0;
        if (lane == 0) ray = atomicAdd(next_ray, 1ull);
        ray = __shfl_sync(0xffffffffu, ray, 0);
        if (ray >= (some ? 32ull * __ldg(counts + 1) : (unsigned long long)n_rays)) break;
        if (some) ray = 32ull * left[ray >> 5] + (ray & 31ull);
        if (some && ray >= (unsigned long long)n_rays) continue;
        const int64_t s = (int64_t)ray / n_dirs, j = (int64_t)ray - s * n_dirs;
        float ds[3];
        sensor_ray(dirs, j, ds);
        const LidarSlot* sl = slots + s * K;
        float T = 1.f, D = 0.f;
        uint64_t last = 0;                             // keys <= last are composited
        bool first = true, done = false;
        while (!done) {                                // a round: nearly always the only one
            const float t_lo = first ? LP.r_min : __uint_as_float((uint32_t)(last >> 32));
            float t_hi = LP.r_max;
            uint64_t maxkey = ~0ull;                   // farthest kept key once the buffer was cut
            int cnt = 0, sp = 0, next_slot = 0, flush_at = 32, cur = -1;
            NodeRay R{};
            LidarTreeDev tr{};
            int levels = 0;
            while (!done) {
                if (sp == 0) {
                    if (next_slot >= K) break;
                    // the roots of the next 32 slots, one per lane
                    const int slot = next_slot + lane;
                    bool in = false;
                    float en = 0.f;
                    if (slot < K) {
                        const LidarSlot& S = sl[slot];
                        if (S.node >= 0 && trees[S.node].n > 0) {
                            const NodeRay r = node_ray(S, ds);
                            const float4 lo = trees[S.node].box[2], hi = trees[S.node].box[3];
                            in = slab(lo, hi, r.o, r.id, t_lo, t_hi);
                            en = fmaxf(slab_enter(lo, hi, r.o, r.id), t_lo) + 0.f;   // (never -0: ordered as bits below)
                        }
                    }
                    __syncwarp();
                    push_sorted(W, sp, in, en, 1u, (uint32_t)slot, lane);
                    next_slot += 32;
                    continue;
                }
                const uint32_t node = W.node[sp - 1], slot = W.slot[sp - 1];
                const float enter = W.enter[sp - 1];
                if (enter > t_hi) { --sp; continue; }
                if ((int)slot != cur) {
                    cur = (int)slot;
                    const LidarSlot& S = sl[cur];
                    R = node_ray(S, ds);
                    tr = trees[S.node];
                    levels = 63 - __clzll(tr.P);
                }
                if ((int64_t)node < tr.P) {
                    // the node below on the stack too, if it is an inner one of the same tree
                    const int at2 = max(sp - 2, 0);
                    const uint32_t node2 = W.node[at2];
                    const bool pair = sp >= 2 && W.slot[at2] == slot && (int64_t)node2 < tr.P && W.enter[at2] <= t_hi;
                    const uint32_t mine = lane >= 16 ? node2 : node;
                    const int below = levels - (31 - __clz(mine));          // levels left to the leaves, >= 1
                    const int st = below % 4 ? below % 4 : 4, sub = lane & 15;
                    const uint32_t child = (mine << st) + (uint32_t)sub;
                    sp -= pair ? 2 : 1;
                    bool in = false;
                    float en = 0.f;
                    if (sub < (1 << st) && (lane < 16 || pair)) {
                        const float4 lo = __ldg(tr.box + 2 * (size_t)child), hi = __ldg(tr.box + 2 * (size_t)child + 1);
                        in = slab(lo, hi, R.o, R.id, t_lo, t_hi);
                        en = fmaxf(slab_enter(lo, hi, R.o, R.id), t_lo) + 0.f;
                    }
                    __syncwarp();                      // every lane has read the popped entry
                    if (sp + 32 > kStack) {            // cannot happen for trees of the documented sizes
                        if (lane == 0) atomicOr(err, kErrCapacity);
                        done = true;
                        break;
                    }
                    push_sorted(W, sp, in, en, child, slot, lane);
                    continue;
                }
                // the leaves of this slot on top of the stack, at most four
                const int at = sp - 1 - lane;
                const unsigned lm = __ballot_sync(0xffffffffu, lane < 4 && at >= 0 && W.slot[max(at, 0)] == slot &&
                                                                   (int64_t)W.node[max(at, 0)] >= tr.P);
                const int nl = __ffs(~lm) - 1, li = lane >> 3;
                int64_t g = -1;
                if (li < nl && W.enter[sp - 1 - li] <= t_hi)
                    g = ((int64_t)W.node[sp - 1 - li] - tr.P) * kLeaf + (lane & (kLeaf - 1));
                sp -= nl;
                __syncwarp();
                bool hit = false;
                float t = 0.f, alpha = 0.f;
                if (g >= 0 && g < tr.n) {
                    const float4* rp = tr.rec + 4 * g;
                    const float4 r0 = __ldg(rp), r1 = __ldg(rp + 1), r2 = __ldg(rp + 2), r3 = __ldg(rp + 3);
                    float q;
                    if (peak(r0, r1, r2, r3, R, LP, t, q)) {
                        const uint64_t key = ((uint64_t)__float_as_uint(t) << 32) | (uint32_t)(tr.gbase + g);
                        if ((first || key > last) && key < maxkey) {
                            alpha = hit_alpha(r0.w, q, LP);
                            hit = alpha >= LP.alpha_min;
                        }
                    }
                }
                const unsigned hm = __ballot_sync(0xffffffffu, hit);
                if (hm == 0) continue;
                if (hit) {
                    const int p = cnt + __popc(hm & ((1u << lane) - 1u));
                    W.t[p] = __float_as_uint(t);
                    W.g[p] = (uint32_t)(tr.gbase + g);
                    W.a[p] = alpha;
                }
                cnt += __popc(hm);
                __syncwarp();
                if (cnt < flush_at) continue;
                // final hits: before the entry of every node left, less a margin for the rounding of
                // the boxes' entries and of t* (hits of unvisited slots may lie anywhere)
                if (next_slot >= K) {
                    float bound = INFINITY;
                    for (int i = lane; i < sp; i += 32) bound = fminf(bound, W.enter[i]);
                    bound = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(bound)));   // >= 0: ordered as bits
                    done = composite_pending(W, cnt, fmaf(bound, 1.f - 1e-5f, -1e-5f), LP.t_min, lane, T, D);
                    if (done) break;
                }
                if (cnt > kPend - 32) {
                    maxkey = cut_pending(W, cnt, lane);
                    t_hi = __uint_as_float((uint32_t)(maxkey >> 32));
                }
                flush_at = min(cnt + 24, kPend - 31);
            }
            if (done) break;
            if (composite_pending(W, cnt, INFINITY, LP.t_min, lane, T, D) || maxkey == ~0ull) break;
            last = maxkey;
            first = false;
        }
        if (lane == 0) {
            out_d[ray] = D;
            out_a[ray] = 1.f - T;
        }
        __syncwarp();
    }
}

// The packets listed as together, 32 neighbouring rays of one sensor each: warp = packet, lane = ray.  The
// packet walks each tree together on a warp-uniform stack: a box is descended if any lane's interval meets
// it, the children in the order of the first such lane's entries; boxes and records are read once for
// the packet.  A lane keeps the kHits nearest hits of a round, sorted, in shared memory; a round's hits
// are composited in order and the next resumes after the last of them, until every lane's
// transmittance has ended or its hits have run out.  A packet that takes too many nodes (rays grazing a
// surface, an object's dense centre: up to 10 ms for one packet) is left to k_lidar_trace, which
// finds the same hits.
//
// Rays so close that they meet the same leaves cost k_lidar_trace 32 walks of them, 5 ns a ray with the
// chip full; a packet walks the union once.  Bound by latency (16 warps an SM, one dependent load per
// step), so packets pay where there are enough of them and their cones are narrow.  Whole calls, 300k
// Gaussians of a room, against k_lidar_trace alone: 1024 x 1024 beams over 5 x 2.5 degrees 5.10 -> 1.22 ms,
// over 160 x 80 6.89 -> 2.66; 512 x 512 over 20 x 10 1.50 -> 0.53, over 80 x 40 2.06 -> 1.40 (with four
// objects of 20k beside it 2.88 -> 3.00); 256 x 256 over 10 x 5 0.41 -> 0.21.  Not taken, for what they would
// take: 64 x 1024 over 360 x 41 degrees 0.52 against 1.23, 512 x 512 over 160 x 80 1.79 against 1.39 (with
// the objects 2.28 against 2.77).  Budgets of 512 and 2048 nodes: 1.67 and 1.28 ms for 512 x 512 over
// 80 x 40, 2.87 and 4.25 with the objects.
constexpr int kPacketThreads = 128;
constexpr int kHits = 32;
constexpr int kWalk = 64;            // a level's sibling on the stack at most: 29
constexpr int kPacketSteps = 1024;   // nodes a packet may take before its rays are left
constexpr size_t kPacketSmem = (size_t)3 * kHits * kPacketThreads * sizeof(uint32_t);   // [entry][thread]: t bits, id, alpha

__global__ void __launch_bounds__(kPacketThreads, 4) k_lidar_packets(const LidarTreeDev* __restrict__ trees,
                                                                  const LidarSlot* __restrict__ slots, int K,
                                                                  const float* __restrict__ dirs, int n_dirs,
                                                                  int64_t n_rays, LidarParams LP,
                                                                  float* __restrict__ out_d,
                                                                  float* __restrict__ out_a, uint32_t* __restrict__ err,
                                                                  LidarPackets packets) {
    __shared__ uint32_t s_stack[kPacketThreads / 32][kWalk];
    extern __shared__ uint32_t s_hits[];
    uint32_t* const kt = s_hits + threadIdx.x;                      // entry i at kt[i * kPacketThreads]
    uint32_t* const kg = kt + kHits * kPacketThreads;
    float* const ka = reinterpret_cast<float*>(kg + kHits * kPacketThreads);
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    uint32_t* const stk = s_stack[threadIdx.x >> 5];
    if (!packets_taken(packets.counts, n_rays)) return;
    for (;;) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(packets.next, 1u);
        at = __shfl_sync(full, at, 0);
        if (at >= packets.counts[0]) break;
        const uint32_t pk = packets.together[at];
        const int64_t ray0 = (int64_t)pk * 32, s = ray0 / n_dirs;
        float ds[3];
        sensor_ray(dirs, ray0 - s * n_dirs + lane, ds);
        int steps = 0;                                 // nodes taken from the stack
        const LidarSlot* sl = slots + s * K;
        float T = 1.f, D = 0.f;
        uint64_t last = 0;                             // keys <= last are composited
        bool first = true, done = false;
        while (__any_sync(full, !done) && steps <= kPacketSteps) {   // a round
            int cnt = 0;
            uint64_t maxkey = ~0ull;                   // key of the last entry once the buffer is full
            const float t_lo = first ? LP.r_min : __uint_as_float((uint32_t)(last >> 32));
            float t_hi = LP.r_max;
            for (int slot = 0; slot < K; ++slot) {
                const LidarSlot& S = sl[slot];
                if (S.node < 0) continue;
                const LidarTreeDev tr = trees[S.node];
                if (tr.n == 0) continue;
                const NodeRay R = node_ray(S, ds);
                int sp = 0;
                if (__any_sync(full, !done && slab(tr.box[2], tr.box[3], R.o, R.id, t_lo, t_hi))) {
                    if (lane == 0) stk[0] = 1u;
                    sp = 1;
                }
                __syncwarp();
                while (sp > 0 && ++steps <= kPacketSteps) {
                    const uint32_t k = stk[--sp];
                    __syncwarp();                      // every lane has read before lane 0 writes
                    if ((int64_t)k < tr.P) {
                        const float4* b = tr.box + 4 * (size_t)k;      // the children 2k and 2k + 1
                        const float4 l0 = __ldg(b), h0 = __ldg(b + 1), l1 = __ldg(b + 2), h1 = __ldg(b + 3);
                        const unsigned b0 = __ballot_sync(full, !done && slab(l0, h0, R.o, R.id, t_lo, t_hi));
                        const unsigned b1 = __ballot_sync(full, !done && slab(l1, h1, R.o, R.id, t_lo, t_hi));
                        if (!(b0 | b1)) continue;
                        const int more = b0 && b1 ? 2 : 1;
                        bool zero = b0 != 0;
                        if (more == 2) {
                            const bool near0 = slab_enter(l0, h0, R.o, R.id) <= slab_enter(l1, h1, R.o, R.id);
                            zero = __shfl_sync(full, near0, __ffs(b0 | b1) - 1);
                        }
                        if (sp + more > kWalk) {       // cannot happen for trees of the documented sizes
                            if (lane == 0) atomicOr(err, kErrCapacity);
                            break;
                        }
                        if (lane == 0) {               // far child below, near on top
                            if (more == 2) stk[sp] = 2u * k + (zero ? 1u : 0u);
                            stk[sp + more - 1] = 2u * k + (zero ? 0u : 1u);
                        }
                        sp += more;
                        __syncwarp();
                        continue;
                    }
                    const int64_t g0 = ((int64_t)k - tr.P) * kLeaf, g1 = min(g0 + kLeaf, tr.n);
                    // the next Gaussian's record is loaded while this one is tested
                    float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0, n3 = n0;
                    auto load = [&](int64_t g) {
                        const float4* rp = tr.rec + 4 * g;
                        n0 = __ldg(rp); n1 = __ldg(rp + 1); n2 = __ldg(rp + 2); n3 = __ldg(rp + 3);
                    };
                    if (g0 < g1) load(g0);
                    for (int64_t g = g0; g < g1; ++g) {
                        const float4 r0 = n0, r1 = n1, r2 = n2, r3 = n3;
                        if (g + 1 < g1) load(g + 1);
                        float t, q;
                        if (done || !peak(r0, r1, r2, r3, R, LP, t, q)) continue;
                        const uint64_t key = ((uint64_t)__float_as_uint(t) << 32) | (uint32_t)(tr.gbase + g);
                        if ((!first && key <= last) || key >= maxkey) continue;
                        const float alpha = hit_alpha(r0.w, q, LP);
                        if (alpha < LP.alpha_min) continue;
                        // insert in order; a full buffer drops its last entry
                        int i = min(cnt, kHits - 1);
                        for (; i > 0; --i) {
                            const uint32_t pt = kt[(i - 1) * kPacketThreads], pg = kg[(i - 1) * kPacketThreads];
                            if ((((uint64_t)pt << 32) | pg) < key) break;
                            kt[i * kPacketThreads] = pt;
                            kg[i * kPacketThreads] = pg;
                            ka[i * kPacketThreads] = ka[(i - 1) * kPacketThreads];
                        }
                        kt[i * kPacketThreads] = (uint32_t)(key >> 32);
                        kg[i * kPacketThreads] = (uint32_t)key;
                        ka[i * kPacketThreads] = alpha;
                        cnt = min(cnt + 1, kHits);
                        if (cnt == kHits) {
                            const uint32_t lt = kt[(kHits - 1) * kPacketThreads];
                            maxkey = ((uint64_t)lt << 32) | kg[(kHits - 1) * kPacketThreads];
                            t_hi = __uint_as_float(lt);
                        }
                    }
                    __syncwarp();
                }
                __syncwarp();
            }
            if (!done) {
                for (int i = 0; i < cnt && !done; ++i) {
                    const float a = ka[i * kPacketThreads], Tn = fmaf(-a, T, T);
                    if (Tn < LP.t_min) {
                        done = true;
                    } else {
                        D = fmaf(a * T, __uint_as_float(kt[i * kPacketThreads]), D);
                        T = Tn;
                    }
                }
                done |= cnt < kHits;
                last = maxkey;
                first = false;
            }
        }
        if (steps > kPacketSteps) {                          // given up: its rays one by one
            if (lane == 0) packets.left[atomicAdd(packets.counts + 1, 1u)] = pk;
            continue;
        }
        out_d[ray0 + lane] = D;
        out_a[ray0 + lane] = 1.f - T;
    }
}

}  // namespace

size_t lidar_tree_nodes(int64_t n) {
    if (n <= 0) return 0;
    const int64_t leaves = (n + kLeaf - 1) / kLeaf;
    int64_t P = 1;
    while (P < leaves) P <<= 1;
    return (size_t)(2 * P);
}

void launch_lidar_records(const Launch& L, const NodeDesc& nd, float q_max, float4* rec, float4* box, int64_t P) {
    if (nd.n <= 0) return;
    const int64_t threads = P * kLeaf;              // every leaf, padding leaves included
    const unsigned blocks = (unsigned)((threads + 255) / 256);
    const float sq = sqrtf(q_max);
    switch (nd.dtype) {
        case DGS_BF16: k_lidar_records<DGS_BF16><<<blocks, 256, 0, L.stream>>>(nd, sq, rec, box, P); break;
        case DGS_F16: k_lidar_records<DGS_F16><<<blocks, 256, 0, L.stream>>>(nd, sq, rec, box, P); break;
        default: k_lidar_records<DGS_F32><<<blocks, 256, 0, L.stream>>>(nd, sq, rec, box, P); break;
    }
    ++*L.launches;
}

void launch_lidar_level(const Launch& L, const void* jobs, int n_jobs, int64_t h, int64_t total) {
    if (total <= 0) return;
    k_lidar_level<<<(unsigned)((total + 255) / 256), 256, 0, L.stream>>>(static_cast<const LevelJob*>(jobs), n_jobs,
                                                                           h, total);
    ++*L.launches;
}

size_t lidar_level_job_bytes() { return sizeof(LevelJob); }

void lidar_level_job(void* jobs, int i, float4* box, int64_t first) {
    static_cast<LevelJob*>(jobs)[i] = LevelJob{box, first};
}

// Rays from which packets are looked for: with fewer, the slowest packet is longer than all rays one by one,
// but for beams a tenth of a degree apart or less.  The cone widens with the number of packets, which
// hides the slow ones.
constexpr int64_t kPacketRays = 1 << 16;
constexpr float kPacketCone = 0.010471976f;             // 0.6 degrees, from
constexpr int64_t kPacketConeRays = 1 << 17;            // this many rays on, in proportion below

size_t lidar_packet_words(int64_t n_rays) { return n_rays >= kPacketRays ? 2 * (size_t)((n_rays + 31) / 32) : 0; }

LidarPackets lidar_packets(int64_t n_rays, uint32_t* scratch, uint32_t* counters) {
    LidarPackets p{};
    p.n = (uint32_t)(lidar_packet_words(n_rays) / 2);
    p.cone = kPacketCone * std::min(1.f, (float)n_rays / (float)kPacketConeRays);
    p.together = scratch;
    p.left = scratch + p.n;
    p.next = counters;
    p.counts = counters + 1;
    return p;
}

void launch_lidar_setup(const Launch& L, const LidarSensorDev* sensors, int S, const int32_t* slot_node, int K,
                        const float* node_poses, LidarSlot* out, uint32_t* err, const float* dirs, int n_dirs,
                        int64_t n_rays, const LidarPackets& packets) {
    const int n = S * K;
    if (n == 0) return;
    const int threads = packets.n ? kSetupThreads : 128;
    const unsigned blocks = (unsigned)((n + threads - 1) / threads);
    k_lidar_setup<<<blocks + (packets.n + 31) / 32, threads, 0, L.stream>>>(sensors, S, slot_node, K, node_poses, out, err,
                                                                           blocks, dirs, n_dirs, n_rays, packets);
    ++*L.launches;
}

template <class Kernel>
static unsigned resident_blocks(Kernel* k, int threads, size_t smem) {
    int dev = 0, sms = 0, r = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (smem) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k, threads, smem);
    return (unsigned)(std::max(r, 1) * sms);
}

void launch_lidar_trace(const Launch& L, const LidarTreeDev* trees, const LidarSlot* slots, int K, const float* dirs,
                        int n_dirs, int64_t n_rays, const LidarParams& LP, float* out_d, float* out_a, uint32_t* err,
                        unsigned long long* next_ray, const LidarPackets& packets) {
    if (n_rays <= 0) return;
    if (packets.n) {
        static const unsigned most = resident_blocks(k_lidar_packets, kPacketThreads, kPacketSmem);
        const unsigned need = (packets.n + kPacketThreads / 32 - 1) / (kPacketThreads / 32);
        k_lidar_packets<<<std::min(need, most), kPacketThreads, kPacketSmem, L.stream>>>(
            trees, slots, K, dirs, n_dirs, n_rays, LP, out_d, out_a, err, packets);
        ++*L.launches;
    }
    auto* kern = packets.n ? k_lidar_trace<true> : k_lidar_trace<false>;
    static const unsigned most = std::min(resident_blocks(k_lidar_trace<true>, kRayWarps * 32, 0),
                                          resident_blocks(k_lidar_trace<false>, kRayWarps * 32, 0));
    const unsigned blocks = (unsigned)std::min<int64_t>((n_rays + kRayWarps - 1) / kRayWarps, most);
    kern<<<blocks, kRayWarps * 32, 0, L.stream>>>(trees, slots, K, dirs, n_dirs, n_rays, LP, out_d, out_a, err, next_ray,
                                                  packets.left, packets.counts);
    ++*L.launches;
}

}  // namespace dgs
