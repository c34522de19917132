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
// Tracing: one warp per ray, its lanes testing 32 boxes or 32 Gaussians at a time (see
// k_lidar_trace).
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

// Per (sensor, slot): the sensor's rotation and origin expressed in the node's frame.
__global__ void k_lidar_setup(const LidarSensorDev* __restrict__ sensors, int S, const int32_t* __restrict__ slot_node,
                              int K, const float* __restrict__ node_poses, LidarSlot* __restrict__ out,
                              uint32_t* __restrict__ err) {
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
// Bound by latency (boxes and records come from L2, one dependent load per step) and at 66 % issue;
// 64 registers keep 32 warps an SM.  Same outputs bit for bit, one sensor of 32 x 1024 beams through
// 380k Gaussians and 16 sensors through 580k: a packet of 32 rays per warp with a 32-hit buffer per
// lane 7.4 and 28 ms (with one sensor the slowest packet was the time); one ray per warp, one node
// of five levels per expansion, 72 registers 0.592 and 5.59 ms; two nodes 0.588 and 5.51; with 64
// registers 0.555 and 5.04.
__global__ void __launch_bounds__(kRayWarps * 32, 8) k_lidar_trace(const LidarTreeDev* __restrict__ trees,
                                                                const LidarSlot* __restrict__ slots, int K,
                                                                const float* __restrict__ dirs, int n_dirs,
                                                                int64_t n_rays, LidarParams LP,
                                                                float* __restrict__ out_d, float* __restrict__ out_a,
                                                                uint32_t* __restrict__ err,
                                                                unsigned long long* __restrict__ next_ray) {
    __shared__ RayWarp s_warp[kRayWarps];
    const int lane = threadIdx.x & 31;
    RayWarp& W = s_warp[threadIdx.x >> 5];
    for (;;) {
        unsigned long long ray = 0;
        if (lane == 0) ray = atomicAdd(next_ray, 1ull);
        ray = __shfl_sync(0xffffffffu, ray, 0);
        if (ray >= (unsigned long long)n_rays) break;
        const int64_t s = (int64_t)ray / n_dirs, j = (int64_t)ray - s * n_dirs;
        float ds[3] = {dirs[3 * j], dirs[3 * j + 1], dirs[3 * j + 2]};
        {
            const float r = rsqrtf(ds[0] * ds[0] + ds[1] * ds[1] + ds[2] * ds[2]);
            ds[0] *= r; ds[1] *= r; ds[2] *= r;
        }
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
                    const float v0 = R.o[0] - r0.x, v1 = R.o[1] - r0.y, v2 = R.o[2] - r0.z;
                    const float x0 = fmaf(v1, R.d[2], -v2 * R.d[1]), x1 = fmaf(v2, R.d[0], -v0 * R.d[2]),
                                x2 = fmaf(v0, R.d[1], -v1 * R.d[0]);
                    if (!(fmaf(x0, x0, fmaf(x1, x1, x2 * x2)) > r3.y)) {   // |d| = 1 up to rounding
                        const float op0 = fmaf(r1.x, v0, fmaf(r1.y, v1, r1.z * v2));
                        const float op1 = fmaf(r1.w, v0, fmaf(r2.x, v1, r2.y * v2));
                        const float op2 = fmaf(r2.z, v0, fmaf(r2.w, v1, r3.x * v2));
                        const float dp0 = fmaf(r1.x, R.d[0], fmaf(r1.y, R.d[1], r1.z * R.d[2]));
                        const float dp1 = fmaf(r1.w, R.d[0], fmaf(r2.x, R.d[1], r2.y * R.d[2]));
                        const float dp2 = fmaf(r2.z, R.d[0], fmaf(r2.w, R.d[1], r3.x * R.d[2]));
                        const float dd = fmaf(dp0, dp0, fmaf(dp1, dp1, dp2 * dp2));
                        const float od = fmaf(op0, dp0, fmaf(op1, dp1, op2 * dp2));
                        const float c0 = fmaf(op1, dp2, -op2 * dp1), c1 = fmaf(op2, dp0, -op0 * dp2),
                                    c2 = fmaf(op0, dp1, -op1 * dp0);
                        const float idd = 1.f / dd;
                        t = -od * idd;
                        const float q = fmaf(c0, c0, fmaf(c1, c1, c2 * c2)) * idd;
                        if (q <= LP.q_max && t >= LP.r_min && t <= LP.r_max) {
                            const uint64_t key = ((uint64_t)__float_as_uint(t) << 32) | (uint32_t)(tr.gbase + g);
                            if ((first || key > last) && key < maxkey) {
                                alpha = fminf(LP.alpha_max, r0.w * fast_exp2(kHalfLog2e * q));
                                hit = alpha >= LP.alpha_min;
                            }
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

void launch_lidar_setup(const Launch& L, const LidarSensorDev* sensors, int S, const int32_t* slot_node, int K,
                        const float* node_poses, LidarSlot* out, uint32_t* err) {
    const int n = S * K;
    if (n == 0) return;
    k_lidar_setup<<<(n + 127) / 128, 128, 0, L.stream>>>(sensors, S, slot_node, K, node_poses, out, err);
    ++*L.launches;
}

void launch_lidar_trace(const Launch& L, const LidarTreeDev* trees, const LidarSlot* slots, int K, const float* dirs,
                        int n_dirs, int64_t n_rays, const LidarParams& LP, float* out_d, float* out_a, uint32_t* err,
                        unsigned long long* next_ray) {
    if (n_rays <= 0) return;
    static int resident = 0, sms = 0;           // blocks per SM at this kernel's resources
    if (!resident) {
        int dev = 0, r = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k_lidar_trace, kRayWarps * 32, 0);
        resident = std::max(r, 1);
    }
    const int64_t need = (n_rays + kRayWarps - 1) / kRayWarps;
    const unsigned blocks = (unsigned)std::min<int64_t>(need, (int64_t)resident * sms);
    k_lidar_trace<<<blocks, kRayWarps * 32, 0, L.stream>>>(trees, slots, K, dirs, n_dirs, n_rays, LP, out_d, out_a, err,
                                                           next_ray);
    ++*L.launches;
}

}  // namespace dgs
