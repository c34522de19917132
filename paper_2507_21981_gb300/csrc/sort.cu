// Stable LSD radix sort of (32-bit key, 32-bit value) pairs in the onesweep style (kernel K3).
//
// Sec. III-A: the 3DGS rasterizer orders the (tile, depth) pairs of every view with a fast
// GPU sort before blending.  Here the order is built in two stable sorts of 32-bit keys: the
// projected instances by depth key (28 bits) and then by their view in the view group (a more
// significant key carried by the values), then the (tile, instance) pairs -- emitted in that
// order -- by their tile within the view.  Stability carries the depth order, and the id order
// of equal depths, into every (view, tile) run.
//
// Structure: one upfront pass builds the histograms of every digit at once, its last block to
// finish turning them into the digits' first places; then each digit is
// one kernel in which a block takes the next 3072-key partition from an atomic counter, ranks
// its keys by digit inside the block (per-bit warp ballots + per-warp counters), publishes its
// digit counts, scatters its keys into shared memory in digit order, and only then finds its
// global offset per digit by decoupled look-back over the partitions before it (status word =
// 2-bit flag | 30-bit count), which have had that long to publish their prefixes.  Measured on
// the benchmark's key sets (17.9M depth keys, 59.7M tile keys), the ballot ranking with 12 keys
// per thread at 4 blocks per SM sorts 13-17 % faster than warp-match ranking with 16 keys at 3
// blocks (either change alone gains nothing), and the late look-back 4 % faster than one right
// after the ranking.  Digits are D = ceil(bits / passes) bits wide with passes = ceil(bits / 8),
// the last pass taking the remaining bits so that exactly the requested key bits are sorted
// (bits above them keep their input order: the tile keys hold the view there, ordered by the
// depth sort before); measured on this path, wider digits (fewer passes) lose what they save to
// the scatter, whose runs per partition shrink to a few keys.  Look-back spins are bounded by
// a wall-clock limit (SortCtl::spin_ns, 1 s by default); on expiry the kernel sets
// kErrTimeout and finishes: its output is then not a permutation of the input, the kernels
// that use sorted values as indices return at once when they see kErrTimeout, and the host
// reports the timeout.
#include <algorithm>
#include <utility>

#include "dgs_internal.cuh"

namespace dgs {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 12;
constexpr int kTile = kThreads * kItems;          // 3072 keys per partition
constexpr int kWarps = kThreads / 32;
constexpr int kMaxD = 8;                          // widest digit: 256 bins
constexpr int kMaxR = 1 << kMaxD;
constexpr int kWindow = 4;                        // predecessors read per digit and look-back round
constexpr int kSmem = kTile * 8 + kWarps * kMaxR * 4;
constexpr int kKeysIn = 0, kKeysGather = 1, kKeysPacked = 2;   // where a pass's key comes from

__device__ __forceinline__ uint32_t live_count(uint32_t n, const uint32_t* d_n) { return d_n ? min(*d_n, n) : n; }

// Histograms of every pass's digit (digit width D) in one read of the keys; hist[p * kMaxR + b].
// Each warp counts into its own shared-memory copy (the copies are summed at the end).  RUNS:
// each thread counts 16 consecutive keys (four 16-byte loads) and issues one shared atomic per
// run of equal digits -- for keys whose high digits repeat over neighbours (tile keys emitted
// instance by instance, depth keys emitted node chunk by node chunk), whose lanes would
// otherwise all add to one counter; else a grid-stride loop with one atomic per key and pass.
// The last block to finish (done: a zeroed counter) replaces every pass's counts by their exclusive
// scan, and adds the view passes' (VH.passes > 0) from the count scan: view j of the group holds
// inst_off[view_tab[v0 + j + 1]] - inst_off[view_tab[v0 + j]] instance numbers.
struct ViewHist {
    const uint32_t* inst_off = nullptr;
    const int64_t* view_tab = nullptr;
    int v0 = 0, nv = 0, passes = 0, D = 0, last_bits = 0;
};

// Exclusive scans of up to four values per thread over the block, all at once.
__device__ __forceinline__ void block_excl_scan4(uint32_t (&v)[4]) {
    __shared__ uint32_t s_w[4][kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t y[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) y[p] = v[p];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, y[p], o);
            if (lane >= o) y[p] += t;
        }
    if (lane == 31) {
#pragma unroll
        for (int p = 0; p < 4; ++p) s_w[p][warp] = y[p];
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        v[p] = y[p] - v[p];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) v[p] += w < warp ? s_w[p][w] : 0u;
    }
    __syncthreads();
}

template <bool RUNS>
__global__ void __launch_bounds__(kThreads) k_hist(const uint32_t* __restrict__ keys, uint32_t n,
                                                   const uint32_t* __restrict__ d_n, int passes, int D,
                                                   int last_bits, uint32_t* hist, uint32_t* done, ViewHist VH) {
    __shared__ uint32_t sh_all[kWarps][4 * kMaxR];   // one private histogram per warp
    __shared__ bool s_last;
    uint32_t* sh = sh_all[threadIdx.x >> 5];
    n = live_count(n, d_n);
    // every pass's digit is D bits but the last one's, last_bits (the key bits above are not sorted)
    const uint32_t R = 1u << D;
    auto dmask = [&](int p) { return p == passes - 1 ? (1u << last_bits) - 1u : R - 1u; };
    for (int i = threadIdx.x; i < kWarps * 4 * kMaxR; i += kThreads) (&sh_all[0][0])[i] = 0;
    __syncthreads();
    if constexpr (RUNS) {
        const uint32_t stride = gridDim.x * kThreads * 16u;
        for (uint32_t base = (blockIdx.x * kThreads + threadIdx.x) * 16u; base < n; base += stride) {
            uint32_t k[16];
            if (base + 16 <= n) {
                const uint4* q = reinterpret_cast<const uint4*>(keys + base);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 v = __ldg(q + j);
                    k[4 * j] = v.x; k[4 * j + 1] = v.y; k[4 * j + 2] = v.z; k[4 * j + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) k[j] = base + j < n ? keys[base + j] : 0u;
            }
            const int cnt = (int)min(16u, n - base);
            for (int p = 0; p < passes; ++p) {
                const uint32_t mask = dmask(p);
                uint32_t cur = (k[0] >> (D * p)) & mask, run = 1;
#pragma unroll
                for (int j = 1; j < 16; ++j) {
                    if (j >= cnt) break;
                    const uint32_t d = (k[j] >> (D * p)) & mask;
                    if (d == cur) { ++run; continue; }
                    atomicAdd(&sh[p * R + cur], run);
                    cur = d;
                    run = 1;
                }
                atomicAdd(&sh[p * R + cur], run);
            }
        }
    } else {
        for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
            const uint32_t k = keys[i];
            for (int p = 0; p < passes; ++p) atomicAdd(&sh[p * R + ((k >> (D * p)) & dmask(p))], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * (int)R; i += kThreads) {
        uint32_t t = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) t += sh_all[w][i];
        if (t) atomicAdd(&hist[(i / R) * kMaxR + (i % R)], t);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    static_assert(kMaxR <= kThreads, "one bin per thread");
    const int b = threadIdx.x;
    uint32_t x[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) x[p] = p < passes && b < kMaxR ? __ldcg(hist + p * kMaxR + b) : 0u;   // (bins past the digit's are zero)
    block_excl_scan4(x);
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if (p < passes && b < kMaxR) hist[p * kMaxR + b] = x[p];
    if (VH.passes == 0) return;
    uint32_t* const vh = &sh_all[0][0];
    for (int i = threadIdx.x; i < VH.passes * kMaxR; i += kThreads) vh[i] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < VH.nv; j += kThreads) {
        const uint32_t c = VH.inst_off[VH.view_tab[VH.v0 + j + 1]] - VH.inst_off[VH.view_tab[VH.v0 + j]];
        if (!c) continue;
        for (int p = 0; p < VH.passes; ++p) {
            const uint32_t mask = (1u << (p == VH.passes - 1 ? VH.last_bits : VH.D)) - 1u;
            atomicAdd(&vh[p * kMaxR + (((uint32_t)j >> (VH.D * p)) & mask)], c);
        }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; ++p) x[p] = p < VH.passes && b < kMaxR ? vh[p * kMaxR + b] : 0u;
    block_excl_scan4(x);
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if (p < VH.passes && b < kMaxR) hist[(passes + p) * kMaxR + b] = x[p];
}

// One digit pass.  Thread t owns digits t, t + 256, ... (< 2^D) in the per-digit phases
// (prefix over warps, look-back, block scan); digits are (key >> shift) & (2^D - 1).
// MODE kKeysIn reads the keys; the other two derive a more significant key from the value (the
// keys sorted by the earlier passes are dropped): kKeysGather reads key = ind[value], kKeysPacked
// takes the value's high bits, key = value >> vshift.  Those two write no keys.  Every mode
// stores value & vmask (the last pass over packed values strips the key bits).  A null kout
// also skips the key writes (keys that no later pass reads).
template <int D, int MODE>
__global__ void __launch_bounds__(kThreads, 4) k_onesweep(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                      uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, uint32_t n,
                                                      const uint32_t* __restrict__ d_n, int shift,
                                                      const uint32_t* __restrict__ digit_off, uint32_t* status,
                                                      uint32_t* counter, uint32_t* err, uint64_t spin_ns,
                                                      uint32_t mute_part, const uint32_t* __restrict__ ind, int vshift,
                                                      uint32_t vmask) {
    constexpr int R = 1 << D;
    constexpr uint32_t M = R - 1;
    constexpr int DPT = (R + kThreads - 1) / kThreads;   // digits per thread
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* s_keys = reinterpret_cast<uint32_t*>(smem);                          // kTile
    uint32_t* s_vals = reinterpret_cast<uint32_t*>(smem + kTile * 4);               // kTile
    uint32_t* s_whist = reinterpret_cast<uint32_t*>(smem + kTile * 8);              // kWarps x R
    __shared__ uint32_t s_dexcl[R];
    __shared__ uint32_t s_gbase[R];
    __shared__ uint32_t s_wsum[kWarps];
    __shared__ uint32_t s_part;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_part = atomicAdd(counter, 1u);
    for (int i = tid; i < kWarps * R; i += kThreads) s_whist[i] = 0;
    __syncthreads();
    const uint32_t part = s_part;
    n = live_count(n, d_n);
    // a capacity-sized grid: partitions past the live count have no keys (and no later
    // partition looks back at them)
    if (part * (uint64_t)kTile >= n && part > 0) return;
    const uint32_t base = part * (uint32_t)kTile;

    uint32_t k[kItems], v[kItems], rank[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const uint32_t idx = base + warp * (kItems * 32) + j * 32 + lane;
        if (idx < n) {
            v[j] = vin[idx];
            // (a value outside 0..n-1, left by an earlier pass that gave up waiting, reads nothing)
            k[j] = MODE == kKeysGather ? (v[j] < n ? __ldg(ind + v[j]) : ~0u)
                   : MODE == kKeysPacked ? v[j] >> vshift
                                         : kin[idx];
        } else {
            k[j] = ~0u; v[j] = 0;
        }
    }
    // rank within the warp, in original order (round j covers 32 consecutive keys); the lanes
    // holding the same digit are found by one ballot per digit bit
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t* wh = s_whist + warp * R;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const uint32_t dg = (k[j] >> shift) & M;
        uint32_t peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < D; ++b) {
            const bool bit = (dg >> b) & 1u;
            const uint32_t bal = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bal : ~bal;
        }
        const uint32_t pre = wh[dg];
        rank[j] = pre + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0) wh[dg] = pre + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // per owned digit: exclusive prefix over warps and the partition total
    uint32_t total[DPT], excl[DPT];
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
        const int d = tid + q * kThreads;
        total[q] = 0;
        excl[q] = 0;
        if (d < R) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t c = s_whist[w * R + d];
                s_whist[w * R + d] = total[q];
                total[q] += c;
            }
        }
    }
    // publish this partition's digit counts at once (the inclusive prefix for partition 0);
    // partition mute_part (a test of the bounded wait, never a real partition index by
    // default) publishes nothing, so the partitions after it wait for it until spin_ns runs out
    const bool publish = part != mute_part;
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
        const int d = tid + q * kThreads;
        if (d < R && publish) st_relaxed(&status[(size_t)part * R + d], (part == 0 ? kFlagInc : kFlagAgg) | total[q]);
    }
    // block exclusive scan of the digit totals in digit order -> local digit offsets; slab q
    // holds digits [q * 256, q * 256 + 256)
    uint32_t carry = 0;
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
        uint32_t x = total[q];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_wsum[warp] = x;
        __syncthreads();
        uint32_t wpre = 0, slab = 0;
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) wpre += s_wsum[w];
            slab += s_wsum[w];
        }
        const int d = tid + q * kThreads;
        if (d < R) s_dexcl[d] = carry + wpre + x - total[q];
        carry += slab;
        __syncthreads();
    }
    // local scatter: digit-major order inside the partition
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const uint32_t dj = (k[j] >> shift) & M;
        const uint32_t pos = s_dexcl[dj] + s_whist[warp * R + dj] + rank[j];
        s_keys[pos] = k[j];
        s_vals[pos] = v[j];
    }
    // decoupled look-back over earlier partitions, all owned digits at once, after the local
    // scatter: the partitions before this one have had that long to publish their prefixes
    if (part > 0) {
        int64_t p[DPT];
        bool done[DPT];
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            const int d = tid + q * kThreads;
            done[q] = d >= R;
            p[q] = (int64_t)part - 1;
        }
        uint64_t t0 = 0;
        uint32_t spins = 0;
        while (true) {
            uint32_t sv[DPT][kWindow];
#pragma unroll
            for (int q = 0; q < DPT; ++q)
#pragma unroll
                for (int w = 0; w < kWindow; ++w)
                    sv[q][w] = (!done[q] && p[q] - w >= 0)
                                   ? ld_relaxed(&status[(size_t)(p[q] - w) * R + tid + q * kThreads]) : kFlagInc;
            bool all = true, stall = false;
#pragma unroll
            for (int q = 0; q < DPT; ++q) {
                if (done[q]) continue;
                bool stop = false;
#pragma unroll
                for (int w = 0; w < kWindow; ++w) {
                    if (stop || done[q]) continue;
                    const uint32_t f = sv[q][w] & ~kCountMask;
                    if (f == 0) { stop = true; continue; }
                    excl[q] += sv[q][w] & kCountMask;
                    if (f == kFlagInc) done[q] = true; else --p[q];
                }
                if (!done[q]) { all = false; stall |= stop; }
            }
            if (all) break;
            if (stall && (++spins & 1023u) == 0) {
                const uint64_t now = global_timer_ns();
                if (t0 == 0) t0 = now;
                else if (now - t0 > spin_ns) { atomicOr(err, kErrTimeout); break; }
            }
        }
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            const int d = tid + q * kThreads;
            if (d < R && publish) st_relaxed(&status[(size_t)part * R + d], kFlagInc | (excl[q] + total[q]));
        }
    }
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
        const int d = tid + q * kThreads;
        if (d < R) s_gbase[d] = digit_off[d] + excl[q];
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < kTile; i += kThreads) {
        const uint32_t key = s_keys[i];
        const uint32_t dj = (key >> shift) & M;
        const uint32_t g = s_gbase[dj] + (uint32_t)i - s_dexcl[dj];
        // every live key lands below n (the padding keys, ~0, sort past the end and are dropped)
        if (kDebugChecks && key != ~0u && !in_bounds(g, n, err, kSiteSortScatter)) continue;
        if (g < n) {
            if (MODE == kKeysIn && kout) kout[g] = key;
            vout[g] = s_vals[i] & vmask;
        }
    }
}

using OnesweepFn = void (*)(const uint32_t*, const uint32_t*, uint32_t*, uint32_t*, uint32_t, const uint32_t*, int,
                            const uint32_t*, uint32_t*, uint32_t*, uint32_t*, uint64_t, uint32_t, const uint32_t*, int,
                            uint32_t);

template <int MODE>
OnesweepFn onesweep_for(int D) {
    switch (D) {
        case 1: return k_onesweep<1, MODE>;
        case 2: return k_onesweep<2, MODE>;
        case 3: return k_onesweep<3, MODE>;
        case 4: return k_onesweep<4, MODE>;
        case 5: return k_onesweep<5, MODE>;
        case 6: return k_onesweep<6, MODE>;
        case 7: return k_onesweep<7, MODE>;
        default: return k_onesweep<8, MODE>;
    }
}

}  // namespace

// Streaming multiprocessors of the current device (read once per process and device).
uint32_t sm_count() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    if (!cached[dev]) {
        int n = 0;
        cached[dev] = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 152;
    }
    return (uint32_t)cached[dev];
}

int sort_passes(int key_bits) { return std::max(1, (key_bits + kMaxD - 1) / kMaxD); }

namespace {

// Passes of a sort of n keys and the places of its parts in the zeroed scratch: histograms, then
// counters (one per pass, and the histogram's), then every pass's look-back status.
struct SortPlan {
    int passes, D, last, vpasses, vD, vlast;
    uint32_t parts;
    size_t counters, status[8], words;
    SortPlan(uint32_t n, int key_bits, int view_bits, bool compact) {
        const int bits = std::max(1, key_bits);
        passes = sort_passes(bits);
        D = (bits + passes - 1) / passes;
        last = bits - D * (passes - 1);               // exactly key_bits bits are sorted
        vpasses = view_bits > 0 ? sort_passes(view_bits) : 0;
        vD = vpasses ? (view_bits + vpasses - 1) / vpasses : 0;
        vlast = vpasses ? view_bits - vD * (vpasses - 1) : 0;
        parts = (n + kTile - 1) / kTile;
        counters = (size_t)kMaxR * (passes + vpasses);
        const size_t first = counters + 16;
        words = first;
        for (int p = 0; p < passes + vpasses; ++p) {
            status[p] = compact ? first : words;
            words = std::max(words, status[p] + status_words(p));
        }
        words = (words + 3) & ~size_t(3);
    }
    size_t status_words(int p) const { return (size_t)parts << digit_bits(p); }
    int digit_bits(int p) const {
        return p < passes ? (p == passes - 1 ? last : D) : (p - passes == vpasses - 1 ? vlast : vD);
    }
};

}  // namespace

size_t sort_scratch_words(uint32_t n, int key_bits, int view_bits, bool compact) {
    return SortPlan(n, key_bits, view_bits, compact).words;
}

void sort_prepare() {
    static bool attr_set = false;
    if (!attr_set) {
        for (int D = 1; D <= kMaxD; ++D) {
            cudaFuncSetAttribute(onesweep_for<kKeysIn>(D), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            cudaFuncSetAttribute(onesweep_for<kKeysGather>(D), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            cudaFuncSetAttribute(onesweep_for<kKeysPacked>(D), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        }
        attr_set = true;
    }
}

void launch_sort(const Launch& L, uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, uint32_t n,
                 int key_bits, uint32_t* scratch, uint32_t* err, uint32_t** keys_out, uint32_t** vals_out,
                 const uint32_t* d_n, SortCtl ctl, const ViewKey* vk) {
    *keys_out = keys;
    *vals_out = vals;
    // with a device-side count every pass runs (the output lands in the same buffer whatever
    // the count); a host-known count of 0 or 1 is already sorted, but a single packed value still has to
    // lose the view in its high bits, which its readers would take for an instance number
    const bool by_view = vk && vk->bits > 0, packed = by_view && vk->vshift > 0;
    if (n == 0 || (n == 1 && !d_n && !packed)) return;
    const SortPlan S(n, key_bits, by_view ? vk->bits : 0, ctl.compact);
    sort_prepare();
    uint32_t* const hist = scratch;
    uint32_t* const counters = scratch + S.counters;
    ViewHist VH;
    if (by_view) VH = ViewHist{vk->inst_off, vk->view_tab, vk->v0, vk->nv, S.vpasses, S.vD, S.vlast};
    const int hist_blocks = (int)std::min<uint32_t>(4 * sm_count(), (n + kThreads * 8 - 1) / (kThreads * 8));
    auto* hk = ctl.runs ? k_hist<true> : k_hist<false>;
    hk<<<hist_blocks, kThreads, 0, L.stream>>>(keys, n, d_n, S.passes, S.D, S.last, hist, counters + 15, VH);
    ++*L.launches;
    uint32_t *ki = keys, *ko = keys_alt;
    uint32_t *vi = vals, *vo = vals_alt;
    for (int p = 0; p < S.passes + S.vpasses; ++p) {
        // the last passes' key is the most significant one, the view, derived from the values (their
        // high bits, stripped by the last pass, or vig[value]); no keys are written for them
        const bool view = p >= S.passes;
        const int Dp = S.digit_bits(p), shift = view ? S.vD * (p - S.passes) : S.D * p;
        const OnesweepFn fn = !view ? onesweep_for<kKeysIn>(Dp) : packed ? onesweep_for<kKeysPacked>(Dp)
                                                                         : onesweep_for<kKeysGather>(Dp);
        uint32_t* kw = by_view && p >= S.passes - 1 ? nullptr : ko;
        const uint32_t vmask = packed && p == S.passes + S.vpasses - 1 ? (1u << vk->vshift) - 1u : 0xFFFFFFFFu;
        if (ctl.compact && p > 0)
            cudaMemsetAsync(scratch + S.status[p], 0, sizeof(uint32_t) * S.status_words(p), L.stream);
        fn<<<S.parts, kThreads, kSmem, L.stream>>>(ki, vi, kw, vo, n, d_n, shift, hist + p * kMaxR,
                                                   scratch + S.status[p], counters + p, err, ctl.spin_ns,
                                                   p == 0 ? ctl.mute_part : 0xFFFFFFFFu, view ? vk->vig : nullptr,
                                                   view ? vk->vshift : 0, vmask);
        ++*L.launches;
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
    *keys_out = by_view ? nullptr : ki;
    *vals_out = vi;
}

}  // namespace dgs
