// Wave-particle state kernels of the hybrid ocean (sm_103a):
//   advection + expiry + stable compaction  (Sec. 3.1 Lagrangian propagation,
//     with the survivors' bin keys            Sec. 4.1 WP updates),
//   boundary injection and wake emission     (Sec. 3.3 Eqs. 15-17, Sec. 4.3),
//   per-bucket integer binning               (Sec. 4.2: the particles of a
//                                            bucket share radius and kernel):
//                                            a stable LSD radix sort of the bin
//                                            keys, one launch per 8-bit digit
//                                            (decoupled look-back for the
//                                            blocks' digit offsets).
// All particle state is integer (Q16.16 cell units); every decision is an
// integer test, so the state is bit-exact against any other implementation of
// the same rules.  No float atomics anywhere; integer atomics only for counts.
#include <cuda_runtime.h>

#include <algorithm>
#include <stdint.h>
#include <string.h>
#include <type_traits>

#include "internal.h"
#include "philox.h"

namespace scwp {
namespace {

constexpr int kTpb = 256;
constexpr int kItems = 4;                 // per thread in the compaction tiles
constexpr int kTileC = kTpb * kItems;     // 1024 particles per compaction block
static_assert(kTileC == kStepTile, "compaction words");
constexpr int kTileS = kSortTile;     // keys per bin-key block
constexpr int32_t kQi = 65536, kHalfi = 32768;

// The patches of one launch, by value in the kernel's parameters (constant
// bank: no load stands ahead of a block's first access).  Every particle
// kernel runs over all patches of a frame at once, patch blockIdx.y, blocks
// past a patch's own tiles returning at once: the stages of one patch are
// short serial chains (4-7 us each on patches of up to 200k particles,
// mostly latency), so one launch per patch and stage left the GPU nearly
// idle and cost a launch each.  Packs of 1, 8 or 32 patches keep the
// parameter copy near the patches there are (about 0.3 KB a patch).
constexpr int kPackMax = 32;
template <int M>
struct PatchPack {
    static constexpr int kM = M;
    PatchDev p[M];
};

// Texel centres of [0, n) strictly inside (C - R, C + R) along one axis.
__device__ __forceinline__ int span_count(int32_t C, int32_t R, int n) {
    int64_t lo = (((int64_t)C - R - kHalfi) >> 16) + 1;
    int64_t hi = ((int64_t)C + R - kHalfi - 1) >> 16;
    if (lo < 0) lo = 0;
    if (hi > n - 1) hi = n - 1;
    return hi >= lo ? (int)(hi - lo + 1) : 0;
}

// floor(x / d) and x - d floor(x / d) (in [0, d)) for d > 0: the quotient
// estimated in FP32 (relative error below 2^-21, so off by at most one where
// |x / d| < 2^19), then corrected in integers; exact integer division beyond
// that range.
__device__ __forceinline__ int32_t floor_divmod(int32_t x, int32_t d, int32_t& rem) {
    const float qf = floorf(__fdividef((float)x, (float)d));
    if (fabsf(qf) >= 524288.f) {   // 2^19: not in the estimate's range
        int32_t q = x / d, r = x % d;
        if (r < 0) {
            --q;
            r += d;
        }
        rem = r;
        return q;
    }
    int32_t q = (int32_t)qf;
    int64_t r = (int64_t)x - (int64_t)q * d;
    if (r < 0) {
        --q;
        r += d;
    } else if (r >= d) {
        ++q;
        r -= d;
    }
    rem = (int32_t)r;
    return q;
}

__device__ __forceinline__ int4 lookup_vq(const PatchDev& p, uint32_t bd) {
    const int b = (int)(bd >> 16), j = (int)(bd & 0xFFFFu);
    const int idx = j < p.nth ? b * p.nth + j : p.nb * p.nth + (j - p.nth);
    return p.vq[idx];
}

__device__ __forceinline__ float lookup_amp(const PatchDev& p, uint32_t bd) {
    const int b = (int)(bd >> 16), j = (int)(bd & 0xFFFFu);
    return j < p.nth ? p.amp[b * p.nth + j] : p.wake_amp;
}

// 8-bit digits of a patch's bin keys
__host__ __device__ __forceinline__ int sort_passes(const PatchDev& p) { return (p.key_bits + 7) / 8; }

// look-back word: flag in the top two bits, a count below
constexpr uint32_t kLbAggregate = 1u << 30, kLbPrefix = 2u << 30, kLbCount = (1u << 30) - 1u;
constexpr long long kLbWaitCycles = 2000000000ll;  // the frame's limit: ~1 s at 2 GHz

// A look-back word carries its flag and count together, so plain relaxed
// accesses (atomic per word, no ordering against other data) suffice, and
// the loads of one batch overlap.
__device__ __forceinline__ void st_relaxed(uint32_t* a, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* a) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a));
    return v;
}

// The live particles a patch's kernels take: none once one of its bounded waits
// has run out.  A step or a sort pass that gave up leaves counts, digit totals
// and keys that no longer agree; a later pass that trusted them would store
// past the key buffers, the records would be gathered by ids from places that
// nothing wrote, and the synthesis would follow bin offsets that run backwards.
// From the kernel after the one that gave up on, the patch is empty instead:
// no keys, every bin offset zero.
// count[2] holds a bit for each kernel of a frame that may give up, and one
// for an earlier frame (set by the record pass).  A kernel looks only at the
// bits of kernels before it, so that all its threads see the same count; the
// bits come with the count in one load.
constexpr int kGaveUpStep = 1, kGaveUpBefore = 1 << 8, kGaveUpAny = ~0;
__host__ __device__ constexpr int gave_up_pass(int ps) { return 2 << ps; }
static_assert(gave_up_pass(kMaxSortPasses - 1) < kGaveUpBefore, "one bit each");

__device__ __forceinline__ int live_count(const PatchDev& p, int gave_up) {
    const int4 c = *reinterpret_cast<const int4*>(p.count);
    return (c.z & gave_up) ? 0 : c.x;
}
__device__ __forceinline__ void give_up(const PatchDev& p, int bit) {
    atomicOr(&p.stats[2], (unsigned long long)kErrTimeout);
    atomicOr(&p.count[2], bit);
}

// ---- a6: bin keys -------------------------------------------------------------
// A block's counts while it makes keys: every sort pass's digits (so the
// passes need no histogram launch), live particles per bucket, evaluations
// and binned bumps.
struct KeyCounts {
    uint32_t h[kMaxSortPasses][256];
    unsigned int live[kMaxBuckets];
    unsigned long long ev[kTpb / 32];
    unsigned int bin[kTpb / 32];
};
static_assert(kTpb == 256, "one digit counter per thread");

__device__ __forceinline__ void keys_begin(KeyCounts& C, const PatchDev& p) {   // (a block barrier must follow)
    for (int i = threadIdx.x; i < p.nb; i += kTpb) C.live[i] = 0;
#pragma unroll
    for (int ps = 0; ps < kMaxSortPasses; ++ps) C.h[ps][threadIdx.x] = 0;
}

// block b of a kernel clears the look-back words of sort-pass block b
__device__ __forceinline__ void clear_sort_words(const PatchDev& p) {
    if ((int)blockIdx.x < p.nblk_o)
        for (int ps = 0; ps < sort_passes(p); ++ps)
            p.sort_status[((size_t)ps * p.nblk_o + blockIdx.x) * 256 + threadIdx.x] = 0u;
}

// The crest's and trough's keys of a particle (total_bins: the bump reaches
// no texel) and its counts' share; whether either bump reaches the patch.
__device__ __forceinline__ bool make_keys(const PatchDev& p, int32_t x, int32_t y, uint32_t bd, int4 vq,
                                          uint32_t (&key)[2], unsigned long long& ev, unsigned int& binned) {
    const BucketDev bk = p.bk[bd >> 16];
    bool any = false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int32_t cx = k ? x - vq.z : x;
        const int32_t cy = k ? y - vq.w : y;
        const int nx = span_count(cx, bk.R, p.W), ny = span_count(cy, bk.R, p.H);
        key[k] = (uint32_t)p.total_bins;
        if (nx > 0 && ny > 0) {
            // (cx + R, cy + R > 0 here: the support reaches the patch)
            int32_t rx, ry;
            const int bx = floor_divmod(cx + bk.R, bk.C, rx);
            const int by = floor_divmod(cy + bk.R, bk.C, ry);
            key[k] = (uint32_t)(bk.base + by * bk.nbx + bx);
            ev += (unsigned long long)nx * (unsigned long long)ny;
            ++binned;
            any = true;
        }
    }
    return any;
}

// A live particle's keys and bucket in the block's counts (where `ok`; every
// lane of the warp calls).  Neighbours mostly share their bucket: one shared
// atomic for such a warp (one per particle met 32 ways in one word).
__device__ __forceinline__ void count_keys(KeyCounts& C, const PatchDev& p, uint32_t bd, const uint32_t (&key)[2],
                                           bool ok) {
    const unsigned act = __ballot_sync(0xffffffffu, ok);
    if (act == 0u) return;
    const uint32_t b = bd >> 16, b0 = __shfl_sync(0xffffffffu, b, __ffs(act) - 1);
    const bool same = __all_sync(0xffffffffu, !ok || b == b0);
    if (!ok) return;
    if (!same)
        atomicAdd(&C.live[b], 1u);
    else if ((act & ((1u << (threadIdx.x & 31)) - 1u)) == 0u)
        atomicAdd(&C.live[b], (unsigned)__popc(act));
#pragma unroll
    for (int k = 0; k < 2; ++k)
        for (int ps = 0; ps < sort_passes(p); ++ps) atomicAdd(&C.h[ps][(key[k] >> (8 * ps)) & 255u], 1u);
}

// Particle i's keys, and its state packed for the record pass (one 16-byte
// gather per bump instead of three 4-byte ones).
__device__ __forceinline__ void store_keys(const PatchDev& p, int i, int32_t x, int32_t y, uint32_t bd,
                                           const uint32_t (&key)[2]) {
    p.pk[i] = make_int4(x, y, (int)bd, 0);
    reinterpret_cast<uint2*>(p.keys[0])[i] = make_uint2(key[0], key[1]);
}

// The block's counts to the frame's (stats_acc, which the record pass
// publishes and clears) and the passes' digit totals; every thread calls.
__device__ __forceinline__ void keys_end(KeyCounts& C, const PatchDev& p, unsigned long long ev, unsigned int binned) {
    // block reductions (integers: order-independent)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        ev += __shfl_down_sync(0xffffffffu, ev, o);
        binned += __shfl_down_sync(0xffffffffu, binned, o);
    }
    if (lane == 0) {
        C.ev[warp] = ev;
        C.bin[warp] = binned;
    }
    __syncthreads();
    unsigned long long* const acc = stats_acc(p);
    if (threadIdx.x == 0) {
        unsigned long long e = 0, bb = 0;
        for (int w = 0; w < kTpb / 32; ++w) {
            e += C.ev[w];
            bb += C.bin[w];
        }
        if (e) atomicAdd(&acc[0], e);
        if (bb) atomicAdd(&acc[1], bb);
    }
    for (int i = threadIdx.x; i < p.nb; i += kTpb)
        if (C.live[i]) atomicAdd(&acc[2 + i], (unsigned long long)C.live[i]);
    for (int ps = 0; ps < sort_passes(p); ++ps)   // (after the barrier above)
        if (C.h[ps][threadIdx.x]) atomicAdd(&p.hist[ps * 256 + threadIdx.x], C.h[ps][threadIdx.x]);
}

// ---- a3: advect, expire, compact ------------------------------------------------
// One pass over the state: a block takes tiles of 1024 particles in ticket
// order, advects them, finds the survivors' new places by decoupled look-back
// over the earlier tiles' counts (as the sort passes below do) and writes
// them, with their bin keys, to the other buffer.  Separate launches for the
// advection, the compaction and the keys moved 90 bytes a particle (the state
// written and read back twice) and took three of a small frame's nine serial
// launches; this moves 48 and is one.  The tile of the last particle
// publishes the new count: by then every block with a tile has read the old
// one, since that tile has seen all their counts.  A tile that gives up on its
// look-back (after wait_cycles SM clocks) sets the error flag and has summed a
// subset of the earlier tiles' counts: its stores stay in bounds, and the
// stages after it take the patch as empty (live_count).  Tickets start at tile
// first_tile: 0 in every frame, 1 in the failure-detection self-test, whose
// tile 0 nothing publishes.
template <int M>
__global__ void __launch_bounds__(kTpb) k_step(const __grid_constant__ PatchPack<M> pk, long long wait_cycles,
                                               int first_tile) {
    __shared__ KeyCounts C;
    __shared__ uint32_t s_cnt[32], s_off;   // survivors of 32-particle runs, then the runs' offsets
    __shared__ int s_bid;
    static_assert(kItems * kTpb / 32 == 32, "one run per lane of the scanning warp");
    const PatchDev& p = pk.p[M == 1 ? 0 : blockIdx.y];
    pdl_enter();
    if (M > 1 && (int)blockIdx.x >= p.nblk_c) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* const words = p.blk;          // [nblk_c] look-back words, then the ticket
    if (tid == 0) s_bid = (int)atomicAdd(words + p.nblk_c, 1u) + first_tile;
    clear_sort_words(p);
    keys_begin(C, p);
    __syncthreads();
    const int bid = s_bid;
    const int n = live_count(p, kGaveUpBefore), base = bid * kTileC;
    if (base >= n) {   // (uniform)
        if (n == 0 && bid == 0 && tid == 0) p.count[0] = p.count[1] = 0;
        return;
    }
    const int32_t* X = p.x[p.cur];
    const int32_t* Y = p.y[p.cur];
    const uint32_t* BD = p.bd[p.cur];
    int32_t xs[kItems], ys[kItems];
    uint32_t bs[kItems], rank[kItems];
    // particle of item k: base + k kTpb + tid; every load first
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int i = base + k * kTpb + tid;
        bs[k] = i < n ? BD[i] : 0u;
        xs[k] = i < n ? X[i] : 0;
        ys[k] = i < n ? Y[i] : 0;
    }
    // a particle lives on while either of its bumps reaches the patch: the
    // test that gives it its keys
    int4 vq[kItems];
    uint32_t alive = 0u, key[kItems][2];
    unsigned long long ev = 0;
    unsigned int binned = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) vq[k] = lookup_vq(p, bs[k]);
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        xs[k] += vq[k].x;
        ys[k] += vq[k].y;
        const bool a = base + k * kTpb + tid < n && make_keys(p, xs[k], ys[k], bs[k], vq[k], key[k], ev, binned);
        const uint32_t m = __ballot_sync(0xffffffffu, a);
        rank[k] = (uint32_t)__popc(m & ((1u << lane) - 1u));
        alive |= (a ? 1u : 0u) << k;
        if (lane == 0) s_cnt[k * (kTpb / 32) + warp] = (uint32_t)__popc(m);
        count_keys(C, p, bs[k], key[k], a);
    }
    __syncthreads();
    if (warp == 0) {
        const uint32_t v = s_cnt[lane];
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        s_cnt[lane] = inc - v;
        const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
        // survivors of the earlier tiles: 32 words at a time, back to the
        // nearest inclusive prefix; an unpublished word is read again
        uint32_t excl = 0;
        if (bid > 0) {
            if (lane == 0) st_relaxed(words + bid, kLbAggregate | total);
            const long long t0 = clock64();
            for (int j = bid - 1;;) {
                const uint32_t w = j - lane >= 0 ? ld_relaxed(words + (j - lane)) : kLbPrefix;
                const uint32_t pf = __ballot_sync(0xffffffffu, (w & ~kLbCount) == kLbPrefix);
                const uint32_t un = __ballot_sync(0xffffffffu, (w & ~kLbCount) == 0u);
                const int fp = pf ? __ffs(pf) - 1 : 32, fu = un ? __ffs(un) - 1 : 32;
                const bool done = fp < fu;
                const bool use = done ? lane <= fp : lane < fu;
                excl += __reduce_add_sync(0xffffffffu, use ? w & kLbCount : 0u);
                if (done) break;
                j -= fu;
                bool late = false;
                if (lane == 0 && fu < 32) late = clock64() - t0 > wait_cycles;
                if (__any_sync(0xffffffffu, late)) {
                    // (excl is then below the true offset: every store stays in bounds)
                    if (lane == 0) give_up(p, kGaveUpStep);
                    break;
                }
            }
        }
        if (lane == 0) {
            st_relaxed(words + bid, kLbPrefix | (excl + total));
            s_off = excl;
            if (base + kTileC >= n) p.count[0] = p.count[1] = (int32_t)(excl + total);
        }
    }
    __syncthreads();
    int32_t* Xd = p.x[1 - p.cur];
    int32_t* Yd = p.y[1 - p.cur];
    uint32_t* Bd = p.bd[1 - p.cur];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        const int o = (int)(s_off + s_cnt[k * (kTpb / 32) + warp] + rank[k]);
        if ((alive >> k) & 1u) {
            Xd[o] = xs[k];
            Yd[o] = ys[k];
            Bd[o] = bs[k];
            store_keys(p, o, xs[k], ys[k], bs[k], key[k]);
        }
    }
    keys_end(C, p, ev, binned);
}

// ---- a4 + a5: injection and wake emission -------------------------------------
// The injected particles follow the survivors, with their bin keys.  ip: the
// frame's plan (InjectParams, or its InjectHead); seg, gx, gy, ga: its
// segments and host-placed particles.
template <typename IP>
__device__ __forceinline__ void inject_body(const PatchDev& p, const IP& ip, const Segment* seg, const int32_t* gx,
                                            const int32_t* gy, const int32_t* ga) {
    __shared__ KeyCounts C;
    const int base = p.count[1];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t want = (int64_t)base + ip.total;
        p.count[0] = (int32_t)(want > p.cap ? p.cap : want);
        if (want > p.cap) atomicOr(&p.stats[2], (unsigned long long)kErrCapacity);
    }
    if ((int)(blockIdx.x * kTpb) >= ip.total) return;   // (uniform)
    keys_begin(C, p);
    __syncthreads();
    int32_t* X = p.x[p.cur];
    int32_t* Y = p.y[p.cur];
    uint32_t* BD = p.bd[p.cur];
    unsigned long long ev = 0;
    unsigned int binned = 0;
    for (int e0 = blockIdx.x * kTpb; e0 < ip.total; e0 += gridDim.x * kTpb) {
        const int e = e0 + threadIdx.x;
        const int64_t idx = (int64_t)base + e;
        const bool ok = e < ip.total && idx < p.cap;
        int32_t x = 0, y = 0;
        uint32_t bd = 0u;
        if (ok) {
            // the last segment that starts at or before e
            int sidx = 0;
            for (int hi = ip.nseg - 1; sidx < hi;) {
                const int mid = (sidx + hi + 1) >> 1;
                if (seg[mid].first <= e)
                    sidx = mid;
                else
                    hi = mid - 1;
            }
            const Segment sg = seg[sidx];
            const int le = e - sg.first;
            if (sg.s < 2) {
                const int g = le / sg.ndir, kk = le - g * sg.ndir;
                const int j = p.dirlist[(sg.bucket * 2 + sg.s) * p.nth + kk];
                const uint32_t ord = (uint32_t)(g * ip.nth + j);
                const U4 u = philox4x32_10(ip.frame, ip.patch, (uint32_t)sg.bucket | ((uint32_t)sg.s << 16), ord,
                                           ip.seed);
                const int4 vq = p.vq[sg.bucket * p.nth + j];
                const int32_t vn = sg.s == 0 ? vq.x : vq.y;
                const uint64_t avn = (uint64_t)(vn < 0 ? -(int64_t)vn : (int64_t)vn);
                const uint64_t len = (uint64_t)(sg.s == 0 ? ip.H : ip.W) * (uint64_t)kQi;
                const int32_t along = (int32_t)(((uint64_t)u.x * len) >> 32);
                const int32_t off = (int32_t)(((uint64_t)u.y * avn) >> 32);
                const int32_t far = (sg.s == 0 ? ip.W : ip.H) * kQi;
                const int32_t across = vn > 0 ? off : far - off;
                x = sg.s == 0 ? across : along;
                y = sg.s == 0 ? along : across;
                bd = ((uint32_t)sg.bucket << 16) | (uint32_t)j;
            } else {   // wake arms and ring ripples: positions placed on the host
                const int gi = sg.given + le;
                x = gx[gi];
                y = gy[gi];
                bd = ((uint32_t)sg.bucket << 16) | (uint32_t)(ip.nth + ga[gi]);
            }
            X[idx] = x;
            Y[idx] = y;
            BD[idx] = bd;
        }
        uint32_t key[2] = {0u, 0u};
        if (ok) {
            make_keys(p, x, y, bd, lookup_vq(p, bd), key, ev, binned);
            store_keys(p, (int)idx, x, y, bd, key);
        }
        count_keys(C, p, bd, key, ok);
    }
    keys_end(C, p, ev, binned);
}

// one patch, its plan by value
__global__ void __launch_bounds__(kTpb) k_inject(const __grid_constant__ PatchDev p,
                                                 const __grid_constant__ InjectParams ip) {
    pdl_enter();
    inject_body(p, ip, ip.seg, ip.gx, ip.gy, ip.ga);
}

// up to eight patches, their plans by value with only the segments and
// placed particles in use (an InjectParams is 6.5 KB, a kernel's parameters
// at most 32,764 bytes): patch k's segments start at word seg0[k] of `words`
// and its placed particles (x, y, direction arrays of given[k]) at giv0[k]
constexpr int kInjectMax = 8;
constexpr int kInjectWords = 6400;   // 25,600 bytes: three patches with every segment in use
struct InjectHead {
    int nseg, total;
    uint32_t frame, patch;
    uint64_t seed;
    int W, H, nth;
};
struct InjectPack {
    PatchDev p[kInjectMax];
    InjectHead h[kInjectMax];
    int32_t seg0[kInjectMax], giv0[kInjectMax], given[kInjectMax];
    uint32_t words[kInjectWords];
};
static_assert(sizeof(InjectPack) <= 32000, "kernel parameters");
static_assert(sizeof(Segment) % 4 == 0, "segments in words");

__global__ void __launch_bounds__(kTpb) k_inject_pack(const __grid_constant__ InjectPack pk) {
    const int k = blockIdx.y;
    pdl_enter();
    const int32_t* g = reinterpret_cast<const int32_t*>(pk.words + pk.giv0[k]);
    inject_body(pk.p[k], pk.h[k], reinterpret_cast<const Segment*>(pk.words + pk.seg0[k]), g, g + pk.given[k],
                g + 2 * pk.given[k]);
}

// the frame's plans in device memory, one per patch (CUDA-graph replay and
// the server's ticks)
template <int M>
__global__ void __launch_bounds__(kTpb) k_inject_dev(const __grid_constant__ PatchPack<M> pk, const InjectParams* ips) {
    pdl_enter();
    const InjectParams& ip = ips[blockIdx.y];
    inject_body(pk.p[M == 1 ? 0 : blockIdx.y], ip, ip.seg, ip.gx, ip.gy, ip.ga);
}

// ---- a6: binning ---------------------------------------------------------------
// The keys of a state as it stands (a resynthesis: no step made them).  Block
// b takes the kTileS / 2 particles of key tile b.
template <int M>
__global__ void __launch_bounds__(kTpb) k_bin_keys(const __grid_constant__ PatchPack<M> pk) {
    __shared__ KeyCounts C;
    const PatchDev& p = pk.p[M == 1 ? 0 : blockIdx.y];
    pdl_enter();
    if (M > 1 && (int)blockIdx.x >= p.nblk_s) return;
    clear_sort_words(p);
    const int n = live_count(p, kGaveUpAny);
    const int32_t* X = p.x[p.cur];
    const int32_t* Y = p.y[p.cur];
    const uint32_t* BD = p.bd[p.cur];
    unsigned long long ev = 0;
    unsigned int binned = 0;
    // the thread's kBinItems particles: every independent load first
    constexpr int kBinItems = (kTileS / 2) / kTpb;
    static_assert(kBinItems * kTpb == kTileS / 2, "whole particles per thread");
    const int b0 = blockIdx.x * (kTileS / 2), i0 = b0 + threadIdx.x;
    if (b0 >= n) return;   // (uniform)
    keys_begin(C, p);
    uint32_t bd[kBinItems];
    int32_t px[kBinItems], py[kBinItems];
#pragma unroll
    for (int m = 0; m < kBinItems; ++m) {
        const int i = i0 + m * kTpb;
        bd[m] = i < n ? BD[i] : 0u;
        px[m] = i < n ? X[i] : 0;
        py[m] = i < n ? Y[i] : 0;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kBinItems; ++m) {
        const int i = i0 + m * kTpb;
        uint32_t key[2] = {0u, 0u};
        if (i < n) {
            make_keys(p, px[m], py[m], bd[m], lookup_vq(p, bd[m]), key, ev, binned);
            store_keys(p, i, px[m], py[m], bd[m], key);
        }
        count_keys(C, p, bd[m], key, i < n);
    }
    keys_end(C, p, ev, binned);
}

// ---- one LSD radix-sort pass (8-bit digit, stable) -----------------------------
// A pass's block: 512 threads of 8 keys.  The ranking is a serial chain of one
// round per key of a thread, so a tile's time goes with the keys per thread:
// with 256 threads of 16 keys a pass over 4M keys took 42 us and one over a
// single tile 9.6 us.
constexpr int kSortTpb = 512;
constexpr int kSortWarps = kSortTpb / 32;

// Exclusive scan over the block's threads 0 .. 255 (v = 0 beyond them); one
// barrier inside, s_warp free on entry.
__device__ __forceinline__ uint32_t block_exscan256(uint32_t v, uint32_t* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31 && warp < 8) s_warp[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w)
        if (w < warp) before += s_warp[w];
    return before + x - v;
}

constexpr int kPassItems = kSortPassTile / kSortTpb;   // keys per thread
static_assert(kSortPassTile < 65536, "tile ranks and counts kept in 16 bits");
constexpr int kPassWarpKeys = 32 * kPassItems;     // keys per warp: a contiguous run of the tile
constexpr int kLbBatch = 8;                        // look-back words read per round trip

// One pass: a persistent grid whose blocks take tiles of kSortPassTile keys
// in ticket order.  A block ranks a tile's keys by digit (warp w holds the
// tile's keys [256 w, 256 w + 256) in order, so ranks follow the input
// order), publishes the tile's digit counts, and finds for each digit the
// keys of that digit in the earlier tiles by looking back over their
// published words (an inclusive prefix ends the walk) — the single-pass scan
// with decoupled look-back of Merrill and Garland.  Output position of a key:
// keys of smaller digits (the pass's digit totals, counted by the key kernel)
// + keys of its digit in earlier tiles + its rank in the tile.  The tile is
// reordered in shared memory first, so each digit's run leaves as
// consecutive stores.  A block only ever waits on tiles with earlier
// tickets, which running blocks hold or finished; every wait is bounded (the
// error flag records a timeout, after wait_cycles SM clocks).  The last block
// to finish clears the pass's digit totals and ticket for the next sort.
// Tickets start at tile first_tile: 0 in every frame; the failure-detection
// self-test starts at 1, so that tile 0's word is never published and the
// waits on it run out.  A block that gave up has summed a subset of the
// earlier tiles' counts, so its output positions stay below the true ones
// (in bounds, though the order is then wrong).
// Pass ps of every patch of the pack that has so many digits (pass ps reads
// key buffer ps & 1).  A patch's blocks share its own tickets, so its grid
// may be any size.
template <int M>
__global__ void __launch_bounds__(kSortTpb, 3) k_sort_pass(const __grid_constant__ PatchPack<M> pk, int ps,
                                                    long long wait_cycles, int first_tile) {
    __shared__ uint32_t s_k[kSortPassTile];
    __shared__ uint32_t s_v[kSortPassTile];
    __shared__ uint16_t s_wh[kSortWarps][256];   // per-warp digit counts, then the warp's offset in the digit
    __shared__ uint32_t s_ls[256];              // the digit's first position in the reordered tile
    __shared__ uint32_t s_gb[256];              // output position of reordered tile position 0 of the digit
    __shared__ uint32_t s_warp[8];
    __shared__ int s_bid;
    __shared__ bool s_last;
    const PatchDev& p = pk.p[M == 1 ? 0 : blockIdx.y];
    pdl_enter();
    if (M > 1 && ps >= sort_passes(p)) return;
    const uint32_t* const kin = p.keys[ps & 1];
    const uint32_t* const vin = p.vals[ps & 1];
    uint32_t* const kout = p.keys[1 - (ps & 1)];
    uint32_t* const vout = p.vals[1 - (ps & 1)];
    const int shift = 8 * ps;
    uint32_t* const dtot = p.hist + 256 * ps;
    uint32_t* const status = p.sort_status + (size_t)ps * p.nblk_o * 256;
    uint32_t* const ticket = p.sort_ticket + 2 * ps;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = 2 * live_count(p, kGaveUpBefore | (gave_up_pass(ps) - 1));
    const uint32_t gd = block_exscan256(tid < 256 ? dtot[tid] : 0u, s_warp);   // keys of smaller digits, all tiles
    const uint32_t lt = (1u << lane) - 1u;
    for (;;) {
        if (tid == 0) s_bid = (int)atomicAdd(ticket, 1u) + first_tile;
#pragma unroll
        for (int w = tid; w < kSortWarps * 128; w += kSortTpb) reinterpret_cast<uint32_t*>(&s_wh[0][0])[w] = 0u;
        __syncthreads();   // (also: the previous tile's shared data is no longer read)
        const int bid = s_bid;
        const int base = bid * kSortPassTile;
        if (base >= n) break;   // (uniform)
        const int i0 = base + warp * kPassWarpKeys + lane;
        uint32_t kk[kPassItems], vv[kPassItems], rk[kPassItems / 2];   // ranks (< 4096): two per word
#pragma unroll
        for (int k = 0; k < kPassItems / 2; ++k) rk[k] = 0u;
#pragma unroll
        for (int k = 0; k < kPassItems; ++k) {   // every load first
            const int i = i0 + 32 * k;
            kk[k] = i < n ? kin[i] : 0u;
            vv[k] = ps == 0 ? (uint32_t)i : i < n ? vin[i] : 0u;   // (the keys come in bump order)
        }
#pragma unroll
        for (int k = 0; k < kPassItems; ++k) {
            const bool act = i0 + 32 * k < n;
            const uint32_t d = act ? (kk[k] >> shift) & 255u : 256u + (uint32_t)lane;   // inactive: alone
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const uint32_t r = __popc(peers & lt);
            const uint32_t before = act ? s_wh[warp][d] : 0u;
            rk[k / 2] |= (before + r) << (16 * (k & 1));
            __syncwarp();
            if (act && r == 0) s_wh[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // digit tid: each warp's offset within the tile's keys of the digit
        uint32_t c = 0, excl = 0;
        if (tid < 256) {
#pragma unroll
            for (int w = 0; w < kSortWarps; ++w) {
                const uint32_t x = s_wh[w][tid];
                s_wh[w][tid] = (uint16_t)c;
                c += x;
            }
            // keys of digit tid in the earlier tiles: walk back over their words,
            // kLbBatch at a time, summing aggregates up to the nearest inclusive
            // prefix; an unpublished word ends the batch and is read again
            uint32_t* mine = status + (size_t)bid * 256 + tid;
            if (bid == 0) {
                st_relaxed(mine, kLbPrefix | c);
            } else {
                st_relaxed(mine, kLbAggregate | c);
                const long long t0 = clock64();
                int j = bid - 1;   // the nearest word not yet summed
                for (;;) {
                    uint32_t w[kLbBatch];
#pragma unroll
                    for (int q = 0; q < kLbBatch; ++q)
                        w[q] = j - q >= 0 ? ld_relaxed(status + (size_t)(j - q) * 256 + tid) : kLbPrefix;
                    bool done = false, stalled = false;
#pragma unroll
                    for (int q = 0; q < kLbBatch; ++q) {
                        if (done || stalled) continue;
                        const uint32_t f = w[q] & ~kLbCount;
                        if (f == 0u) {
                            stalled = true;   // not yet published: read again from here
                        } else {
                            excl += w[q] & kLbCount;
                            --j;
                            done = f == kLbPrefix;
                        }
                    }
                    if (done) break;
                    if (stalled && clock64() - t0 > wait_cycles) {
                        give_up(p, gave_up_pass(ps));
                        break;
                    }
                }
                st_relaxed(mine, kLbPrefix | (excl + c));
            }
        }
        const uint32_t ls = block_exscan256(c, s_warp);   // (its barrier orders s_wh above)
        if (tid < 256) {
            s_ls[tid] = ls;
            s_gb[tid] = gd + excl - ls;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPassItems; ++k) {
            if (i0 + 32 * k < n) {
                const uint32_t d = (kk[k] >> shift) & 255u;
                const uint32_t pos = s_ls[d] + s_wh[warp][d] + ((rk[k / 2] >> (16 * (k & 1))) & 0xFFFFu);
                s_k[pos] = kk[k];
                s_v[pos] = vv[k];
            }
        }
        __syncthreads();
        const int m = min(kSortPassTile, n - base);
        for (int i = tid; i < m; i += kSortTpb) {
            const uint32_t key = s_k[i];
            const uint32_t o = s_gb[(key >> shift) & 255u] + (uint32_t)i;
            kout[o] = key;
            vout[o] = s_v[i];
        }
    }
    // the last block out (every block has read the digit totals by then)
    // clears them and the ticket
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(ticket + 1, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        if (tid < 256) dtot[tid] = 0u;
        if (tid == 0) {
            ticket[0] = 0u;
            ticket[1] = 0u;
        }
        __threadfence();
    }
}

int sort_pass_blocks_per_sm() {
    static int cache[kMaxCachedDevices];
    return cached_per_device(cache, [] {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_sort_pass<1>, kSortTpb, 0) != cudaSuccess) {
            cudaGetLastError();
            return -1;
        }
        return nb > 0 ? nb : -1;
    });
}

int sm_count() {
    static int cache[kMaxCachedDevices];
    return cached_per_device(cache, [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return -1;
        }
        return n > 0 ? n : -1;
    });
}

// One pass over the sorted (key, bump id) pairs:
//  * offsets[k] = first sorted position with key >= k (k = 0..total_bins):
//    position e is the answer for every k in (key[e-1], key[e]] (for e = 0
//    from 0, for e = n up to total_bins);
//  * the bump records in bin order (X, Y, signed amplitude, id and the
//    kernel phase pairs) of the entries with a bin (key < total_bins; the
//    others sort last).
constexpr int kRecItems = 4;   // sorted entries per thread and round, loads issued together

template <int M>
__global__ void __launch_bounds__(kTpb) k_offsets_records(const __grid_constant__ PatchPack<M> pk) {
    // per warp: the 32 records of its 32 consecutive entries (1 KB), stored
    // out as 16-byte chunks of consecutive addresses (whole sectors)
    __shared__ uint4 s_rec[kTpb / 32][64];
    const PatchDev& p = pk.p[M == 1 ? 0 : blockIdx.y];
    pdl_enter();
    const uint32_t* const keys = p.keys[sort_passes(p) & 1];
    const uint32_t* const vals = p.vals[sort_passes(p) & 1];
    // the frame's statistics (the error flags stay; the synthesis counts its
    // stages and candidates from zero), and the step's look-back words and
    // ticket cleared for the next frame
    if (blockIdx.x == 0) {
        unsigned long long* const acc = stats_acc(p);
        const int t = threadIdx.x;
        if (t < 2) {
            p.stats[t] = acc[t];
            if (t == 0) p.stats[4 + p.nb] += acc[0];   // running total over frames
            acc[t] = 0ull;
        }
        if (t < p.nb) {
            p.stats[3 + t] = acc[2 + t];
            acc[2 + t] = 0ull;
        }
        if (t == p.nb) p.stats[3 + p.nb] = p.stats[5 + p.nb] = 0ull;
    }
    for (int i = blockIdx.x * kTpb + threadIdx.x; i <= p.nblk_c; i += gridDim.x * kTpb) p.blk[i] = 0u;
    const int n = 2 * live_count(p, kGaveUpAny);
    if (blockIdx.x == 0 && threadIdx.x == 0 && n == 0 && p.count[2]) p.count[2] = kGaveUpBefore;
    const int4* PK = p.pk;
    const uint32_t tb = (uint32_t)p.total_bins;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stride = gridDim.x * kTpb * kRecItems;
    // (the loop is uniform over a warp: its lanes take entries eb + lane)
    for (int eb = blockIdx.x * kTpb * kRecItems + (threadIdx.x & ~31); eb <= n; eb += stride) {
        const int e0 = eb + lane;
        uint32_t key[kRecItems], prev[kRecItems], id[kRecItems];
#pragma unroll
        for (int q = 0; q < kRecItems; ++q) {
            const int e = e0 + q * kTpb;
            key[q] = e < n ? keys[e] : tb;
            prev[q] = (e > 0 && e <= n) ? keys[e - 1] : 0u;
            id[q] = e < n ? vals[e] : 0u;
        }
        int4 st[kRecItems];
#pragma unroll
        for (int q = 0; q < kRecItems; ++q) {   // the particles' state: every gather first
            const int e = e0 + q * kTpb;
            const bool ok = e < n && key[q] < tb;
            st[q] = ok ? PK[id[q] >> 1] : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int q = 0; q < kRecItems; ++q) {
            const int e = e0 + q * kTpb;
            if (e <= n) {
                const int lo = e == 0 ? 0 : (int)prev[q] + 1;
                const int hi = e == n ? p.total_bins : min((int)key[q], p.total_bins);
                for (int k = lo; k <= hi; ++k) p.offsets[k] = (uint32_t)e;
            }
            const bool valid = e < n && key[q] < tb;
            uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0;
            if (valid) {
                const uint32_t bd = (uint32_t)st[q].z;
                const bool trough = id[q] & 1u;
                const int4 vq = lookup_vq(p, bd);
                const float A = lookup_amp(p, bd);
                const BucketDev& bk = p.bk[bd >> 16];
                const int32_t x = trough ? st[q].x - vq.z : st[q].x;
                const int32_t y = trough ? st[q].y - vq.w : st[q].y;
                // e^{-i pi (x mod 2R)/R}: exact integer reduction (2R < 2^31),
                // then sincospi of the FP32 quotient (within a few ulp of the
                // exact one)
                const int32_t R2 = 2 * bk.R;
                int32_t xm, ym;
                floor_divmod(x, R2, xm);
                floor_divmod(y, R2, ym);
                const float invR = bk.invR;
                float sx, cx, sy, cy;
                sincospif((float)xm * invR, &sx, &cx);
                sincospif((float)ym * invR, &sy, &cy);
                // BumpRec {x, cx, -sx, id, y, cy, -sy, amp}
                r0 = make_uint4((uint32_t)x, __float_as_uint(cx), __float_as_uint(-sx), id[q]);
                r1 = make_uint4((uint32_t)y, __float_as_uint(cy), __float_as_uint(-sy), __float_as_uint(trough ? -A : A));
            }
            s_rec[warp][2 * lane] = r0;
            s_rec[warp][2 * lane + 1] = r1;
            __syncwarp();
            // entries eb + q kTpb + r, r = 0 .. 31; chunk c (16 bytes) belongs
            // to entry r = c / 2 and leaves only if that entry has a record
            const unsigned vm = __ballot_sync(0xffffffffu, valid);
            uint4* const dst = reinterpret_cast<uint4*>(p.rec + (eb + q * kTpb));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = lane + 32 * h;
                if ((vm >> (c >> 1)) & 1u) dst[c] = s_rec[warp][c];
            }
            __syncwarp();
        }
    }
}

// f(pack, patches in it) over packs of the n patches at ps
template <typename F>
cudaError_t for_packs(const PatchDev* ps, int n, F&& f) {
    auto run = [&](auto tag, const PatchDev* q, int m) {
        PatchPack<decltype(tag)::value> pk;
        for (int k = 0; k < m; ++k) pk.p[k] = q[k];
        return f(pk, m);
    };
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < n && e == cudaSuccess; k += kPackMax) {
        const int m = std::min(kPackMax, n - k);
        e = m == 1   ? run(std::integral_constant<int, 1>(), ps + k, m)
            : m <= 8 ? run(std::integral_constant<int, 8>(), ps + k, m)
                     : run(std::integral_constant<int, kPackMax>(), ps + k, m);
    }
    return e;
}

template <typename PK, typename G>
int pack_max(const PK& pk, int m, G&& g) {
    int v = 1;
    for (int k = 0; k < m; ++k) v = std::max(v, (int)g(pk.p[k]));
    return v;
}

template <typename PK>
cudaError_t launch_keys(const PK& pk, int m, cudaStream_t st) {
    count_launches(1);
    return launch_pdl(k_bin_keys<PK::kM>, dim3(pack_max(pk, m, [](const PatchDev& p) { return p.nblk_s; }), m), kTpb, 0,
                      st, pk);
}

// a sort pass: up to the blocks that fit at once per patch (they take tiles
// in turn)
template <typename PK>
cudaError_t launch_sort(const PK& pk, int m, int ps, long long wait_cycles, int first_tile, cudaStream_t st) {
    const int fit = std::max(1, sort_pass_blocks_per_sm()) * std::max(1, sm_count());
    const int grid = std::min(fit, pack_max(pk, m, [](const PatchDev& p) { return p.nblk_o; }));
    count_launches(1);
    return launch_pdl(k_sort_pass<PK::kM>, dim3(grid, m), kSortTpb, 0, st, pk, ps, wait_cycles, first_tile);
}

}  // namespace

// ---- launchers -------------------------------------------------------------------
cudaError_t launch_step(const PatchDev* ps, int n, cudaStream_t st) {
    return for_packs(ps, n, [&](const auto& pk, int m) {
        constexpr int M = std::decay_t<decltype(pk)>::kM;
        count_launches(1);
        return launch_pdl(k_step<M>, dim3(pack_max(pk, m, [](const PatchDev& p) { return p.nblk_c; }), m), kTpb, 0, st,
                          pk, kLbWaitCycles, 0);
    });
}

cudaError_t launch_inject(const PatchDev* ps, const InjectParams* ips, int n, cudaStream_t st) {
    auto blocks = [](int total) { return std::min(1024, std::max(1, (total + kTpb - 1) / kTpb)); };
    // the patches that inject in this frame
    int idx[kInjectMax];
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < n && e == cudaSuccess;) {
        int m = 0, used = 0, most = 1;
        for (; k < n && m < kInjectMax; ++k) {
            const InjectParams& ip = ips[k];
            if (ip.total <= 0) continue;
            const int need = ip.nseg * (int)(sizeof(Segment) / 4) + 3 * ip.given;
            if (m > 0 && used + need > kInjectWords) break;
            idx[m++] = k;
            used += need;
            most = std::max(most, blocks(ip.total));
        }
        if (m == 0) break;
        count_launches(1);
        if (m == 1) {
            e = launch_pdl(k_inject, most, kTpb, 0, st, ps[idx[0]], ips[idx[0]]);
            continue;
        }
        InjectPack pk;
        int w = 0;
        for (int j = 0; j < m; ++j) {
            const InjectParams& ip = ips[idx[j]];
            pk.p[j] = ps[idx[j]];
            pk.h[j] = InjectHead{ip.nseg, ip.total, ip.frame, ip.patch, ip.seed, ip.W, ip.H, ip.nth};
            pk.seg0[j] = w;
            memcpy(pk.words + w, ip.seg, ip.nseg * sizeof(Segment));
            w += ip.nseg * (int)(sizeof(Segment) / 4);
            pk.giv0[j] = w;
            pk.given[j] = ip.given;
            for (const int32_t* src : {ip.gx, ip.gy, ip.ga}) {
                memcpy(pk.words + w, src, ip.given * sizeof(int32_t));
                w += ip.given;
            }
        }
        e = launch_pdl(k_inject_pack, dim3(most, m), kTpb, 0, st, pk);
    }
    return e;
}

cudaError_t launch_inject_dev(const PatchDev* ps, const InjectParams* ips_dev, int n, cudaStream_t st) {
    const InjectParams* d = ips_dev;
    return for_packs(ps, n, [&](const auto& pk, int m) {
        constexpr int M = std::decay_t<decltype(pk)>::kM;
        count_launches(1);
        // the frame's counts are not known here: 8,192 particles a pass of the grid
        const cudaError_t e = launch_pdl(k_inject_dev<M>, dim3(32, m), kTpb, 0, st, pk, d);
        d += m;
        return e;
    });
}

cudaError_t launch_bin(const PatchDev* ps, int n, bool keys, cudaStream_t st) {
    return for_packs(ps, n, [&](const auto& pk, int m) {
        constexpr int M = std::decay_t<decltype(pk)>::kM;
        const int passes = pack_max(pk, m, [](const PatchDev& p) { return sort_passes(p); });
        cudaError_t e = keys ? launch_keys(pk, m, st) : cudaSuccess;
        for (int s = 0; s < passes && e == cudaSuccess; ++s) e = launch_sort(pk, m, s, kLbWaitCycles, 0, st);
        if (e != cudaSuccess) return e;
        const int rb = pack_max(pk, m, [](const PatchDev& p) {
            return (2 * (int64_t)p.cap + 1 + kTpb * kRecItems - 1) / (kTpb * kRecItems);
        });
        count_launches(1);
        return launch_pdl(k_offsets_records<M>, dim3(std::min(rb, std::max(1, sm_count()) * 8), m), kTpb, 0, st, pk);
    });
}

cudaError_t launch_step_stall(const PatchDev& p, long long wait_cycles, cudaStream_t st) {
    PatchPack<1> pk;
    pk.p[0] = p;
    count_launches(1);
    return launch_pdl(k_step<1>, dim3(p.nblk_c), kTpb, 0, st, pk, wait_cycles, 1);
}

int sorted_buffer_index(const PatchDev& p) { return sort_passes(p) & 1; }

cudaError_t launch_sort_stall(const PatchDev& p, long long wait_cycles, cudaStream_t st) {
    // the frame's keys and digit totals, then the first pass with tile 0
    // never taken: every block that looks back to it waits wait_cycles
    PatchPack<1> pk;
    pk.p[0] = p;
    const cudaError_t e = launch_keys(pk, 1, st);
    return e == cudaSuccess ? launch_sort(pk, 1, 0, wait_cycles, 1, st) : e;
}

}  // namespace scwp
