// Summed-area synthesis of the wave-particle maps: the per-bucket kernel
// sums of Sec. 4.2 (kernel reading O11, analytic displacement O12) computed
// from the structure of the raised-cosine kernel instead of one evaluation
// per (bump, texel) pair.
//
// On its support |X - x_b| < R a bump's x factor is
//     1 + cos(pi (X - x_b)/R) = u(X) . p_b,   sin(pi (X - x_b)/R) = u'(X) . p_b,
// with u(X) = (1, cos a_X, -sin a_X), u'(X) = (0, sin a_X, cos a_X),
// a_X = pi (X mod 2R)/R and p_b = (1, c_b, s_b) = (1, e^{-i pi (x_b mod 2R)/R})
// (the bump record's phase pair); likewise v(Y), v'(Y), q_b for y.  Within a
// tile the support is a box [alpha_b, beta_b) x [gamma_b, delta_b) of texel
// indices, so
//     h(X, Y)  = 1/4     sum_ij u_i(X)  v_j(Y)  S_ij(X, Y),
//     Dx(X, Y) = lam/4   sum_ij u'_i(X) v_j(Y)  S_ij(X, Y),
//     Dy(X, Y) = lam/4   sum_ij u_i(X)  v'_j(Y) S_ij(X, Y),
//     S_ij(X, Y) = sum_b A_b p_i(b) q_j(b) [alpha_b <= X < beta_b][gamma_b <= Y < delta_b],
// and S_ij is the 2-D inclusive prefix sum of a difference array that holds
// +-A_b p_i q_j at the four corners of each box (corners at index 64 fall
// outside the tile and are dropped).  These are the same sums as the direct
// gather in another association.  Per (tile, bucket) the work is four corner
// events per bump, two prefix passes and a 3 x 3 contraction per texel: it
// no longer grows with the number of bumps covering a texel.
//
// Exactness of the prefix sums: the corner weights are rounded once to
// 32-bit integers with a per-pass scale 2^30 / (1.001 m A_max), m the
// candidate bumps of the pass and A_max the bucket's bound on |A| (its
// direction amplitudes, and the wake's).  Every S_ij then fits in 31 bits, the
// events accumulate exactly in any order (integer shared-memory atomics:
// deterministic results), and the prefix sums are exact modulo 2^32 (their
// intermediate values may wrap; the final ones do not).  The contraction is
// FP32.  The rounding error of a weight is at most 2^-31 m A_max; those of the
// n candidates covering a texel add up to about sqrt(n) m A_max 2^-31, so a
// (tile, bucket) whose n is large against the bound the host sets per bucket
// (BucketDev::sat_c) is split into passes of fewer candidates, each with its
// own scale, prefix sums and contraction (the FP32 accumulators carry over).
//
// Organisation: a persistent grid, one 1024-thread CTA per SM, pulls (tile,
// bucket group) items from a work queue (an atomic ticket over the plan's
// heaviest-first order; the last CTA to finish resets the queue for the next
// launch, so no CTA ever waits on another).  All nine S_ij planes of a
// bucket live in shared memory at once (144 KB), so each candidate bump
// enters exactly once per pass.  An item is worked off in batches: the bin
// rows of its buckets that reach the tile are read into a row table (all of
// them, in nearly every item; a bucket with more rows than the table spans
// several segments, each a pass of its own).  Two batches are held: eight
// warps build the next one (the next item's ticket, descriptors, bucket
// geometry and row table: five dependent round trips to L2) in the x-prefix
// phase of this one's last pass but one, which leaves them idle, so an item
// starts without a wait and its first records are already on their way
// (512^2 patch, 100k particles: frame 144.7 -> 136.1 us).  One thread
// describes the next pass in the y-prefix phase.
// Within a pass each thread takes the candidates c0 + tid, c0 + tid + 1024,
// ... on its own, with no barrier until the pass ends: its warp finds the
// candidates' bin rows (a ballot over the row table) and it copies the
// record with asynchronous 16-byte copies (cp.async) into its own slot of
// two, one candidate ahead, so the copy of its next candidate (of this pass,
// or the first of the next pass) overlaps the current one's events, and the
// next pass's first copies overlap the prefix passes.  As each thread reads
// only the slots it filled, no barrier guards them.  Each thread clips its
// candidate's support box to the tile and adds the nine weights at up to
// four corners; bumps whose box starts at the tile's first texel in both axes
// (every bump covering the whole tile among them) sum their (0, 0) corner in
// registers, added per lane to 32 words per plane that the x prefix sums.
// Then the x prefix (one row of one plane per thread), the y prefix (one column of one plane per
// thread, stored only at the first row of each 4-row segment of the
// contraction) and the contraction (one column of a segment per thread),
// which finishes the y prefix of the segment's other rows in registers and
// zeroes every difference-array element it reads, so no pass needs a
// clearing phase.
//
// What bounds it: shared-memory wavefronts and issue.  A pass of 1,000
// candidates (1024^2 patch, 200k particles) takes about 13,000 cycles: events
// 3,100 (75 a warp's 32 candidates), x prefix 3,250, y prefix 2,300,
// contraction 3,100; the prefixes and the contraction alone are 6,048
// wavefronts.  The description and the lane-wise corner took it from 16,000
// (frame 311 -> 292 us; 8 patches of 2M particles 6.75 -> 6.45 ms).  Walking
// quads of four columns along y with 144 threads, and scanning them along x
// by shuffles in the contraction, was 15-20 % slower: too few warps to keep
// the pipe busy, and as many wavefronts for the shuffles as they saved.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "blend_dev.cuh"
#include "internal.h"

namespace scwp {
namespace {

constexpr int kT = 64;                       // tile side in texels
constexpr int kSatThreads = 1024;
constexpr int kSegs = kSatThreads / kT;      // row segments of the contraction
constexpr int kSegRows = kT / kSegs;         // rows per segment
constexpr int kPlanes = 9;                   // S_ij, plane 3 i + j
constexpr int kScanThreads = kPlanes * kT;   // one row (or column) scan per thread
constexpr int kRowCap = 256;                 // bin rows held at once (all segments of a batch)
constexpr int kMaxSeg = 64;                  // segments per batch
constexpr int32_t kQs = 65536, kHalfs = 32768;
static_assert(kSegs * kSegRows == kT && kSegs == 16, "contraction mapping");
static_assert(kScanThreads % 32 == 0, "whole scan warps");

constexpr int kBuildWarp0 = 24;              // warps 24 .. 31 build the next batch
constexpr int kBuildThreads = kSatThreads - 32 * kBuildWarp0;
static_assert(kScanThreads + 2 * kT + 32 <= 32 * kBuildWarp0, "phase threads and builders apart");

// A batch of one item: segments (bucket, row range) whose bin rows fit the row table.
struct Batch {
    int32_t rs[kRowCap];                  // first record of each bin row of the batch
    int32_t cum[kRowCap];                 // candidates of the segment before the row
    // the segments: bucket, half-width, |A| bound, first table row, candidates, candidates per pass
    int32_t sgb[kMaxSeg], sgR[kMaxSeg], sgrb[kMaxSeg + 1], sgnc[kMaxSeg], sgm[kMaxSeg];
    float sgA[kMaxSeg];
    int32_t item, nseg, last;             // last: the item's last batch
    int32_t t_next, r0_next;              // else the bucket (item-relative) and row the next one starts at
    int32_t tx0, ty0, planes, plane, K, part;   // partial planes of the item's tile and its own; parts
    int32_t patch;                        // the patch whose descriptors pd, spd hold (-1: none)
    alignas(16) unsigned char pd[sizeof(PatchDev)];
    alignas(16) unsigned char spd[sizeof(SynthParams)];
};

// A pass as its threads read it: written once, by one thread, in the y-prefix
// phase of the pass before (worked out by every warp for itself, it took
// about 1,000 of a pass's 16,000 cycles).
struct alignas(16) PassDesc {
    int32_t s, c0, c1, rb, re;            // segment (kEmpty, kDone: none), candidates, row table rows
    int32_t R, bucket, batch;
    int32_t X0, Y0;                       // Q16.16 centre of the tile's first texel
    float scale, inv;
    int32_t fetched;                      // its first copies are on their way already
    int32_t build;                        // its x-prefix phase builds the next batch
    int32_t built;                        // ... is there after that phase
    int32_t last;                         // the batch's last pass
    int32_t f_batch, f_c0, f_c1, f_rb, f_re;   // the pass whose first copies this one starts (f_c0 == f_c1: none)
};
constexpr int kEmpty = -1, kDone = -2;    // a batch without a pass; no more items
constexpr int kDescThread = 32 * kBuildWarp0 - 32;   // a thread of a warp that neither scans nor builds

struct SatSmem {
    uint32_t E[kPlanes][kT * kT];         // difference arrays, then prefix sums; zero between passes
    alignas(128) BumpRec raw[2][kSatThreads];   // two record slots per thread
    alignas(16) float2 ph[2 * kT];        // texel phases (cos, sin) a of the pass's bucket: rows, then columns
    alignas(16) uint32_t Z[kPlanes][32];  // the (0, 0) corner of the pass, per lane; zero between passes
    PassDesc pass[2];
    Batch bt[2];
    // the builders' table of the item's buckets, and the segments' first rows
    int32_t mR[kMaxBuckets], mnbx[kMaxBuckets], mbase[kMaxBuckets];
    int32_t mbx_lo[kMaxBuckets], mbx_hi[kMaxBuckets], mby_lo[kMaxBuckets], mnrows[kMaxBuckets];
    float mamax[kMaxBuckets], msatc[kMaxBuckets];
    int32_t sgr0[kMaxSeg];
};
static_assert(sizeof(SatSmem) <= 227 * 1024, "shared memory of one CTA");
static_assert(sizeof(BumpRec) == 32, "32-byte records (two 16-byte copies)");

// element (row y, column x) of a 64 x 64 plane: columns XOR-swizzled by the
// row so that a warp walking a row (one row per lane) or a column (one
// column per lane) touches 32 different banks
__device__ __forceinline__ int sw(int y, int x) { return y * kT + (x ^ (y & 31)); }

__device__ __forceinline__ int clamp_t(int t) { return min(max(t, 0), kT); }

// the nine components of one corner event
__device__ __forceinline__ void event9(SatSmem& S, int x, int y, const uint32_t (&w)[kPlanes]) {
    const int o = sw(y, x);
#pragma unroll
    for (int k = 0; k < kPlanes; ++k) atomicAdd(&S.E[k][o], w[k]);
}

// inclusive warp scan of v
__device__ __forceinline__ uint32_t warp_scan(uint32_t v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += t;
    }
    return v;
}

// passes of segment candidates: a (tile, bucket) of n candidates goes in
// ceil(n^1.5 / sat_c) passes, so that the integer rounding of its corner
// weights stays within the bound the host set
__device__ __forceinline__ int pass_size(int ncand, float satc) {
    const float nf = (float)ncand;
    const int kch = max(1, (int)ceilf(nf * sqrtf(nf) / satc));
    return (ncand + kch - 1) / kch;
}

// ---- asynchronous 16-byte copies global -> shared (L2 only)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// wait until at most one group of this thread's copies is still in flight
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Record slots are 32 bytes per thread.  Threads with bit 2 of their index
// set keep the two 16-byte halves of their record in swapped order, so that
// the eight threads of a quarter warp (whose 16-byte accesses one shared
// memory wavefront serves) touch eight different 16-byte bank groups: the
// copies into the slots and the reads from them are free of bank conflicts
// (with the halves in order, threads t and t + 4 met in the same banks).
__device__ __forceinline__ int half_swap(int tid) { return (tid >> 2) & 1; }

// A pass of this CTA's part: segment s, its candidates [c0, c1); s < 0: none.
struct Pass {
    int s, c0, c1;
};

__device__ __forceinline__ Pass make_pass(const Batch& B, int s, int c0) {
    return Pass{s, c0, min(B.sgnc[s], c0 + B.sgm[s])};
}

// The part's first pass of segments s0, s0 + 1, ... with candidates.
__device__ __forceinline__ Pass first_pass_from(const Batch& B, int s0) {
    for (int s = s0; s < B.nseg; ++s)
        if (B.part * B.sgm[s] < B.sgnc[s]) return make_pass(B, s, B.part * B.sgm[s]);
    return Pass{-1, 0, 0};
}

// The pass after P in this part's order: the part's next pass of the same
// segment (parts take every K-th pass), else the first of a later segment.
__device__ __forceinline__ Pass next_pass(const Batch& B, Pass P) {
    const int c0 = P.c0 + B.K * B.sgm[P.s];
    if (c0 < B.sgnc[P.s]) return make_pass(B, P.s, c0);
    return first_pass_from(B, P.s + 1);
}

// This thread's copy of candidate j0 + lane (if below c1) of the segment whose
// table rows are [qb, re) into its slot; qb moves on to the row of j0.  A
// candidate's row is the last one that starts at or before it (empty rows
// start where the next one does): the warp finds that of its first candidate
// with one load and a ballot per 32 rows, each lane steps on from there (a
// bisection per lane took twice the instructions).
__device__ __forceinline__ void fetch(BumpRec* slot, const Batch& B, int& qb, int re, int j0, int c1, int tid) {
    const int lane = tid & 31;
    for (;;) {
        const unsigned m = __ballot_sync(0xffffffffu, qb + lane < re && B.cum[qb + lane] <= j0);
        if (m != 0xffffffffu) {   // (the rows that start at or before j0 come first)
            qb += __popc(m) - 1;
            break;
        }
        qb += 32;
    }
    const int j = j0 + lane;
    if (j < c1) {
        int r = qb;
        while (r + 1 < re && B.cum[r + 1] <= j) ++r;
        const BumpRec* const rec = reinterpret_cast<const PatchDev*>(B.pd)->rec;
        const unsigned char* src = reinterpret_cast<const unsigned char*>(rec + B.rs[r] + (j - B.cum[r]));
        unsigned char* dst = reinterpret_cast<unsigned char*>(slot + tid);
        const int hs = half_swap(tid);
        cp_async16(dst + 16 * hs, src);
        cp_async16(dst + 16 * (hs ^ 1), src + 16);
    }
}

// Pass P of batch b into D.  built: the batch after it is built (so that P can
// start the copies of that one's first pass).  One thread.
__device__ void describe(SatSmem& S, PassDesc& D, int b, Pass P, bool fetched, bool built, int n_items) {
    const Batch& B = S.bt[b];
    D.batch = b;
    D.s = P.s;
    D.last = 1;
    if (P.s < 0) {
        D.s = kEmpty;
        return;
    }
    const float bound = 1.001f * (float)(P.c1 - P.c0) * B.sgA[P.s];   // >= every |S_ij| of the pass
    D.scale = 1073741824.f / bound;                                  // 2^30 / bound
    D.inv = bound * (1.f / 1073741824.f);                            // 1 / scale
    D.c0 = P.c0;
    D.c1 = P.c1;
    D.rb = B.sgrb[P.s];
    D.re = B.sgrb[P.s + 1];
    D.R = B.sgR[P.s];
    D.bucket = B.sgb[P.s];
    D.X0 = B.tx0 * kQs + kHalfs;
    D.Y0 = B.ty0 * kQs + kHalfs;
    D.fetched = fetched;
    const Pass Pn = next_pass(B, P);
    D.last = Pn.s < 0;
    // the next batch, as late as its first copies allow (a ticket taken early
    // is work other CTAs cannot take)
    D.build = !built && (Pn.s < 0 || next_pass(B, Pn).s < 0);
    D.built = built || D.build;
    Pass Pf = Pn;
    D.f_batch = b;
    if (Pn.s < 0 && built) {
        D.f_batch = b ^ 1;
        if (S.bt[b ^ 1].item < n_items) Pf = first_pass_from(S.bt[b ^ 1], 0);
    }
    const Batch& Bf = S.bt[D.f_batch];
    D.f_c0 = Pf.s < 0 ? 0 : Pf.c0;
    D.f_c1 = Pf.s < 0 ? 0 : Pf.c1;
    D.f_rb = Pf.s < 0 ? 0 : Bf.sgrb[Pf.s];
    D.f_re = Pf.s < 0 ? 0 : Bf.sgrb[Pf.s + 1];
}

// The first pass of batch b into D.
__device__ void describe_first(SatSmem& S, PassDesc& D, int b, bool fetched, int n_items) {
    if (S.bt[b].item >= n_items) {
        D.s = kDone;
        return;
    }
    describe(S, D, b, first_pass_from(S.bt[b], 0), fetched, false, n_items);
}

__device__ __forceinline__ void builders_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(kBuildThreads) : "memory");
}

// Build the batch after batch nx ^ 1 into batch nx (the eight builder warps;
// bt: thread among them): more of the same item if that one was not its
// last, else the next item of the queue.  Readers need a block barrier.
__device__ void build_batch(SatSmem& S, int nx, bool more, const TcItem* items, int n_items, const PatchDev* pdevs,
                            const SynthParams* sps, unsigned int* queue, int bt) {
    Batch& B = S.bt[nx];
    const Batch& A = S.bt[nx ^ 1];
    const int lane = bt & 31, bw = bt >> 5;
    if (bt == 0) B.item = more ? A.item : (int)atomicAdd(queue, 1u);
    builders_sync();
    const int ti = B.item;
    if (ti >= n_items) return;
    const TcItem it = items[ti];
    if (it.patch != B.patch) {   // (uniform) items of one patch share its descriptors
        static_assert(sizeof(PatchDev) % 4 == 0 && sizeof(SynthParams) % 4 == 0, "descriptor copy");
        const uint32_t* a = reinterpret_cast<const uint32_t*>(pdevs + it.patch);
        const uint32_t* b = reinterpret_cast<const uint32_t*>(sps + it.patch);
        for (int k = bt; k < (int)(sizeof(PatchDev) / 4); k += kBuildThreads) reinterpret_cast<uint32_t*>(B.pd)[k] = a[k];
        for (int k = bt; k < (int)(sizeof(SynthParams) / 4); k += kBuildThreads)
            reinterpret_cast<uint32_t*>(B.spd)[k] = b[k];
        builders_sync();
        if (bt == 0) B.patch = it.patch;
    }
    const PatchDev& p = *reinterpret_cast<const PatchDev*>(B.pd);
    const SynthParams& sp = *reinterpret_cast<const SynthParams*>(B.spd);
    const int G = item_groups(it), g = item_group(it), K = item_parts(it), part = item_part(it);
    const int ntx = (sp.W + kT - 1) / kT;
    const int tx0 = (it.tile % ntx) * kT, ty0 = (it.tile / ntx) * kT;
    const int b_begin = max((g * sp.nb) / G, sp.b_lo);
    const int nbk = max(0, min(((g + 1) * sp.nb) / G, sp.b_hi) - b_begin);
    // Q16.16 centres of the tile's first and last texel columns and rows
    const int32_t X0 = tx0 * kQs + kHalfs, X1 = X0 + (kT - 1) * kQs;
    const int32_t Y0 = ty0 * kQs + kHalfs, Y1 = Y0 + (kT - 1) * kQs;
    // ---- the item's buckets, one thread each: bins hold x_b + R in
    // [bx C, (bx + 1) C); the bin rows and columns that reach the tile
    static_assert(kMaxBuckets <= 64 && kMaxSeg >= kMaxBuckets && kMaxBuckets <= kBuildThreads, "two buckets per lane");
    if (bt < nbk) {
        const BucketDev bk = p.bk[b_begin + bt];
        const float amax = p.amax[b_begin + bt];
        const int bx_lo = (int)((int64_t)X0 / bk.C);
        const int bx_hi = min((int)(((int64_t)X1 + 2 * (int64_t)bk.R - 1) / bk.C), bk.nbx - 1);
        const int by_lo = (int)((int64_t)Y0 / bk.C);
        const int by_hi = min((int)(((int64_t)Y1 + 2 * (int64_t)bk.R - 1) / bk.C), bk.nby - 1);
        S.mR[bt] = bk.R;
        S.mnbx[bt] = bk.nbx;
        S.mbase[bt] = bk.base;
        S.mbx_lo[bt] = bx_lo;
        S.mbx_hi[bt] = bx_hi;
        S.mby_lo[bt] = by_lo;
        S.mnrows[bt] = (bx_lo > bx_hi || by_lo > by_hi || !(amax > 0.f)) ? 0 : by_hi - by_lo + 1;
        S.mamax[bt] = amax;
        S.msatc[bt] = bk.sat_c;
    }
    builders_sync();
    // ---- segments (bucket, row range) whose bin rows fit the row table
    if (bw == 0) {
        const int t0 = more ? A.t_next : 0, r0 = more ? A.r0_next : 0;
        int rows[2], before[2], nrow = 0, n = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = lane + 32 * h;
            rows[h] = t >= t0 && t < nbk ? S.mnrows[t] - (t == t0 ? r0 : 0) : 0;
            const uint32_t inc = warp_scan((uint32_t)rows[h], lane);
            before[h] = nrow + (int)inc - rows[h];
            nrow += (int)__shfl_sync(0xffffffffu, inc, 31);
        }
        if (nrow <= kRowCap) {   // all that are left
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = lane + 32 * h;
                const unsigned m = __ballot_sync(0xffffffffu, rows[h] > 0);
                if (rows[h] > 0) {
                    const int s = n + __popc(m & ((1u << lane) - 1u));
                    B.sgb[s] = t;
                    S.sgr0[s] = t == t0 ? r0 : 0;
                    B.sgrb[s] = before[h];
                }
                n += __popc(m);
            }
            if (lane == 0) {
                B.sgrb[n] = nrow;
                B.nseg = n;
                B.last = 1;
            }
        } else if (lane == 0) {
            int rws = 0, t = t0, r = r0;
            while (t < nbk && n < kMaxSeg) {
                const int left = S.mnrows[t] - r;
                if (left <= 0) {
                    ++t;
                    r = 0;
                    continue;
                }
                const int take = min(left, kRowCap - rws);
                if (take <= 0) break;
                B.sgb[n] = t;
                S.sgr0[n] = r;
                B.sgrb[n] = rws;
                rws += take;
                ++n;
                r += take;
                if (r >= S.mnrows[t]) {
                    ++t;
                    r = 0;
                }
            }
            B.sgrb[n] = rws;
            B.nseg = n;
            B.last = t >= nbk ? 1 : 0;
            B.t_next = t;
            B.r0_next = r;
        }
        if (lane == 0) {
            B.tx0 = tx0;
            B.ty0 = ty0;
            B.planes = G * K;
            B.plane = g * K + part;
            B.K = K;
            B.part = part;
        }
    }
    builders_sync();
    // ---- the row table: first record of every row, and the exclusive prefix
    // of the rows' lengths within each segment (warp w: segments w, w + 8, ...)
    for (int s = bw; s < B.nseg; s += kBuildThreads / 32) {
        const int t = B.sgb[s], q0 = B.sgrb[s], q1 = B.sgrb[s + 1], nbx = S.mnbx[t];
        const uint32_t* const off = p.offsets + (S.mbase[t] + (S.mby_lo[t] + S.sgr0[s]) * nbx);
        const int lo = S.mbx_lo[t], hi = S.mbx_hi[t] + 1;
        uint32_t carry = 0u;
        for (int q = q0; q < q1; q += 32) {
            uint32_t l = 0u;
            if (q + lane < q1) {
                const int r = (q - q0 + lane) * nbx;
                const uint32_t s0 = off[r + lo];
                l = off[r + hi] - s0;
                B.rs[q + lane] = (int32_t)s0;
            }
            const uint32_t inc = warp_scan(l, lane);
            if (q + lane < q1) B.cum[q + lane] = (int32_t)(carry + inc - l);
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) {
            B.sgnc[s] = (int32_t)carry;
            B.sgm[s] = carry ? pass_size((int)carry, S.msatc[t]) : 0;
            B.sgR[s] = S.mR[t];
            B.sgA[s] = S.mamax[t];
        }
        __syncwarp();
        if (lane == 0) B.sgb[s] = b_begin + t;   // (absolute from here on; only this warp reads it above)
    }
}

// The record of this thread's slot (its two 16-byte halves in the order
// half_swap gives).
__device__ __forceinline__ BumpRec read_slot(const SatSmem& S, int slot, int tid) {
    const uint4* q = reinterpret_cast<const uint4*>(&S.raw[slot][tid]);
    const int hs = half_swap(tid);
    const uint4 a = q[hs], b = q[hs ^ 1];
    BumpRec r;
    r.x = (int32_t)a.x;
    r.cx = __uint_as_float(a.y);
    r.sx = __uint_as_float(a.z);
    r.id = a.w;
    r.y = (int32_t)b.x;
    r.cy = __uint_as_float(b.y);
    r.sy = __uint_as_float(b.z);
    r.amp = __uint_as_float(b.w);
    return r;
}

__global__ void __launch_bounds__(kSatThreads, 1) k_synth_sat(const TcItem* items, int n_items,
                                                            const PatchDev* pdevs, const SynthParams* sps,
                                                            unsigned int* queue) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SatSmem& S = *reinterpret_cast<SatSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // contraction: this thread owns texel column cx of rows sg*4 .. sg*4 + 3
    const int cx = tid & (kT - 1), sg = tid / kT;
    pdl_enter();
    if (warp >= kBuildWarp0) {   // the first item
        const int bt = tid - 32 * kBuildWarp0;
        if (bt < 2) S.bt[bt].patch = -1;
        build_batch(S, 0, false, items, n_items, pdevs, sps, queue, bt);
    } else {   // E and Z start zeroed, and every pass leaves them zeroed again
        uint4* e4 = reinterpret_cast<uint4*>(&S.E[0][0]);
        for (int k = tid; k < kPlanes * kT * kT / 4; k += 32 * kBuildWarp0) e4[k] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < kPlanes * 32) (&S.Z[0][0])[tid] = 0u;
    }
    __syncthreads();
    if (tid == kDescThread) describe_first(S, S.pass[0], 0, false, n_items);
    __syncthreads();
    float ah[kSegRows], adx[kSegRows], ady[kSegRows];
#pragma unroll
    for (int r = 0; r < kSegRows; ++r) ah[r] = adx[r] = ady[r] = 0.f;
    int dp = 0, k = 0;          // the pass's description; the record slot of the next candidate
    for (;;) {
        const PassDesc& D = S.pass[dp];
        if (D.s == kDone) break;
        const Batch& B = S.bt[D.batch];
        const PatchDev& p = *reinterpret_cast<const PatchDev*>(B.pd);
        const SynthParams& sp = *reinterpret_cast<const SynthParams*>(B.spd);
        if (D.s == kEmpty) {
            __syncthreads();
            if (warp >= kBuildWarp0)
                build_batch(S, D.batch ^ 1, !B.last, items, n_items, pdevs, sps, queue, tid - 32 * kBuildWarp0);
            __syncthreads();
            if (tid == kDescThread) describe_first(S, S.pass[dp ^ 1], D.batch ^ 1, false, n_items);
            __syncthreads();
        } else {
            {
                // ---- the pass's events.  Invariant from here on: if this
                // thread has a candidate (c0 + tid < c1), its record is on
                // the way into slot k (the last commit group).
                const int c1 = D.c1, R = D.R;
                const int32_t X0 = D.X0, Y0 = D.Y0;
                const float scale = D.scale;
                int j0 = D.c0 + 32 * warp, q = D.rb;   // the warp's next candidates and a row at or before theirs
                if (!D.fetched) {
                    if (j0 < c1) fetch(S.raw[k], B, q, D.re, j0, c1, tid);
                    cp_async_commit();
                }
                // the copies of the next pass's first candidates, once this warp has no more of its own
                auto fetch_next = [&](int slot) {
                    const int jf = D.f_c0 + 32 * warp;
                    int qf = D.f_rb;
                    if (jf < D.f_c1) fetch(S.raw[slot], S.bt[D.f_batch], qf, D.f_re, jf, D.f_c1, tid);
                };
                // the (0, 0) corner, shared by every bump whose box starts at
                // the tile's first texel in both axes: per-thread sums
                uint32_t z[kPlanes];
#pragma unroll
                for (int q = 0; q < kPlanes; ++q) z[q] = 0u;
                bool hz = false;
                if (j0 >= c1) {
                    fetch_next(k);
                    cp_async_commit();
                }
                for (; j0 < c1; j0 += kSatThreads) {   // (uniform over the warp)
                    // the copy of this thread's next candidate starts now
                    if (j0 + kSatThreads < c1)
                        fetch(S.raw[k ^ 1], B, q, D.re, j0 + kSatThreads, c1, tid);
                    else
                        fetch_next(k ^ 1);
                    cp_async_commit();
                    cp_async_wait_prev();   // this candidate's record has landed
                    const BumpRec rc = read_slot(S, k, tid);
                    k ^= 1;
                    if (j0 + lane >= c1) continue;
                    // texel t of the tile is inside iff x_b - R < X0 + t Q < x_b + R
                    const int a = clamp_t(((rc.x - R - X0) >> 16) + 1);
                    const int bb = clamp_t(-((X0 - rc.x - R) >> 16));
                    const int c = clamp_t(((rc.y - R - Y0) >> 16) + 1);
                    const int d = clamp_t(-((Y0 - rc.y - R) >> 16));
                    if (a < bb && c < d) {
                        const float A = rc.amp;
                        const float m0 = A * scale, m1 = A * rc.cx * scale, m2 = A * rc.sx * scale;
                        uint32_t w[kPlanes];
                        w[0] = (uint32_t)__float2int_rn(m0);
                        w[1] = (uint32_t)__float2int_rn(m0 * rc.cy);
                        w[2] = (uint32_t)__float2int_rn(m0 * rc.sy);
                        w[3] = (uint32_t)__float2int_rn(m1);
                        w[4] = (uint32_t)__float2int_rn(m1 * rc.cy);
                        w[5] = (uint32_t)__float2int_rn(m1 * rc.sy);
                        w[6] = (uint32_t)__float2int_rn(m2);
                        w[7] = (uint32_t)__float2int_rn(m2 * rc.cy);
                        w[8] = (uint32_t)__float2int_rn(m2 * rc.sy);
                        if (a == 0 && c == 0) {
#pragma unroll
                            for (int q = 0; q < kPlanes; ++q) z[q] += w[q];
                            hz = true;
                        } else {
                            event9(S, a, c, w);
                        }
                        if (bb < kT && d < kT) event9(S, bb, d, w);
#pragma unroll
                        for (int q = 0; q < kPlanes; ++q) w[q] = 0u - w[q];
                        if (bb < kT) event9(S, bb, c, w);
                        if (d < kT) event9(S, a, d, w);
                    }
                }
                // the (0, 0) corner by lane: 32 different banks, where one
                // reduction per warp and plane and an add to nine shared words
                // took 1,100 cycles a pass
                __syncwarp();
                if (__any_sync(0xffffffffu, hz)) {
#pragma unroll
                    for (int q = 0; q < kPlanes; ++q) atomicAdd(&S.Z[q][lane], z[q]);
                }
                __syncthreads();   // E holds the pass's events
                if (tid < kScanThreads) {
                    // ---- prefix along x: one row of one plane per thread, in
                    // chunks of 4 with the next chunk loaded before this one
                    // is stored (the loads need not wait for the stores)
                    uint32_t* E = S.E[tid / kT];
                    const int y = tid % kT;
                    uint32_t cr[4], nx[4], run = 0u;
#pragma unroll
                    for (int k = 0; k < 4; ++k) cr[k] = E[sw(y, k)];
                    if (y == 0) {   // the (0, 0) corner's sum
                        uint4* const Z4 = reinterpret_cast<uint4*>(S.Z[tid / kT]);
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const uint4 v = Z4[k];
                            run += (v.x + v.y) + (v.z + v.w);
                            Z4[k] = make_uint4(0u, 0u, 0u, 0u);
                        }
                    }
#pragma unroll
                    for (int x0 = 0; x0 < kT; x0 += 4) {
                        if (x0 + 4 < kT) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) nx[k] = E[sw(y, x0 + 4 + k)];
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            run += cr[k];
                            E[sw(y, x0 + k)] = run;
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k) cr[k] = nx[k];
                    }
                } else if (tid < kScanThreads + 2 * kT) {
                    // ---- meanwhile spare warps fetch this bucket's texel phases
                    const int h = tid - kScanThreads;
                    S.ph[h] = p.phase[(size_t)D.bucket * p.phase_len + (h < kT ? B.ty0 + h : B.tx0 + (h - kT))];
                } else if (warp >= kBuildWarp0 && D.build) {   // ---- and the builders prepare the next batch
                    build_batch(S, D.batch ^ 1, !B.last, items, n_items, pdevs, sps, queue, tid - 32 * kBuildWarp0);
                }
                __syncthreads();
                if (tid < kScanThreads) {
                    // ---- prefix along y: one column of one plane per thread.
                    // Only the first row of each contraction segment gets its
                    // prefix sum; the contraction adds the segment's other
                    // rows to it in registers
                    static_assert(kSegRows == 4, "one stored row per 4-row segment");
                    uint32_t* E = S.E[tid / kT];
                    const int x = tid % kT;
                    uint32_t cr[4], nx[4], run = 0u;
#pragma unroll
                    for (int k = 0; k < 4; ++k) cr[k] = E[sw(k, x)];
#pragma unroll
                    for (int y0 = 0; y0 < kT; y0 += 4) {
                        if (y0 + 4 < kT) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) nx[k] = E[sw(y0 + 4 + k, x)];
                        }
                        run += cr[0];
                        E[sw(y0, x)] = run;
                        run += cr[1] + cr[2] + cr[3];
#pragma unroll
                        for (int k = 0; k < 4; ++k) cr[k] = nx[k];
                    }
                } else if (tid == kDescThread) {   // ---- meanwhile one thread describes the next pass
                    atomicAdd(p.stats + 5 + p.nb, (unsigned long long)(D.c1 - D.c0));
                    if (D.last)
                        describe_first(S, S.pass[dp ^ 1], D.batch ^ 1, D.f_batch != D.batch, n_items);
                    else
                        describe(S, S.pass[dp ^ 1], D.batch, next_pass(B, Pass{D.s, D.c0, D.c1}), true, D.built, n_items);
                }
                __syncthreads();
                // ---- this thread's texels contracted; each element of E is
                // zeroed once read (the next pass starts from a cleared array).
                // Row r > 0 of the segment: the prefix sum of row r - 1 plus
                // the x prefix of row r (exact modulo 2^32)
                const float2 ux = S.ph[kT + cx];   // (cos a_X, sin a_X) of this column
                const float inv = D.inv;
                const float kh = 0.25f * inv, kd = 0.5f * sp.lam_half * inv;      // (lam / 4)
                uint32_t sy[kPlanes];
#pragma unroll
                for (int r = 0; r < kSegRows; ++r) {
                    const int y = sg * kSegRows + r;
                    const int o = sw(y, cx);
                    float f[kPlanes];
#pragma unroll
                    for (int k = 0; k < kPlanes; ++k) {
                        const uint32_t e = S.E[k][o];
                        sy[k] = r == 0 ? e : sy[k] + e;
                        f[k] = (float)(int32_t)sy[k];
                        S.E[k][o] = 0u;
                    }
                    const float2 vy = S.ph[y];   // (cos a_Y, sin a_Y)
                    float tt[3], tp[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        tt[i] = fmaf(-vy.y, f[3 * i + 2], fmaf(vy.x, f[3 * i + 1], f[3 * i]));   // v . S_i.
                        tp[i] = fmaf(vy.y, f[3 * i + 1], vy.x * f[3 * i + 2]);                 // v' . S_i.
                    }
                    ah[r] = fmaf(kh, fmaf(-ux.y, tt[2], fmaf(ux.x, tt[1], tt[0])), ah[r]);
                    adx[r] = fmaf(kd, fmaf(ux.y, tt[1], ux.x * tt[2]), adx[r]);
                    ady[r] = fmaf(kd, fmaf(-ux.y, tp[2], fmaf(ux.x, tp[1], tp[0])), ady[r]);
                }
                __syncthreads();   // E cleared; the phases may be rewritten
            }
        }

        // ---- the item done: its partial plane, or (one plane) the blended maps
        const int x = B.tx0 + cx;
        const bool done = D.last && B.last;
        if (done && x < sp.W) {
            const bool part_plane = B.planes > 1;
            const int pitch = part_plane ? partial_pitch(sp.W) : sp.W;
            const size_t plane = (size_t)pitch * sp.H;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                float* const dst = (part_plane ? p.partial + ((size_t)B.plane * 3 + f) * plane : p.out + (size_t)f * plane) + x;
#pragma unroll
                for (int r = 0; r < kSegRows; ++r) {
                    const int y = B.ty0 + sg * kSegRows + r;
                    const float v = f == 0 ? ah[r] : (f == 1 ? adx[r] : ady[r]);
                    if (y < sp.H) dst[(size_t)y * pitch] = part_plane ? v : blend1(sp, x, y, f, v);
                }
            }
        }
        if (done) {
#pragma unroll
            for (int r = 0; r < kSegRows; ++r) ah[r] = adx[r] = ady[r] = 0.f;
        }
        dp ^= 1;
    }
    // the last CTA out resets the queue for the next launch: every CTA takes
    // its last ticket before it counts itself out
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(queue + 1, 1u) == gridDim.x - 1) {
            queue[0] = 0u;
            queue[1] = 0u;
            __threadfence();
        }
    }
}

cudaError_t sat_attributes() {
    static int attr[kMaxCachedDevices] = {};
    return cached_per_device(attr, [] {
               return cudaFuncSetAttribute(k_synth_sat, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sizeof(SatSmem)) == cudaSuccess ? 1 : -1;
           }) > 0
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

}  // namespace

int synth_sat_tile() { return kT; }

// resident CTAs per SM from the SM's limits (shared memory, registers, threads)
static int synth_sat_ctas_per_sm_query();
int synth_sat_ctas_per_sm() {
    static int cache[kMaxCachedDevices] = {};
    return max(0, cached_per_device(cache, [] { return max(-1, synth_sat_ctas_per_sm_query()); }));
}
static int synth_sat_ctas_per_sm_query() {
    if (sat_attributes() != cudaSuccess) return 0;
    int dev = 0, smem_sm = 0, resv = 0, regs_sm = 0, thr_sm = 0;
    cudaFuncAttributes a;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncGetAttributes(&a, k_synth_sat) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess)
        return 0;
    const int warps = kSatThreads / 32;
    const int regs_warp = ((a.numRegs * 32 + 255) / 256) * 256;
    int n = smem_sm / (int)(sizeof(SatSmem) + a.sharedSizeBytes + resv);
    n = min(n, regs_sm / (regs_warp * warps));
    n = min(n, thr_sm / kSatThreads);
    return n;
}

cudaError_t launch_synth_sat(const TcItem* items, int n_items, const PatchDev* pdevs, const SynthParams* sps,
                             const BlendSpan* spans, int n_spans, unsigned int* queue, cudaStream_t st) {
    cudaError_t e = sat_attributes();
    if (e != cudaSuccess) return e;
    if (n_items > 0) {
        // persistent grid: one CTA per resident slot, no more than the items
        static int slots[kMaxCachedDevices] = {};
        const int n_slots = cached_per_device(slots, [] {
            int dev = 0, sms = 0;
            if (cudaGetDevice(&dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return 152;
            return sms * max(1, synth_sat_ctas_per_sm());
        });
        const int grid = min(n_items, n_slots);
        e = launch_pdl(k_synth_sat, grid, kSatThreads, sizeof(SatSmem), st, items, n_items, pdevs, sps, queue);
        count_launches(1);
        if (e != cudaSuccess) return e;
    }
    if (n_spans > 0) return launch_blend_spans(spans, n_spans, pdevs, sps, st);
    return cudaGetLastError();
}

}  // namespace scwp
