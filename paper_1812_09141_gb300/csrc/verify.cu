// Verification kernels for sm_103a.
//
// What is computed (Section 3.1 and Table "Similarity Functions"): for every
// listed candidate pair (r, s), the overlap o = |r n s| of the two sorted
// token sets by merging, stopping early once o + min(|r|-i, |s|-j) falls
// below the required overlap (positional filter, Section 2.2.3), and the
// pair is kept iff o*(p+q) >= p*(|r|+|s|) (Jaccard t = p/q).
//
// How the work is laid out (the paper's Alternatives A-C of Section 3.3.2,
// re-designed for one GB300):
//   * plan_kernel (plan.cu): validates the grouped candidate list, drops
//     the pairs that their sets' signatures prove dissimilar and bins the
//     others by their probe's |r|+|s| (estimated as 2|r|; the length filter
//     keeps |s| within [t|r|, |r|/t]): pairs of short probes go to the front
//     of one pair list, the others to its back, where a probe with several
//     pairs left may become lane, block or index work items.
//   * verify_kernel, persistent (one wave of CTAs over the SMs):
//       phase 1 - block items: one CTA per pair, Intersect Path across the
//                 whole CTA (Alternative C, Sections 4.2.2-4.2.3), r kept in
//                 shared memory for the item's candidates; and index items:
//                 the CTA holds r as a bitmap over the token values (one bit
//                 per value, in shared memory) and every thread walks one
//                 candidate s at a time through the merge, s side by s side:
//                 each token of s is tested against r by one bit lookup, so
//                 r's tokens are read once per item instead of once per
//                 pair (Alternative B with the probe in shared memory,
//                 Section 3.3.2; the s-side positional bound of Section
//                 2.2.3 after every 16-byte block);
//       phase 2 - lane items: one candidate per lane, r in the warp's shared
//                 memory; and long pairs, or all pairs when they are few
//                 (few_pairs): one warp per pair, s's tokens looked up in r,
//                 which stays in the warp's shared memory while the next pair
//                 has the same probe (longer probes, and a forced warp
//                 granularity: 32-lane merge path in windows);
//       phase 3 - short pairs, one pair per thread (Alternatives A/B).
//                 The merge compares 16-byte blocks (4 tokens of r against
//                 4 of s, 16 compares; the block with the smaller last token
//                 advances).  Pairs wait with their merge state in a per-warp
//                 shared buffer and are merged 32 at a time; a warp with too
//                 few lanes still merging parks them again and refills.
//     Heavy work goes first so that short pairs fill the tail.  The first
//     unit of each phase is assigned statically (CTA / warp index), later
//     ones through one atomic per unit, so small batches need no atomics.
//   The cooperative merges run in windows of G*D merge steps; the
//   positional bound is tested between windows, and a pair that is not
//   rejected runs to the end of the merge so its overlap is exact.
//   Survivors are compacted into (r, s, o) triples with warp-aggregated
//   atomics on one global cursor (output select, Section 3.3.2), or only
//   counted (output count).
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

#include "arith.h"
#include "checked.cuh"
#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kWarpD = 8;                          // merge steps per lane per window (warp)
constexpr uint32_t kWarpWin = 32 * kWarpD;         // merge steps per window (warp)
constexpr uint32_t kWarpABuf = kWarpRCap + 16;     // r buffer (whole r, or one window of it)
constexpr uint32_t kWarpBBuf = kWarpWin + 16;      // s window buffer
constexpr int kBlockD = 8;                         // merge steps per thread per window (block)
constexpr uint32_t kBlockRCap = 4096;              // r kept whole in shared memory up to this
constexpr uint32_t kFlatGrab = 4;                  // most 32-pair chunks taken per dynamic grab in phase 3
constexpr uint32_t kLongGrab = 8;                  // long pairs taken per dynamic grab in phase 2, about,
constexpr uint32_t kLongScan = 256;                // and entries of their list read for them, at most
constexpr uint32_t kCont = 64;                     // parked pairs per warp in phase 3

// Checked build (SSJ_CHECKED): the functions that are not inlined take the
// token arrays' remaining extents and the error word as extra arguments;
// the product build passes nothing and the checks compile away.
#ifdef SSJ_CHECKED
#define CHK_PARAMS , uint64_t chk_rlim, uint64_t chk_slim, uint32_t* chk_err
#define CHK_ARGS(rl, sl, e) , (rl), (sl), (e)
#define CHK_ERR_PARAM , uint32_t* chk_err
#define CHK_ERR_ARG(e) , (e)
#define CHK_RLIM chk_rlim
#define CHK_SLIM chk_slim
#define CHK_ERR chk_err
#else
#define CHK_PARAMS
#define CHK_ARGS(rl, sl, e)
#define CHK_ERR_PARAM
#define CHK_ERR_ARG(e)
#define CHK_RLIM (~0ull)
#define CHK_SLIM (~0ull)
#define CHK_ERR (static_cast<uint32_t*>(nullptr))
#endif

// Block idx of a token array with lim blocks from base on (the checked
// build reads zeros past the end).
__device__ __forceinline__ uint4 ld_block(const uint4* base, uint64_t idx, uint64_t lim, uint32_t* err) {
    if (!in_bounds(idx, lim, err)) return make_uint4(0u, 0u, 0u, 0u);
    return __ldg(base + idx);
}

// ---------------------------------------------------------------------------
// One-dimensional bulk copies global -> shared memory (cp.async.bulk on the
// copy engine, completion counted in bytes on an mbarrier), used to stage
// the probe set and candidate sets of block and warp items.  Addresses and
// sizes are multiples of 16 bytes (sets start on 16-byte chunks).  Waits are
// bounded: one thread polls the barrier for at most about a second of SM
// clocks and reports a timeout (ERR_GUARD) instead of spinning forever.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The calling thread arrives on bar expecting `bytes` more bytes, then asks
// the copy engine for `bytes` bytes from src to dst (previous generic-proxy
// accesses of dst are ordered before the copy by the proxy fence).
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// Poll bar until the phase with the given parity has completed; false (and
// ERR_GUARD) if that takes more than about a second.
constexpr long long kBulkWaitCycles = 2000000000ll;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t* err) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t done = 0;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > kBulkWaitCycles) {
            atomicOr(err, ERR_GUARD);
            return false;
        }
        __nanosleep(20);
    }
}

// Chunks [c_lo, c_hi) of a token array (16 bytes each) into dst by one bulk
// copy on bar; the checked build tests both ends against the array's and
// the buffer's extents and skips the copy (arriving without bytes) when one
// is out of range.
__device__ __forceinline__ void bulk_stage(uint32_t* dst, const uint4* set4, uint32_t c_lo, uint32_t c_hi, uint64_t lim,
                                           uint32_t dst_blocks, uint64_t* bar, uint32_t* err) {
    const uint32_t n = c_hi - c_lo;
    if (n == 0 || !in_bounds(c_hi - 1, lim, err) || !in_bounds(n - 1, dst_blocks, err)) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
        return;
    }
    bulk_copy(dst, set4 + c_lo, 16u * n, bar);
}

// A parked pair with its merge state.
struct ContEntry {
    uint4 m0;  // r id, s id, current 16-byte block of r, of s (token array indices)
    uint4 m1;  // tokens of r and of s from the current blocks on, required overlap, overlap so far
    uint4 m2;  // instance, unused, unused, unused
};
constexpr uint32_t kDrainMinLive = 16;             // default: pass 2 re-parks a warp's pairs below this many live lanes
constexpr uint32_t kTableBytes = kCont * sizeof(ContEntry);

// Phases 2 and 3 run per warp and the warps of a CTA change phase at
// different times, so each warp owns one fixed slice of shared memory that
// both phases use (phase 1 uses the whole CTA's memory and ends with a
// CTA barrier before any warp moves on).
constexpr uint32_t kWarpPhase2Bytes = (kWarpABuf + kWarpBBuf) * 4;
constexpr uint32_t kWarpSliceBytes =
    ((kWarpPhase2Bytes > kTableBytes ? kWarpPhase2Bytes : kTableBytes) + 15u) & ~15u;

// 1 if x equals one of the four tokens of s (distinct within a block).
__device__ __forceinline__ uint32_t match4(uint32_t x, const uint4& s) {
    return (x == s.x) | (x == s.y) | (x == s.z) | (x == s.w);
}

// Merge state of one pair compared block by block.
struct BlockState {
    uint32_t qi, qj, o;  // current block of r and of s, overlap so far
    bool fin, rej;
};

// Matches between the valid tokens of an r block and an s block whose
// padding repeats the set's last token (the collection layout): a repeated
// s token changes no membership test, and the r lanes past nvr valid ones
// all repeat the last valid token, whose match is subtracted again.
__device__ __forceinline__ uint32_t block_matches(const uint4& rc, const uint4& sc, uint32_t nvr) {
    const uint32_t mw = match4(rc.w, sc);
    return match4(rc.x, sc) + match4(rc.y, sc) + match4(rc.z, sc) + mw - (4u - nvr) * mw;
}

// One block step: count the matches between block qi of r (rc) and block qj
// of s (sc), then advance the block whose last valid token is smaller (both
// on a tie).  Every matching pair of tokens sits in a pair of blocks that is
// current together exactly once, so the count is exact.  Before the step the
// positional bound o + min(|r| - 4qi, |s| - 4qj) < req rejects the pair; the
// bound counts whole current blocks, so it only over-estimates the reachable
// overlap and never rejects a passing pair.  A block's last lane holds its
// last valid token (the padding repeats it).  The step is predicated code:
// the lanes of a warp are at different points of different pairs, so a lane
// whose pair is decided computes and discards instead of branching away.
__device__ __forceinline__ void block_step(const uint4& rc, const uint4& sc, uint32_t nr, uint32_t ns, uint32_t req,
                                           bool early, BlockState& st, bool& adv_r, bool& adv_s) {
    const uint32_t remr = nr - 4 * st.qi, rems = ns - 4 * st.qj;
    const bool bad = !st.fin && early && st.o + min(remr, rems) < req;
    const bool go = !st.fin && !bad;
    st.rej = st.rej || bad;
    const uint32_t c = block_matches(rc, sc, min(remr, 4u));
    st.o += go ? c : 0u;
    adv_r = go && rc.w <= sc.w;
    adv_s = go && sc.w <= rc.w;
    st.qi += adv_r ? 1u : 0u;
    st.qj += adv_s ? 1u : 0u;
    st.fin = st.fin || bad || 4 * st.qi >= nr || 4 * st.qj >= ns;
}

// Equivalent overlap of the instance's similarity function with t = p/q
// (Table "Similarity Functions"; exact, see arith.h): Jaccard and Dice
// divide p(|r|+|s|) by den = p+q or 2q with the precomputed reciprocal,
// Cosine takes the exact ceil(t sqrt(|r||s|)) (den = q), the plain overlap
// threshold is den itself.
__device__ __forceinline__ uint32_t required_overlap(uint32_t sim, uint32_t p, uint32_t den, uint64_t magic,
                                                     uint32_t nr, uint32_t ns) {
    if (sim == SIM_COSINE) return required_overlap_cosine(p, den, nr, ns);
    if (sim == SIM_OVERLAP) return den;
    return required_overlap_magic(nr, ns, p, den, magic);
}

// Write result idx of an instance (if it fits its capacity), as (min, max)
// ids for a self-join.
__device__ __forceinline__ void emit_triple(ssj_triple* out, uint64_t cap, bool self_join, unsigned long long idx,
                                            uint32_t r, uint32_t s, uint32_t o) {
    if (idx < cap) {
        uint32_t x = r, y = s;
        if (self_join && y < x) { x = s; y = r; }
        ssj_triple* t = out + idx;
        t->r = x;
        t->s = y;
        t->overlap = o;
    }
}

// Copy the 16-byte chunks covering tokens [x0, x0+n) of a set into dst
// (16-byte aligned): dst[k] holds token (x0 & ~3) + k.
// (lim: blocks of the token array from set4 on; dst_blocks: room at dst;
// both checked in the checked build only.)
template <int G>
__device__ __forceinline__ void stage(const uint4* __restrict__ set4, uint32_t x0, uint32_t n, uint32_t* dst,
                                      int lane, uint64_t lim, uint32_t dst_blocks, uint32_t* err) {
    const uint32_t c_lo = x0 >> 2, c_hi = (x0 + n + 3) >> 2;
    uint4* d4 = reinterpret_cast<uint4*>(dst);
    for (uint32_t c = c_lo + lane; c < c_hi; c += G)
        if (in_bounds(c - c_lo, dst_blocks, err)) d4[c - c_lo] = ld_block(set4, c, lim, err);
}

// One lane's share of a window: binary search of its cross diagonal
// (merge path with "take r when r[i] <= s[j]"), then up to D merge steps.
// A match is counted by the step that takes r[i] while r[i] == s[j], so
// every match is counted exactly once across lanes (Section 4.2.3 with the
// tie rule fixed).  A, B: window-local views; rw, sw: their valid lengths.
template <int D>
__device__ __forceinline__ void lane_merge(const uint32_t* A, uint32_t rw, const uint32_t* B, uint32_t sw,
                                           uint32_t d, uint32_t de, uint32_t* c_out, uint32_t* i_out,
                                           uint32_t* j_out) {
    uint32_t lo = d > sw ? d - sw : 0u;
    uint32_t hi = min(d, rw);
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (A[mid] <= B[d - 1 - mid]) lo = mid + 1; else hi = mid;
    }
    uint32_t i = lo, j = d - lo, c = 0;
#pragma unroll
    for (int t = 0; t < D; ++t) {
        if (d + (uint32_t)t < de) {
            bool ta;
            if (i >= rw) {
                ta = false;
            } else if (j >= sw) {
                ta = true;
            } else {
                const uint32_t x = A[i], y = B[j];
                ta = x <= y;
                c += (x == y) ? 1u : 0u;
            }
            i += ta ? 1u : 0u;
            j += ta ? 0u : 1u;
        }
    }
    *c_out = c;
    *i_out = i;
    *j_out = j;
}

// -------------------------------------------------------------------------
// Overlap of one pair by a warp, r whole in its shared memory (R): the lanes
// read s's blocks side by side and look each token up in r by binary search,
// a block's four tokens in step.  One memory wait and about log2|r| waits on
// shared memory per 128 tokens of s; a merge in windows waits for both in each
// window, which costs the pairs that the signature test leaves more than its
// early termination saves them (they mostly pass).
// -------------------------------------------------------------------------
__device__ __forceinline__ uint32_t warp_lookup(const uint32_t* R, uint32_t nr, const uint4* __restrict__ s4,
                                                uint32_t ns, int lane, uint64_t slim, uint32_t* err) {
    uint32_t c = 0;
    auto r_at = [&](uint32_t p) -> uint32_t { return in_bounds(p, nr, err) ? R[p] : 0u; };
    if (nr) {
        for (uint32_t b = lane; b < (ns + 3) >> 2; b += 32) {
            const uint4 x = ld_block(s4, b, slim, err);
            uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;  // first token of r not below x's, among the last n
            for (uint32_t n = nr; n > 1;) {
                const uint32_t half = n >> 1;
                p0 += r_at(p0 + half - 1) < x.x ? half : 0u;
                p1 += r_at(p1 + half - 1) < x.y ? half : 0u;
                p2 += r_at(p2 + half - 1) < x.z ? half : 0u;
                p3 += r_at(p3 + half - 1) < x.w ? half : 0u;
                n -= half;
            }
            const uint32_t valid = ns - 4 * b;  // (the tokens past s's end repeat its last one)
            c += (r_at(p0) == x.x ? 1u : 0u) + (valid > 1 && r_at(p1) == x.y ? 1u : 0u) +
                 (valid > 2 && r_at(p2) == x.z ? 1u : 0u) + (valid > 3 && r_at(p3) == x.w ? 1u : 0u);
        }
    }
    return __reduce_add_sync(kFull, c);
}

// -------------------------------------------------------------------------
// Warp-cooperative merge of one pair (all 32 lanes, uniform arguments).
// If r_staged, abuf holds all of r (abuf[k] = r[k]); otherwise abuf is a
// window buffer.  bbuf is the s window buffer, filled per window by the
// lanes' 16-byte loads or, with wbar (bulk staging), by one bulk copy on the
// warp's barrier (phase parity *wph); a copy that does not complete sets
// *failed and ends the merge.
// -------------------------------------------------------------------------
__device__ uint32_t warp_merge(const uint4* __restrict__ r4, uint32_t nr, const uint4* __restrict__ s4, uint32_t ns,
                               uint32_t req, bool early, bool r_staged, uint32_t* abuf, uint32_t* bbuf, int lane,
                               uint64_t* wbar, uint32_t* wph, uint64_t slim, uint32_t* err, bool* failed,
                               bool* rejected CHK_PARAMS) {
    uint32_t i0 = 0, j0 = 0, o = 0;
    *rejected = false;
    *failed = false;
    for (;;) {
        const uint32_t left = min(nr - i0, ns - j0);
        if (early && o + left < req) { *rejected = true; break; }
        if (left == 0) break;
        const uint32_t rem = (nr - i0) + (ns - j0);
        const uint32_t Wc = min(kWarpWin, rem);
        const uint32_t rw = min(nr - i0, Wc), sw = min(ns - j0, Wc);
        const uint32_t* A;
        if (r_staged) {
            A = abuf + i0;
        } else {
            stage<32>(r4, i0, rw, abuf, lane, CHK_RLIM, kWarpABuf / 4, CHK_ERR);
            A = abuf + (i0 & 3u);
        }
        if (wbar) {  // bulk staging: the window of s by one bulk copy, lane 0 waits
            uint32_t ok = 1;
            if (lane == 0) {
                bulk_stage(bbuf, s4, j0 >> 2, (j0 + sw + 3) >> 2, slim, kWarpBBuf / 4, wbar, err);
                ok = mbar_wait(wbar, *wph, err) ? 1u : 0u;
            }
            *wph ^= 1u;
            if (!__shfl_sync(kFull, ok, 0)) {
                *failed = true;
                break;
            }
        } else {
            stage<32>(s4, j0, sw, bbuf, lane, CHK_SLIM, kWarpBBuf / 4, CHK_ERR);
        }
        __syncwarp();
        const uint32_t* B = bbuf + (j0 & 3u);
        const uint32_t d = min((uint32_t)lane * kWarpD, Wc), de = min(d + kWarpD, Wc);
        uint32_t c = 0, ie = 0, je = 0;
        if (d < de) lane_merge<kWarpD>(A, rw, B, sw, d, de, &c, &ie, &je);
        const uint32_t total = __reduce_add_sync(kFull, c);
        const int last = (int)((Wc - 1) / kWarpD);
        ie = __shfl_sync(kFull, ie, last);
        je = __shfl_sync(kFull, je, last);
        __syncwarp();
        i0 += ie;
        j0 += je;
        o += total;
    }
    return o;
}

// -------------------------------------------------------------------------
// Block-cooperative merge of one pair (Alternative C).  r is staged whole in
// rbuf when it fits (r_staged), else per window in wbuf_r; s is staged whole
// in wbuf_s by the caller (s_staged: bulk staging) or per window.
// -------------------------------------------------------------------------
template <int BT>
struct BlockSmem {
    uint64_t bar[3];  // bulk staging: r, and the two candidate buffers
    uint32_t red[BT / 32];
    uint32_t end_i, end_j;
    uint32_t item;
    uint32_t next;       // index items: next candidate of the item
    uint32_t staged[2];  // bulk staging: candidate buffer b holds the whole set s of its candidate
    uint32_t ok;         // bulk staging: the last wait completed
};

template <int BT>
__device__ uint32_t block_merge(const uint4* __restrict__ r4, uint32_t nr, const uint4* __restrict__ s4,
                                uint32_t ns, uint32_t req, bool early, const uint32_t* rbuf, bool r_staged,
                                uint32_t* wbuf_r, uint32_t* wbuf_s, bool s_staged, BlockSmem<BT>* sm,
                                bool* rejected CHK_PARAMS) {
    constexpr uint32_t W = BT * kBlockD;
    const int tid = threadIdx.x;
    uint32_t i0 = 0, j0 = 0, o = 0;
    bool rej = false;
    for (;;) {
        const uint32_t left = min(nr - i0, ns - j0);
        if (early && o + left < req) { rej = true; break; }
        if (left == 0) break;
        const uint32_t rem = (nr - i0) + (ns - j0);
        const uint32_t Wc = min(W, rem);
        const uint32_t rw = min(nr - i0, Wc), sw = min(ns - j0, Wc);
        const uint32_t* A;
        if (r_staged) {
            A = rbuf + i0;
        } else {
            stage<BT>(r4, i0, rw, wbuf_r, tid, CHK_RLIM, (W + 16) / 4, CHK_ERR);
            A = wbuf_r + (i0 & 3u);
        }
        const uint32_t* B;
        if (s_staged) {  // all of s is in wbuf_s already (bulk copy)
            B = wbuf_s + j0;
        } else {
            stage<BT>(s4, j0, sw, wbuf_s, tid, CHK_SLIM, (W + 16) / 4, CHK_ERR);
            B = wbuf_s + (j0 & 3u);
        }
        __syncthreads();
        const uint32_t d = min((uint32_t)tid * kBlockD, Wc), de = min(d + kBlockD, Wc);
        uint32_t c = 0, ie = 0, je = 0;
        if (d < de) lane_merge<kBlockD>(A, rw, B, sw, d, de, &c, &ie, &je);
        c = __reduce_add_sync(kFull, c);
        if ((tid & 31) == 0) sm->red[tid >> 5] = c;
        if (d < de && de == Wc) { sm->end_i = ie; sm->end_j = je; }
        __syncthreads();
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < BT / 32; ++w) total += sm->red[w];
        i0 += sm->end_i;
        j0 += sm->end_j;
        o += total;
        __syncthreads();  // everyone has read red/end_* and the window buffers
    }
    *rejected = rej;
    return o;
}

// Block step of the short-pair phase on a (block cursor, tokens remaining) state; the same
// step as block_step: positional bound, 16 compares between the current
// blocks, then the block with the smaller last valid token advances (both on
// a tie), predicated like block_step.  rn / sn hold the next block of each
// side, loaded one step ahead.
__device__ __forceinline__ void lean_step(uint4& rc, uint4& rn, uint4& sc, uint4& sn, const uint4* rb,
                                          const uint4* sb, uint32_t& rcur, uint32_t& scur, uint32_t& remr,
                                          uint32_t& rems, uint32_t& o, uint32_t req, bool early, bool& fin,
                                          bool& rej, uint64_t rlim, uint64_t slim, uint32_t* err) {
    const bool bad = !fin && early && o + min(remr, rems) < req;
    const bool go = !fin && !bad;
    rej = rej || bad;
    const uint32_t c = block_matches(rc, sc, min(remr, 4u));
    o += go ? c : 0u;
    const bool ar = go && rc.w <= sc.w, as = go && sc.w <= rc.w;
    rc.x = ar ? rn.x : rc.x;
    rc.y = ar ? rn.y : rc.y;
    rc.z = ar ? rn.z : rc.z;
    rc.w = ar ? rn.w : rc.w;
    sc.x = as ? sn.x : sc.x;
    sc.y = as ? sn.y : sc.y;
    sc.z = as ? sn.z : sc.z;
    sc.w = as ? sn.w : sc.w;
    rcur += ar ? 1u : 0u;
    scur += as ? 1u : 0u;
    remr = ar ? (remr > 4 ? remr - 4 : 0u) : remr;
    rems = as ? (rems > 4 ? rems - 4 : 0u) : rems;
    if (ar && remr > 4) rn = ld_block(rb, rcur + 1, rlim, err);
    if (as && rems > 4) sn = ld_block(sb, scur + 1, slim, err);
    fin = fin || bad || remr == 0 || rems == 0;
}

// One step of the short-pair phase: the parked pairs [n_cont - m, n_cont) are
// taken one per lane (lanes may belong to different instances) and merged
// while at least min_live lanes are still undecided; decided pairs are
// emitted, undecided ones parked again, compacted, so that lanes are refilled
// from later pairs instead of idling behind the longest merge of the warp.
// min_live = 1 finishes every pair.  Returns the new number of parked pairs.
__device__ __noinline__ uint32_t drain_parked(ContEntry* cont, uint32_t n_cont, uint32_t m, uint32_t min_live,
                                              const Instance* table, int lane CHK_ERR_PARAM) {
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    const uint32_t base = n_cont - m;
    const bool have = (uint32_t)lane < m && in_bounds(base + lane, kCont, CHK_ERR);
    uint32_t rid = 0, sid = 0, rcur = 0, scur = 0, remr = 0, rems = 0, req = 0, o = 0, inst = 0;
    const uint4* rb = nullptr;
    const uint4* sb = nullptr;
    uint64_t rlim = 0, slim = 0;
    bool early = true, fin = true, rej = false;
    uint4 rc = zero4, rn = zero4, sc = zero4, sn = zero4;
    if (have) {
        const ContEntry* ce = cont + base + lane;
        const uint4 m0 = ce->m0, m1 = ce->m1, m2 = ce->m2;
        rid = m0.x;
        sid = m0.y;
        rcur = m0.z;
        scur = m0.w;
        remr = m1.x;
        rems = m1.y;
        req = m1.z;
        o = m1.w;
        inst = m2.x;
        const Instance& I = table[inst];
        rb = I.r_toks4;
        sb = I.s_toks4;
        rlim = I.r_n_chunks;
        slim = I.s_n_chunks;
        early = !(I.flags & VF_EMIT_ALL);
        fin = remr == 0 || rems == 0;
        if (remr > 0) rc = ld_block(rb, rcur, rlim, CHK_ERR);
        if (remr > 4) rn = ld_block(rb, rcur + 1, rlim, CHK_ERR);
        if (rems > 0) sc = ld_block(sb, scur, slim, CHK_ERR);
        if (rems > 4) sn = ld_block(sb, scur + 1, slim, CHK_ERR);
    }
    __syncwarp();  // every entry is read before any is written again
    while ((uint32_t)__popc(__ballot_sync(kFull, !fin)) >= min_live) {  // two steps per check
        if (!fin) lean_step(rc, rn, sc, sn, rb, sb, rcur, scur, remr, rems, o, req, early, fin, rej, rlim, slim, CHK_ERR);
        if (!fin) lean_step(rc, rn, sc, sn, rb, sb, rcur, scur, remr, rems, o, req, early, fin, rej, rlim, slim, CHK_ERR);
    }
    // survivors: one atomic per instance among the warp's lanes (lanes may hold different instances)
    const bool pass = have && fin && (!early || (!rej && o >= req));
    const uint32_t pmask = __ballot_sync(kFull, pass);
    if (pmask) {
        const uint32_t grp = __match_any_sync(kFull, inst) & pmask;  // passing lanes of my instance
        if (pass) {
            const Instance& I = table[inst];
            const int leader = __ffs(grp) - 1;
            unsigned long long b0 = 0;
            if (lane == leader) b0 = atomicAdd(I.count, (unsigned long long)__popc(grp));
            b0 = __shfl_sync(grp, b0, leader);
            if (!(I.flags & VF_COUNT_ONLY))
                emit_triple(I.out, I.cap, (I.flags & VF_SELF_JOIN) != 0, b0 + __popc(grp & lt_mask), rid, sid, o);
        }
    }
    const bool again = have && !fin;
    const uint32_t amask = __ballot_sync(kFull, again);
    if (again) {
        ContEntry* ce = cont + base + __popc(amask & lt_mask);
        ce->m0 = make_uint4(rid, sid, rcur, scur);
        ce->m1 = make_uint4(remr, rems, req, o);
        ce->m2 = make_uint4(inst, 0u, 0u, 0u);
    }
    __syncwarp();
    return base + __popc(amask);
}

// Warp-local survivor buffer for pairs decided by the whole warp (one work
// item, so one instance): lane k holds the k-th buffered triple; flushed
// with one atomic per 32 and at the end of every item.
struct WarpOut {
    uint32_t r = 0, s = 0, o = 0, n = 0;

    __device__ void push(const Instance& I, int lane, uint32_t pr, uint32_t ps, uint32_t po) {
        if (lane == (int)n) { r = pr; s = ps; o = po; }
        if (++n == 32) flush(I, lane);
    }
    __device__ void flush(const Instance& I, int lane) {
        if (n == 0) return;
        unsigned long long b0 = 0;
        if (lane == 0) b0 = atomicAdd(I.count, (unsigned long long)n);
        b0 = __shfl_sync(kFull, b0, 0);
        if ((uint32_t)lane < n) emit_triple(I.out, I.cap, (I.flags & VF_SELF_JOIN) != 0, b0 + lane, r, s, o);
        n = 0;
    }
};

// One lane item (Alternative B): the item's probe r is staged whole in the
// warp's shared memory (rsm, 16-byte blocks), each lane verifies one of the
// item's pairs (run) at a time with the block merge, reading r's blocks from
// shared memory and s's from global memory one block ahead; a lane that
// finishes takes the item's next candidate.  Survivors are emitted with one
// atomic per warp step.
__device__ __noinline__ void lane_item(const Instance& I, const WorkItem& wi, const PairRef* run, uint32_t nr,
                                       const uint4* rsm, int lane, uint32_t* err) {
    const uint32_t flags = I.flags;
    const bool emit_all = (flags & VF_EMIT_ALL) != 0, early = !emit_all;
    const bool self_join = (flags & VF_SELF_JOIN) != 0;
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t rq = (nr + 3) >> 2;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    uint32_t cursor = 0;  // next candidate of the item (warp-uniform)
    bool active = false;
    uint32_t s_id = 0, ns = 0, req = 0, sq = 0;
    const uint4* s4 = nullptr;
    uint64_t slim = 0;
    BlockState st;
    st.qi = st.qj = st.o = 0;
    st.fin = true;
    st.rej = false;
    uint4 rc = zero4, sc = zero4, sn = zero4;
    for (;;) {
        const uint32_t idle = __ballot_sync(kFull, !active);
        if (idle && cursor < wi.n) {
            const uint32_t my = cursor + __popc(idle & lt_mask);
            if (!active && my < wi.n) {
                const uint32_t s = run[my].s & ~kInItem;
                const uint2 ds = ld_at(I.s_desc, s, I.s_n_sets, err);
                active = true;
                s_id = s;
                ns = ds.y;
                req = required_overlap(I.sim, I.p, I.den, I.magic, nr, ns);
                sq = (ns + 3) >> 2;
                s4 = I.s_toks4 + ds.x;
                slim = I.s_n_chunks - ds.x;
                st.qi = st.qj = st.o = 0;
                st.rej = false;
                st.fin = nr == 0 || ns == 0;
                rc = rq ? rsm[0] : zero4;
                sc = sq ? ld_block(s4, 0, slim, err) : zero4;
                sn = sq > 1 ? ld_block(s4, 1, slim, err) : zero4;
            }
            cursor += __popc(idle);
        }
        if (!__any_sync(kFull, active)) {
            if (cursor >= wi.n) break;
            continue;
        }
        if (active && !st.fin) {
            bool ar, as;
            block_step(rc, sc, nr, ns, req, early, st, ar, as);
            if (ar && st.qi < rq && in_bounds(st.qi, kWarpABuf / 4, err)) rc = rsm[st.qi];
            if (as) {
                sc = sn;
                if (st.qj + 1 < sq) sn = ld_block(s4, st.qj + 1, slim, err);
            }
        }
        const bool done = active && st.fin;
        const bool pass = done && (emit_all || (!st.rej && st.o >= req));
        const uint32_t pmask = __ballot_sync(kFull, pass);
        if (pmask) {
            unsigned long long b0 = 0;
            if (lane == 0) b0 = atomicAdd(I.count, (unsigned long long)__popc(pmask));
            if (!(flags & VF_COUNT_ONLY)) {
                b0 = __shfl_sync(kFull, b0, 0);
                if (pass) emit_triple(I.out, I.cap, self_join, b0 + __popc(pmask & lt_mask), wi.r, s_id, st.o);
            }
        }
        if (done) active = false;
    }
}

// Set (or, with clear, zero the words of) the bits of r's tokens; r's
// padding repeats its last token, so whole blocks are used.
template <int BT>
__device__ __forceinline__ void bm_mark(uint32_t* bm, const uint4* r4, uint32_t nr, uint64_t rlim, uint32_t n_words,
                                        bool clear, int tid, uint32_t* err) {
    for (uint32_t c = tid; c < ((nr + 3) >> 2); c += BT) {
        const uint4 b = ld_block(r4, c, rlim, err);
        const uint32_t v[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t w = v[k] >> 5;
            if (!in_bounds(w, n_words, err)) continue;
            if (clear) bm[w] = 0u;
            else atomicOr(bm + w, 1u << (v[k] & 31u));
        }
    }
}

// Asynchronous 16-byte copy global -> shared memory (cp.async, cached in L2
// only) and its per-thread groups.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One index item: wi.n queued pairs (run) of probe r, verified by every
// thread of the CTA, one candidate per thread at a time.  r is held as a
// bitmap over the token values (bm, all zero on entry and on return).  A
// candidate s is merged against r from the s side: block by block (16
// bytes, 4 tokens), each token tested by one bit lookup, so the state after
// a block is the merge's state after s's token j: o matches, |s| - j tokens
// of s left.  The merge stops when o + (|s| - j) falls below the required
// overlap (the positional bound of Section 2.2.3 with the s side's
// remainder; never stricter than the merge's bound, so no passing pair is
// lost) or when s's block reaches r's last token (no later token of s can
// match); a pair that is not rejected runs to that point, so its overlap is
// exactly |r n s|.
//
// The walk is software-pipelined so that no thread waits on a load it has
// just issued, and its common path is short.  Each warp prepares its
// candidates 32 at a time: their ids are loaded, one round later their
// descriptors, one round later again they enter the warp's queue (shared
// memory) with their required overlap, and the next batch's ids are loaded
// in that same step.  A round is
// kIndexSteps walk steps followed by one maintenance step (preparation,
// survivors out, idle lanes refilled from the queue).  In a walk step a lane
// asks for one more block of s (cp.async into its own ring of kIndexRing
// blocks in shared memory, at most kIndexRing blocks ahead of its walk) and
// merges a block it asked for in an earlier step.
constexpr uint32_t kIndexRing = 4;   // blocks of s per thread in the ring
constexpr uint32_t kIndexQueue = 64; // prepared candidates per warp
constexpr int kIndexSteps = 4;       // walk steps per round

// Bit of token value x in the probe bitmap, as one shift-and-mask of the
// word (the funnel shift takes the shift amount modulo 32).
__device__ __forceinline__ uint32_t bm_test(const uint32_t* bm, uint32_t x, uint32_t n_words, uint32_t* err) {
    const uint32_t w = x >> 5;
    if (!in_bounds(w, n_words, err)) return 0u;
    const uint32_t word = bm[w];
    return __funnelshift_r(word, word, x) & 1u;
}

template <int BT>
__device__ __noinline__ void index_item(const Instance& I, const WorkItem& wi, const PairRef* run, uint32_t nr,
                                        const uint4* r4, uint64_t rlim, uint32_t* bm, uint32_t n_words, uint4* rings,
                                        uint4* queues, BlockSmem<BT>* sm, uint32_t* err) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t flags = I.flags;
    const bool emit_all = (flags & VF_EMIT_ALL) != 0, early = !emit_all;
    const bool self_join = (flags & VF_SELF_JOIN) != 0;
    uint4* ring = rings + (size_t)tid * kIndexRing;
    uint4* queue = queues + (size_t)warp * kIndexQueue;
    // candidate preparation (warp-uniform stage: 0 takes 32 candidates, 1 loads descriptors,
    // 2 queues); queue cursors are free-running.  Warp w's first batch is
    // candidates [32w, 32w + 32): its ids and descriptors are loaded while r's bits are set,
    // so the walk starts one round after the item does; later batches are taken from the
    // item's cursor, which starts after the first batches.
    uint32_t pstage = 0, qhead = 0, qtail = 0;
    bool pdone = 32u * (BT / 32) >= wi.n;  // warp-uniform: no candidates left to take
    const uint32_t my0 = 32u * (uint32_t)warp + (uint32_t)lane;
    bool p_ok = my0 < wi.n;
    uint32_t p_id = p_ok ? run[my0].s & ~kInItem : 0u;
    uint2 p_desc = make_uint2(0u, 0u);
    if (tid == 0) sm->next = 32u * (BT / 32);
    bm_mark<BT>(bm, r4, nr, rlim, n_words, false, tid, err);
    // r's last token (the padding repeats it in the last block's last lane)
    const uint32_t rmax = nr ? ld_block(r4, (nr - 1) >> 2, rlim, err).w : 0u;
    if (32u * (uint32_t)warp < wi.n) {  // warp-uniform: the first batch's descriptors
        if (p_ok) p_desc = ld_at(I.s_desc, p_id, I.s_n_sets, err);
        pstage = 2;
    }
    __syncthreads();

    // the lane's pair: next block to merge (jb) and to ask for (jr), ring slot of its block 0
    // (rb); a finished pair keeps s_id / o until the maintenance step sends it out
    bool active = false, out = false;
    uint32_t s_id = 0, rems = 0, req = 0, o = 0, jb = 0, jr = 0, rb = 0;
    const uint4* s4 = nullptr;
    uint64_t slim = 0;
    for (;;) {
        // ---- walk steps
#pragma unroll
        for (int step = 0; step < kIndexSteps; ++step) {
            const uint32_t avail = jr;      // blocks asked for in earlier steps
            const uint32_t ahead = jr - jb;  // asked for, not yet merged (rems counts tokens from block jb)
            if (active && ahead < kIndexRing && 4 * ahead < rems) {
                if (in_bounds(jr, slim, err)) cp_async16(ring + ((rb + jr) & (kIndexRing - 1)), s4 + jr);
                ++jr;
            }
            cp_async_commit();
            cp_async_wait<1>();  // every block asked for before this step is in
            if (active && jb < avail) {
                const uint4 sc = ring[(rb + jb) & (kIndexRing - 1)];
                const uint32_t bw = bm_test(bm, sc.w, n_words, err);
                o += bm_test(bm, sc.x, n_words, err) + bm_test(bm, sc.y, n_words, err) +
                     bm_test(bm, sc.z, n_words, err) + bw;
                ++jb;
                if (rems <= 4 || sc.w >= rmax) {  // s's last block, or no later token of s can match
                    if (rems < 4) o -= (4u - rems) * bw;  // the lanes past s's end repeat its last token
                    rems = 0;
                    active = false;
                    out = emit_all || o >= req;
                } else {
                    rems -= 4;
                    if (early && o + rems < req) {
                        active = false;
                        out = emit_all;
                    }
                }
            }
        }
        // ---- maintenance: survivors out
        const uint32_t pmask = __ballot_sync(kFull, out);
        if (pmask) {
            unsigned long long b0 = 0;
            if (lane == 0) b0 = atomicAdd(I.count, (unsigned long long)__popc(pmask));
            if (!(flags & VF_COUNT_ONLY)) {
                b0 = __shfl_sync(kFull, b0, 0);
                if (out) emit_triple(I.out, I.cap, self_join, b0 + __popc(pmask & lt_mask), wi.r, s_id, o);
            }
            out = false;
        }
        // ---- preparation (a batch queued here makes room for the next one to be taken in the
        // same step, so a batch is taken every second round)
        if (pstage == 1) {
            if (p_ok) p_desc = ld_at(I.s_desc, p_id, I.s_n_sets, err);
            pstage = 2;
        } else {
            if (pstage == 2) {
                const uint32_t q = p_ok ? required_overlap(I.sim, I.p, I.den, I.magic, nr, p_desc.y) : 0u;
                const uint32_t m = __ballot_sync(kFull, p_ok);
                if (p_ok) queue[(qtail + __popc(m & lt_mask)) % kIndexQueue] = make_uint4(p_id, p_desc.x, p_desc.y, q);
                qtail += __popc(m);
                pstage = 0;
                __syncwarp();
            }
            if (pstage == 0) {
                if (!pdone && qtail - qhead + 32 <= kIndexQueue) {
                    uint32_t base = 0;
                    if (lane == 0) base = atomicAdd(&sm->next, 32u);
                    base = __shfl_sync(kFull, base, 0);
                    if (base + 32 >= wi.n) pdone = true;
                    const uint32_t my = base + (uint32_t)lane;
                    p_ok = my < wi.n;
                    if (p_ok) p_id = run[my].s & ~kInItem;
                    if (base < wi.n) pstage = 1;
                }
            }
        }
        // ---- idle lanes take queued candidates
        const uint32_t idle = __ballot_sync(kFull, !active);
        if (idle && qtail != qhead) {
            const uint32_t k = min((uint32_t)__popc(idle), qtail - qhead);
            const uint32_t rank = __popc(idle & lt_mask);
            if (!active && rank < k) {
                const uint4 e = queue[(qhead + rank) % kIndexQueue];
                rb = (rb + jr) & (kIndexRing - 1);  // continue the lane's ring after its last request
                s_id = e.x;
                rems = e.z;
                req = e.w;
                o = 0;
                jb = 0;
                jr = 0;
                s4 = I.s_toks4 + e.y;
                slim = I.s_n_chunks - e.y;
                if (rems == 0 || nr == 0) {
                    out = emit_all;  // an empty side: overlap 0
                } else {
                    active = true;
                }
            }
            qhead += k;
            __syncwarp();
        }
        if (pdone && pstage == 0 && qhead == qtail && !__any_sync(kFull, active || out)) break;
    }
    cp_async_wait<0>();  // the ring's last copies (asked for past a pair's end) are in
    __syncthreads();     // every thread is done with the bitmap
    bm_mark<BT>(bm, r4, nr, rlim, n_words, true, tid, err);
    __syncthreads();
}

// Instance of a probe slot: the last one whose first tile is not past it.
__device__ __forceinline__ uint32_t instance_of(const Instance* table, uint32_t n_inst, uint32_t slot) {
    uint32_t lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (table[mid].tile_base <= slot >> 5) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace

// -------------------------------------------------------------------------
// Persistent verification kernel.  Instance fields come from the device table
// (table_out).  The queued pairs' ids are valid and no pair is a set with
// itself (the plan kernel's checks).
// -------------------------------------------------------------------------
// MINB: CTAs per SM the registers are budgeted for (1024 / BT: 64 registers
// per thread; fewer CTAs leave more registers per thread).
template <int BT, int MINB>
__global__ void __launch_bounds__(BT, MINB) verify_kernel(VerifyArgs a) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ BlockSmem<BT> bsm;
    __shared__ uint64_t s_wbar[BT / 32];  // bulk staging: one barrier per warp for phase 2
    constexpr uint32_t kBlockWin = BT * kBlockD;
    constexpr int kWarps = BT / 32;

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const uint32_t n_warps_total = gridDim.x * kWarps;
    const uint32_t gwarp = blockIdx.x * kWarps + warp;
    const Instance* table = a.table_out;

    if (a.ctr->err & (ERR_OFFSETS | ERR_GUARD)) return;  // the plan is not trustworthy

    // Static first-round assignment: phase 1 takes CTAs [0, n_bs); lane items start
    // on the warps after those, long pairs on the warps after these, short pairs on the
    // rest, so a small batch spreads over idle warps at once.  Later rounds are dynamic.
    const unsigned long long n_block = min(a.ctr->block_items, (unsigned long long)a.block_item_cap);
    const unsigned long long n_warp = min(a.ctr->warp_items, (unsigned long long)a.warp_item_cap);
    const unsigned long long n_long = min(a.ctr->long_pairs, (unsigned long long)a.pair_cap);
    const unsigned long long n_pairs = min(a.ctr->thread_pairs, (unsigned long long)a.pair_cap);
    const uint32_t n_bs = (uint32_t)min(n_block, (unsigned long long)gridDim.x);
    const uint32_t free2 = n_bs * kWarps;
    const uint32_t slots2 = n_warps_total - free2;
    // Units of the pair lists: few pairs spread over the warps, many go several to a grab.  Of the long
    // pairs, those that work items cover are passed over, 32 at a time, so a grab takes the more of them
    // the fewer the others are (none: no units).  Where all of 1e7 pairs of 20 tokens are in index items
    // the kernel takes 375 us; 920 with every pair of the list read by itself.
    const unsigned long long n_lone = min(a.ctr->warp_pairs, n_long);
    const uint32_t long_grab = (uint32_t)max(
        1ull, min(n_long / (4ull * n_warps_total), min(kLongGrab * (n_long / max(n_lone, 1ull)), (unsigned long long)kLongScan)));
    const unsigned long long long_units = n_lone ? (n_long + long_grab - 1) / long_grab : 0;
    const uint32_t freel = free2 + (uint32_t)min(n_warp, (unsigned long long)slots2);
    const uint32_t slotsl = n_warps_total - freel;
    const uint32_t free3 = freel + (uint32_t)min(long_units, (unsigned long long)slotsl);
    const uint32_t slots3 = n_warps_total - free3;

    // ---------------- phase 1: block-per-pair items ----------------------
    if (n_block) {
        uint32_t* rbuf = smem;                                // kBlockRCap + 16
        uint32_t* wr = smem + kBlockRCap + 16;                // kBlockWin + 16
        uint32_t* ws = wr + kBlockWin + 16;                   // kBlockWin + 16
        uint32_t* bm = smem;                                  // index items' probe bitmap (a.index_words)
        bool bm_zero = false;                                 // CTA-uniform: bm holds zeros only
        uint32_t r_phase = 0;                                 // bulk staging: parity of bar[0]'s next phase
        uint32_t ph[2] = {0u, 0u};                            // the same for the candidate buffers' barriers
        if (a.bulk_stage) {
            if (tid == 0)
                for (int k = 0; k < 3; ++k) mbar_init(&bsm.bar[k], 1);
            __syncthreads();
        }
        for (uint32_t round = 0;; ++round) {
            if (tid == 0) bsm.item = round == 0 ? blockIdx.x : gridDim.x + atomicAdd(&a.ctr->block_cursor, 1u);
            __syncthreads();
            const uint32_t it = bsm.item;
            __syncthreads();
            if (it >= n_block) break;
            const WorkItem bi = a.block_items[it];
            if (!in_bounds(bi.inst, a.n_inst, &a.ctr->err)) continue;  // (uniform over the CTA)
            const Instance& I = table[bi.inst];
            const uint32_t flags = I.flags;
            const bool emit_all = (flags & VF_EMIT_ALL) != 0, early = !emit_all;
            const bool self_join = (flags & VF_SELF_JOIN) != 0;
            if (!in_bounds(bi.r, I.r_n_sets, &a.ctr->err)) continue;
            const uint2 dr = I.r_desc[bi.r];
            const uint32_t nr = dr.y;
            const uint4* r4 = I.r_toks4 + dr.x;
            if (bi.pad == 1) {  // index item (uniform over the CTA)
                if (!bm_zero) {  // the bitmap shares its memory with the block-merge buffers
                    uint4* b4 = reinterpret_cast<uint4*>(bm);
                    for (uint32_t k = tid; k < a.index_words / 4; k += BT) b4[k] = make_uint4(0u, 0u, 0u, 0u);
                    __syncthreads();
                    bm_zero = true;
                }
                uint4* rings = reinterpret_cast<uint4*>(bm + a.index_words);
                if (!in_bounds(bi.c0 + bi.n - 1, a.pair_cap, &a.ctr->err)) continue;
                index_item<BT>(I, bi, a.pairs + bi.c0, nr, r4, I.r_n_chunks - dr.x, bm, a.index_words, rings, rings + BT * kIndexRing,
                               &bsm, &a.ctr->err);
                continue;
            }
            bm_zero = false;
            const bool r_staged = nr + 4 <= kBlockRCap;
            const uint64_t rlim = I.r_n_chunks - dr.x;
            // bulk staging (a.bulk_stage): r by one bulk copy; each candidate's whole s by one bulk
            // copy into buffer m & 1 (wr / ws), issued while the previous candidate merges
            const bool bulk = a.bulk_stage && r_staged;
            uint32_t* sbuf[2] = {wr, ws};
            // thread 0: stage candidate m's s if it fits a buffer
            auto prefetch = [&](uint32_t m) -> uint32_t {
                if (m >= bi.n || !in_bounds(bi.c0 + m, a.pair_cap, &a.ctr->err)) return 0u;
                const uint2 dx = ld_at(I.s_desc, a.pairs[bi.c0 + m].s & ~kInItem, I.s_n_sets, &a.ctr->err);
                if (dx.y == 0 || dx.y + 4 > kBlockWin + 16) return 0u;
                bulk_stage(sbuf[m & 1], I.s_toks4 + dx.x, 0u, (dx.y + 3) >> 2, I.s_n_chunks - dx.x,
                           (kBlockWin + 16) / 4, &bsm.bar[1 + (m & 1)], &a.ctr->err);
                return 1u;
            };
            if (bulk) {
                if (tid == 0) {
                    bulk_stage(rbuf, r4, 0u, (nr + 3) >> 2, rlim, (kBlockRCap + 16) / 4, &bsm.bar[0], &a.ctr->err);
                    bsm.staged[0] = prefetch(0);
                    bsm.staged[1] = 0u;
                    bsm.ok = mbar_wait(&bsm.bar[0], r_phase, &a.ctr->err) ? 1u : 0u;
                    if (!bsm.ok && bsm.staged[0]) mbar_wait(&bsm.bar[1], ph[0], &a.ctr->err);  // own copy in flight
                }
                r_phase ^= 1u;
                __syncthreads();
                if (!bsm.ok) return;  // (uniform) a copy did not complete: reported, the CTA stops
            } else if (r_staged) {
                stage<BT>(r4, 0, nr, rbuf, tid, rlim, (kBlockRCap + 16) / 4, &a.ctr->err);
                __syncthreads();
            }
            for (uint32_t m = 0; m < bi.n; ++m) {
                bool s_whole = false;
                if (bulk) {
                    // candidate m - 1 is merged (its buffer is free again); stage m + 1 into it
                    s_whole = bsm.staged[m & 1] != 0;
                    __syncthreads();
                    if (tid == 0) {
                        bsm.staged[(m + 1) & 1] = prefetch(m + 1);
                        if (s_whole) {
                            bsm.ok = mbar_wait(&bsm.bar[1 + (m & 1)], ph[m & 1], &a.ctr->err) ? 1u : 0u;
                            bsm.staged[m & 1] = 0u;  // consumed
                            if (!bsm.ok && bsm.staged[(m + 1) & 1])  // own copy in flight
                                mbar_wait(&bsm.bar[1 + ((m + 1) & 1)], ph[(m + 1) & 1], &a.ctr->err);
                        }
                    }
                    if (s_whole) ph[m & 1] ^= 1u;
                    __syncthreads();
                    if (s_whole && !bsm.ok) return;  // (uniform) reported, the CTA stops
                }
                if (!in_bounds(bi.c0 + m, a.pair_cap, &a.ctr->err)) break;
                const uint32_t s = a.pairs[bi.c0 + m].s & ~kInItem;
                const uint2 ds = ld_at(I.s_desc, s, I.s_n_sets, &a.ctr->err);
                const uint32_t ns = ds.y;
                const uint32_t req = required_overlap(I.sim, I.p, I.den, I.magic, nr, ns);
                bool rej;
                const uint32_t o = block_merge<BT>(r4, nr, I.s_toks4 + ds.x, ns, req, early, rbuf, r_staged, wr,
                                                   bulk ? sbuf[m & 1] : ws, s_whole, &bsm, &rej
                                                   CHK_ARGS(I.r_n_chunks - dr.x, I.s_n_chunks - ds.x, &a.ctr->err));
                const bool pass = emit_all || (!rej && o >= req);
                if (pass && tid == 0) {
                    const unsigned long long idx = atomicAdd(I.count, 1ull);
                    if (!(flags & VF_COUNT_ONLY)) emit_triple(I.out, I.cap, self_join, idx, bi.r, s, o);
                }
            }
            __syncthreads();  // rbuf reuse
            if (bulk) {
                // a copy issued for a candidate the loop did not reach (it stopped at a bad index
                // of the checked build): wait for it so the barrier phases stay in step
                const uint32_t left0 = bsm.staged[0], left1 = bsm.staged[1];
                if (tid == 0) {
                    if (left0) mbar_wait(&bsm.bar[1], ph[0], &a.ctr->err);
                    if (left1) mbar_wait(&bsm.bar[2], ph[1], &a.ctr->err);
                }
                if (left0) ph[0] ^= 1u;
                if (left1) ph[1] ^= 1u;
                __syncthreads();
            }
        }
    }

    // ---------------- phase 2: lane items, then long pairs, one per warp --
    const bool few = few_pairs(n_long, n_pairs, n_warps_total, a.force_thread);
    if (n_warp || n_lone || (few && n_pairs)) {
        WarpOut wout;
        uint32_t* abuf = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(smem) + warp * kWarpSliceBytes);
        uint32_t* bbuf = abuf + kWarpABuf;
        // bulk staging: the warp's own barrier (phase parity wph, warp-uniform)
        uint64_t* wbar = a.bulk_stage ? &s_wbar[warp] : nullptr;
        uint32_t wph = 0;
        if (wbar) {
            if (lane == 0) mbar_init(wbar, 1);
            __syncwarp();
        }
        // r whole into abuf: by one bulk copy that lane 0 waits for, or by the lanes; false if the copy
        // did not complete (reported)
        auto stage_r = [&](const uint4* r4, uint32_t nr, uint64_t rlim) -> bool {
            __syncwarp();  // abuf reuse
            if (wbar) {
                uint32_t ok = 1;
                if (lane == 0) {
                    bulk_stage(abuf, r4, 0u, (nr + 3) >> 2, rlim, kWarpABuf / 4, wbar, &a.ctr->err);
                    ok = mbar_wait(wbar, wph, &a.ctr->err) ? 1u : 0u;
                }
                wph ^= 1u;
                if (!__shfl_sync(kFull, ok, 0)) return false;
            } else {
                stage<32>(r4, 0, nr, abuf, lane, rlim, kWarpABuf / 4, &a.ctr->err);
            }
            __syncwarp();
            return true;
        };
        for (uint32_t round = 0; n_warp; ++round) {
            uint32_t it = 0;
            if (lane == 0) {
                if (round == 0 && gwarp >= free2) it = gwarp - free2;
                else it = n_warp > slots2 ? slots2 + atomicAdd(&a.ctr->warp_cursor, 1u) : slots2;
            }
            it = __shfl_sync(kFull, it, 0);
            if (it >= n_warp) break;
            const WorkItem wi = a.warp_items[it];
            if (!in_bounds(wi.inst, a.n_inst, &a.ctr->err)) continue;  // (uniform over the warp)
            const Instance& I = table[wi.inst];
            if (!in_bounds(wi.r, I.r_n_sets, &a.ctr->err)) continue;
            if (!in_bounds(wi.c0 + wi.n - 1, a.pair_cap, &a.ctr->err)) continue;
            const uint2 dr = I.r_desc[wi.r];  // (lane items are made of probes that fit abuf)
            if (!stage_r(I.r_toks4 + dr.x, dr.y, I.r_n_chunks - dr.x)) return;  // the warp stops
            lane_item(I, wi, a.pairs + wi.c0, dr.y, reinterpret_cast<const uint4*>(abuf), lane, &a.ctr->err);
        }
        uint32_t held = 0, inst = 0;  // slot + 1 of the r in abuf, instance of the buffered survivors
        uint32_t counted = 0;         // results of that instance that are only counted
        auto flush = [&]() {
            wout.flush(table[inst], lane);
            if (counted && lane == 0) atomicAdd(table[inst].count, (unsigned long long)counted);
            counted = 0;
        };
        // one queued pair; false if a copy did not complete (reported)
        auto verify_pair = [&](const PairRef pr) -> bool {
            const uint32_t i = a.n_inst > 1 ? instance_of(table, a.n_inst, pr.k) : 0u;
            if (i != inst) flush();
            inst = i;
            const Instance& I = table[inst];
            const bool early = !(I.flags & VF_EMIT_ALL);
            if (!in_bounds(pr.k - 32u * I.tile_base, I.n_probes, &a.ctr->err)) return true;
            const uint32_t r = I.probe_ids[pr.k - 32u * I.tile_base];
            if (!in_bounds(r, I.r_n_sets, &a.ctr->err) || !in_bounds(pr.s, I.s_n_sets, &a.ctr->err)) return true;
            const uint2 dr = I.r_desc[r], ds = I.s_desc[pr.s];
            const uint32_t nr = dr.y, ns = ds.y;
            const uint4 *r4 = I.r_toks4 + dr.x, *s4 = I.s_toks4 + ds.x;
            const uint32_t req = required_overlap(I.sim, I.p, I.den, I.magic, nr, ns);
            uint32_t o;
            bool rej = false, failed;
            const bool staged = nr + 4 <= kWarpRCap;
            if (!staged) held = 0;  // (abuf becomes a window buffer)
            if (staged && held != pr.k + 1) {
                if (!stage_r(r4, nr, I.r_n_chunks - dr.x)) return false;
                held = pr.k + 1;
            }
            if (staged && !(I.flags & VF_FORCE_WARP)) {
                o = warp_lookup(abuf, nr, s4, ns, lane, I.s_n_chunks - ds.x, &a.ctr->err);
            } else {  // r is too long, or the merge path is asked for
                o = warp_merge(r4, nr, s4, ns, req, early, staged, abuf, bbuf, lane, wbar, &wph, I.s_n_chunks - ds.x,
                               &a.ctr->err, &failed, &rej CHK_ARGS(I.r_n_chunks - dr.x, I.s_n_chunks - ds.x, &a.ctr->err));
                if (failed) return false;
            }
            if (!early || (!rej && o >= req)) {
                if (I.flags & VF_COUNT_ONLY) ++counted;
                else wout.push(I, lane, r, pr.s, o);
            }
            return true;
        };
        if (few) {  // neighbouring pairs on different SMs
            for (unsigned long long u = (unsigned long long)warp * gridDim.x + blockIdx.x; u < n_long + n_pairs;
                 u += n_warps_total) {
                const unsigned long long at = u < n_long ? a.pair_cap - n_long + u : u - n_long;
                if (!in_bounds(at, a.pair_cap, &a.ctr->err)) continue;  // (uniform over the warp)
                const PairRef pr = a.pairs[at];
                if (!(pr.s & kInItem) && !verify_pair(pr)) return;  // the warp stops
            }
        } else {
            for (uint32_t round = 0; long_units; ++round) {
                uint32_t u = 0;
                if (lane == 0) {
                    if (round == 0 && gwarp >= freel) u = gwarp - freel;
                    else u = long_units > slotsl ? slotsl + atomicAdd(&a.ctr->long_cursor, 1u) : slotsl;
                }
                u = __shfl_sync(kFull, u, 0);
                if (u >= long_units) break;
                const unsigned long long first = a.pair_cap - n_long + (unsigned long long)u * long_grab;
                const unsigned long long end = min(first + long_grab, (unsigned long long)a.pair_cap);
                for (unsigned long long m = first; m < end; m += 32) {
                    PairRef mine;
                    mine.k = 0;
                    mine.s = m + lane < end ? 0u : kInItem;
                    if (m + lane < end) mine = a.pairs[m + lane];
                    for (uint32_t left = __ballot_sync(kFull, !(mine.s & kInItem)); left; left &= left - 1) {
                        PairRef pr;
                        pr.k = __shfl_sync(kFull, mine.k, __ffs(left) - 1);
                        pr.s = __shfl_sync(kFull, mine.s, __ffs(left) - 1);
                        if (!verify_pair(pr)) return;  // the warp stops
                    }
                }
            }
        }
        flush();
        __syncwarp();  // the slice is phase 3's now
    }

    // ---------------- phase 3: short pairs, one per thread ----------------
    if (!few) {
        ContEntry* cont = reinterpret_cast<ContEntry*>(reinterpret_cast<char*>(smem) + warp * kWarpSliceBytes);
        uint32_t n_cont = 0;  // warp-uniform
        const uint32_t grab = n_pairs > 4ull * 32 * n_warps_total ? kFlatGrab : 1u;
        const unsigned long long n_units = (n_pairs + 32 * grab - 1) / (32 * grab);
        const unsigned lt_mask = (1u << lane) - 1u;

        // drain_parked: the last m parked pairs, one per lane, merged while at
        // least min_live lanes still work; the rest are parked again.
        auto drain = [&](uint32_t m, uint32_t live) {
            n_cont = drain_parked(cont, n_cont, m, live, table, lane CHK_ERR_ARG(&a.ctr->err));
        };
        const uint32_t min_live = a.drain_min_live ? min(max(a.drain_min_live, 1u), 24u) : kDrainMinLive;

        for (uint32_t round = 0;; ++round) {
            uint32_t u = 0;
            if (lane == 0) {
                if (round == 0 && gwarp >= free3) u = gwarp - free3;
                else u = n_units > slots3 ? slots3 + atomicAdd(&a.ctr->chunk_cursor, 1u) : slots3;
            }
            u = __shfl_sync(kFull, u, 0);
            if (u >= n_units) break;
            for (uint32_t sub = 0; sub < grab; ++sub) {
                const unsigned long long first = ((unsigned long long)u * grab + sub) * 32;
                if (first >= n_pairs) break;  // warp-uniform
                // the next 32 pairs, parked at their start
                bool live = first + lane < n_pairs;
                uint32_t r = 0, inst = 0, req = 0;
                uint2 dr = make_uint2(0, 0), ds = make_uint2(0, 0);
                PairRef pr;
                pr.k = pr.s = 0;
                if (live) {
                    pr = a.pairs[first + lane];
                    if (a.n_inst > 1) inst = instance_of(table, a.n_inst, pr.k);
                    const Instance& I = table[inst];
                    live = in_bounds(pr.k - 32u * I.tile_base, I.n_probes, &a.ctr->err);
                    if (live) r = I.probe_ids[pr.k - 32u * I.tile_base];
                    live = live && in_bounds(r, I.r_n_sets, &a.ctr->err) && in_bounds(pr.s, I.s_n_sets, &a.ctr->err);
                    if (live) {
                        dr = I.r_desc[r];
                        ds = I.s_desc[pr.s];
                        req = required_overlap(I.sim, I.p, I.den, I.magic, dr.y, ds.y);
                    }
                }
                const uint32_t kmask = __ballot_sync(kFull, live);
                while (n_cont + 32 > kCont) drain(32, min_live);  // room for a full warp of parked pairs
                if (live && in_bounds(n_cont + __popc(kmask & lt_mask), kCont, &a.ctr->err)) {
                    ContEntry* ce = cont + n_cont + __popc(kmask & lt_mask);
                    ce->m0 = make_uint4(r, pr.s, dr.x, ds.x);
                    ce->m1 = make_uint4(dr.y, ds.y, req, 0u);
                    ce->m2 = make_uint4(inst, 0u, 0u, 0u);
                }
                n_cont += __popc(kmask);
                __syncwarp();
                if (n_cont >= 32) drain(32, min_live);
            }
        }
        // the tail: keep refilling lanes while more than a warp is parked, then finish
        while (n_cont) drain(min(n_cont, 32u), n_cont > 32 ? min_live : 1u);
    }
}

// -------------------------------------------------------------------------
// Host side of the launch.
// -------------------------------------------------------------------------

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static uint64_t item_cap(uint64_t n_probes, uint64_t n_cands, uint32_t per_item) {
    const uint64_t cap = n_probes + (n_cands + per_item - 1) / per_item;
    return cap > 0xFFFFFFF0ull ? 0xFFFFFFF0ull : cap;
}

// Candidates per warp / block work item: small batches get one candidate
// per item so that every warp holds at most one pair of the critical path;
// large batches get up to kWarpItemCands / kBlockItemCands to bound the
// number of dynamic-scheduling atomics.  (Estimates: 32 resident warps and
// 4 resident CTAs per SM.)
static void item_sizes(uint64_t n_cands, int num_sms, uint32_t* per_warp_item, uint32_t* per_block_item,
                       uint32_t* per_lane_item) {
    const uint64_t warps = 32ull * (uint64_t)num_sms, ctas = 4ull * (uint64_t)num_sms;
    uint64_t w = n_cands / (64 * warps), b = n_cands / (64 * ctas), l = n_cands / (8 * warps);
    *per_warp_item = (uint32_t)(w < 1 ? 1 : (w > kWarpItemCands ? kWarpItemCands : w));
    *per_block_item = (uint32_t)(b < 1 ? 1 : (b > kBlockItemCands ? kBlockItemCands : b));
    l = l < 32 ? 32 : (l > kLaneItemCands ? kLaneItemCands : l);
    *per_lane_item = (uint32_t)(l & ~31ull);
}

static uint64_t pair_cap(const LaunchShape& sh) { return sh.total_cands + 32ull * sh.n_tiles + 32; }

// Whole rounds of a wave's warps (plan kernel: 32 per SM), of chunks of at most
// about 1024; small chunks for small batches, so that all warps share the work.
// At least 64 once block items hold several pairs, so that the runs of pairs
// that chunk borders cut (one more work item each) fit the item lists (see
// bind_workspace).
uint32_t plan_chunk(uint64_t total_cands, int num_sms) {
    uint32_t wc, bc, lc;
    item_sizes(total_cands, num_sms, &wc, &bc, &lc);
    const uint64_t warps = plan_wave(num_sms);
    const uint64_t rounds = std::max<uint64_t>((total_cands + 1024 * warps - 1) / (1024 * warps), 1);
    const uint64_t per = (total_cands + warps * rounds - 1) / (warps * rounds);
    const uint32_t c = std::max<uint32_t>((uint32_t)((per + 31) & ~31ull), 32u);
    return bc > 1 && c < 64 ? 64u : c;
}

LaunchShape single_shape(uint32_t n_probes, uint64_t n_cands, int num_sms) {
    LaunchShape sh;
    sh.n_inst = 1;
    sh.n_tiles = (n_probes + 31) / 32;
    sh.total_probes = n_probes;
    sh.total_cands = n_cands;
    sh.n_chunks = chunks_of(n_probes, n_cands, plan_chunk(n_cands, num_sms));
    return sh;
}

size_t workspace_bytes(const LaunchShape& sh, int num_sms) {
    uint32_t wc, bc, lc;
    item_sizes(sh.total_cands, num_sms, &wc, &bc, &lc);
    const uint64_t slots = 32ull * sh.n_tiles + 1, pc = pair_cap(sh);
    // (the terms by probe slot and pc / 8 are room for work items, see bind_workspace)
    return align256(sizeof(Counters)) + align256(sizeof(Instance) * ((size_t)sh.n_inst + 1)) +
           align256(sizeof(uint2) * slots) + align256(sizeof(uint32_t) * slots) +
           align256(sizeof(uint32_t) * (pc / 32 + 1)) + align256(sizeof(PairRef) * pc) +
           align256(sizeof(WorkItem) * ((size_t)item_cap(sh.total_probes, sh.total_cands, wc) + 1)) +
           align256(sizeof(WorkItem) * ((size_t)item_cap(sh.total_probes, sh.total_cands, bc) + 1));
}

size_t workspace_bytes(uint32_t n_probes, uint64_t n_cands, int num_sms) {
    return workspace_bytes(single_shape(n_probes, n_cands, num_sms), num_sms);
}

void bind_workspace(VerifyArgs& a, void* ws, const LaunchShape& sh, int num_sms) {
    char* p = static_cast<char*>(ws);
    uint32_t wc;
    item_sizes(sh.total_cands, num_sms, &wc, &a.block_item_cands, &a.lane_item_cands);
    a.n_inst = sh.n_inst;
    a.n_tiles = sh.n_tiles;
    a.total_probes = sh.total_probes;
    a.total_cands = sh.total_cands;
    a.chunk = plan_chunk(sh.total_cands, num_sms);
    a.n_chunks = sh.n_chunks;
    a.chunk_begin = 0;
    a.ctr = reinterpret_cast<Counters*>(p);
    p += align256(sizeof(Counters));
    a.table_out = reinterpret_cast<Instance*>(p);
    p += align256(sizeof(Instance) * ((size_t)sh.n_inst + 1));
    a.pair_cap = pair_cap(sh);
    a.pairs = reinterpret_cast<PairRef*>(p);
    p += align256(sizeof(PairRef) * a.pair_cap);
    // Work items are made of runs, a probe's pairs of one chunk that are queued together: at most one
    // per probe, one more per chunk border and one more per early flush (every kPlanFlush pairs; chunks
    // are longer than that only in large batches).  Lane items take up to 32 pairs or more of a run,
    // block items up to block_item_cands; neither are more than the pairs.  The lists share what the
    // workspace holds beside the pair list, at least 48 bytes per probe and 36 (single pairs per warp
    // and block item) to 4.6 bytes per candidate.
    const uint64_t cuts = sh.n_chunks + sh.total_cands / kPlanFlush + 1;
    const uint64_t lane_items = std::min<uint64_t>(sh.total_probes + cuts + sh.total_cands / 32,
                                                   item_cap(sh.total_probes, sh.total_cands, wc));
    a.warp_items = reinterpret_cast<WorkItem*>(p);
    a.warp_item_cap = (uint32_t)std::min<uint64_t>(lane_items, 0xFFFFFFF0ull);
    p += align256(sizeof(WorkItem) * ((size_t)a.warp_item_cap + 1));
    a.block_items = reinterpret_cast<WorkItem*>(p);
    const size_t left = static_cast<char*>(ws) + workspace_bytes(sh, num_sms) - p;
    a.block_item_cap = (uint32_t)(left / sizeof(WorkItem) > 0xFFFFFFF0ull ? 0xFFFFFFF0ull : left / sizeof(WorkItem));
}

void bind_workspace(VerifyArgs& a, void* ws, uint32_t n_probes, uint64_t n_cands, int num_sms) {
    bind_workspace(a, ws, single_shape(n_probes, n_cands, num_sms), num_sms);
}

// Dynamic shared memory of the verify kernel: the largest of the block
// phase's buffers, the per-warp slices of phases 2 and 3, and the index
// items' probe bitmap (index_words words; it overlaps the others).
template <int BT>
static size_t verify_smem_bytes(uint32_t index_words) {
    constexpr uint32_t kBlockWin = BT * kBlockD;
    const size_t block_phase = sizeof(uint32_t) * (kBlockRCap + 16 + 2 * (kBlockWin + 16));
    const size_t warp_phases = (size_t)(BT / 32) * kWarpSliceBytes;
    // index items: the bitmap, then each thread's block ring, then each warp's candidate queue
    const size_t bitmap = index_words ? sizeof(uint32_t) * (size_t)index_words +
                                            sizeof(uint4) * ((size_t)BT * kIndexRing + (size_t)(BT / 32) * kIndexQueue)
                                      : 0;
    size_t m = block_phase > warp_phases ? block_phase : warp_phases;
    return bitmap > m ? bitmap : m;
}

// CTAs per SM of the persistent kernel for a dynamic shared-memory size, per
// device: the size attribute is raised once per device and variant to the
// largest size any launch uses, the occupancy query runs once per size
// (sizes come in 4 KiB steps above the fixed part).
template <int BT, int MINB>
static cudaError_t resident_ctas(size_t smem, int* per_sm) {
    constexpr int kMaxDev = 64;
    constexpr int kSteps = 64;
    static std::atomic<int> attr_set[kMaxDev];
    static std::atomic<int> cache[kMaxDev][kSteps];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const size_t base = verify_smem_bytes<BT>(0);
    const size_t step = smem > base ? (smem - base + 4095) / 4096 : 0;
    const bool cacheable = dev >= 0 && dev < kMaxDev && step < (size_t)kSteps;
    if (cacheable && cache[dev][step].load() > 0) {
        *per_sm = cache[dev][step].load();
        return cudaSuccess;
    }
    if (!(dev >= 0 && dev < kMaxDev && attr_set[dev].load())) {
        const size_t most = verify_smem_bytes<BT>(kIndexMaxWords);
        e = cudaFuncSetAttribute(verify_kernel<BT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDev) attr_set[dev].store(1);
    }
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, verify_kernel<BT, MINB>, BT, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) n = 1;
    if (cacheable) cache[dev][step].store(n);
    *per_sm = n;
    return cudaSuccess;
}

template <int BT, int MINB>
static cudaError_t launch_bt(const VerifyArgs& a, cudaStream_t st, int num_sms) {
    int per_sm = 0;
    const size_t smem = verify_smem_bytes<BT>(a.index_words);
    cudaError_t e = resident_ctas<BT, MINB>(smem, &per_sm);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(num_sms * per_sm));
    cfg.blockDim = dim3(BT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (a.l2_base && a.l2_bytes) {
        // the collection's tokens persist in the L2 set-aside during this launch
        memset(attr, 0, sizeof(attr));
        attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[0].val.accessPolicyWindow.base_ptr = const_cast<void*>(a.l2_base);
        attr[0].val.accessPolicyWindow.num_bytes = a.l2_bytes;
        attr[0].val.accessPolicyWindow.hitRatio = a.l2_hit_ratio;
        attr[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
        attr[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    e = cudaLaunchKernelEx(&cfg, verify_kernel<BT, MINB>, a);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// block_threads: 128, 256 or 512, optionally | kWideRegisters (the variant
// budgeted for fewer CTAs per SM, with more registers per thread: 7 of 8
// CTAs of 128 threads, 3 of 4 of 256, 1 of 2 of 512) and | kBulkStaging (a
// launch argument, not a variant).
template <class F>
static cudaError_t dispatch_variant(uint32_t block_threads, F&& f) {
    const bool wide = (block_threads & kWideRegisters) != 0;
    switch (block_threads & ~(kWideRegisters | kBulkStaging)) {
        case 128: return wide ? f.template operator()<128, 7>() : f.template operator()<128, 8>();
        case 512: return wide ? f.template operator()<512, 1>() : f.template operator()<512, 2>();
        default: return wide ? f.template operator()<256, 3>() : f.template operator()<256, 4>();
    }
}

struct PrepareVariant {
    uint32_t index_words;
    template <int BT, int MINB>
    cudaError_t operator()() const {
        int per_sm = 0;
        return resident_ctas<BT, MINB>(verify_smem_bytes<BT>(index_words), &per_sm);
    }
};

struct LaunchVariant {
    const VerifyArgs& a;
    cudaStream_t st;
    int num_sms;
    template <int BT, int MINB>
    cudaError_t operator()() const {
        return launch_bt<BT, MINB>(a, st, num_sms);
    }
};

cudaError_t prepare_verify(uint32_t block_threads, uint32_t index_words) {
    return dispatch_variant(block_threads, PrepareVariant{index_words});
}

cudaError_t launch_verify(const VerifyArgs& a, cudaStream_t st, int num_sms, uint32_t block_threads,
                          cudaEvent_t* ev) {
    cudaError_t e = cudaMemsetAsync(a.ctr, 0, sizeof(Counters), st);
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[0], st);
    if (a.n_inst == 0) {
        if (ev) {
            cudaEventRecord(ev[1], st);
            cudaEventRecord(ev[2], st);
        }
        return cudaSuccess;
    }
    // the plan kernel also runs for empty batches: it clears the instances' counts
    e = launch_plan(a, st, num_sms);
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[1], st);
    e = launch_merge(a, st, num_sms, block_threads);
    if (ev) cudaEventRecord(ev[2], st);
    return e;
}

// The verify kernel on the pairs and items that a's lists hold.
cudaError_t launch_merge(const VerifyArgs& a, cudaStream_t st, int num_sms, uint32_t block_threads) {
    VerifyArgs va = a;
    va.bulk_stage = (block_threads & kBulkStaging) ? 1u : 0u;
    return dispatch_variant(block_threads, LaunchVariant{va, st, num_sms});
}

// Items: at most one per probe's run and per kJoinBlockCands pairs, and one more wherever a run is
// cut (every kJoinRun - 32 pairs).  Runs: full ones, and one per warp of the join kernel.
constexpr uint32_t kJoinBlockCands = 8;
static uint64_t join_items(uint32_t n_probes, uint64_t pairs) {
    return std::min<uint64_t>(pairs, (uint64_t)n_probes + pairs / 4) + 1;
}
static uint64_t join_runs(uint64_t pairs, int num_sms) { return pairs / (kJoinRun - 32) + 64ull * num_sms + 1; }

size_t join_workspace_bytes(uint32_t n_probes, uint64_t pairs, int num_sms) {
    return align256(sizeof(Counters)) + align256(2 * sizeof(Instance)) + align256(sizeof(PairRef) * pairs) +
           2 * align256(sizeof(WorkItem) * join_items(n_probes, pairs)) + align256(sizeof(uint2) * pairs) +
           align256(sizeof(ulonglong2) * join_runs(pairs, num_sms));
}

JoinQueue bind_join_workspace(VerifyArgs& a, void* ws, uint32_t n_probes, uint64_t pairs, int num_sms) {
    char* p = static_cast<char*>(ws);
    auto take = [&](size_t bytes) {
        char* at = p;
        p += align256(bytes);
        return at;
    };
    a.block_item_cands = kJoinBlockCands;
    a.lane_item_cands = 32;
    a.n_inst = 1;
    a.n_tiles = (n_probes + 31) / 32;
    a.total_probes = n_probes;
    a.total_cands = pairs;
    a.ctr = reinterpret_cast<Counters*>(take(sizeof(Counters)));
    a.table_out = reinterpret_cast<Instance*>(take(2 * sizeof(Instance)));
    a.pair_cap = pairs;
    a.pairs = reinterpret_cast<PairRef*>(take(sizeof(PairRef) * pairs));
    const uint64_t items = join_items(n_probes, pairs);
    a.warp_item_cap = a.block_item_cap = (uint32_t)std::min<uint64_t>(items, 0xFFFFFFF0ull);
    a.warp_items = reinterpret_cast<WorkItem*>(take(sizeof(WorkItem) * items));
    a.block_items = reinterpret_cast<WorkItem*>(take(sizeof(WorkItem) * items));
    JoinQueue q;
    q.pairs = reinterpret_cast<uint2*>(take(sizeof(uint2) * pairs));
    q.run_cap = join_runs(pairs, num_sms);
    q.runs = reinterpret_cast<ulonglong2*>(take(sizeof(ulonglong2) * q.run_cap));
    q.pair_cap = pairs;
    return q;
}

}  // namespace ssj
