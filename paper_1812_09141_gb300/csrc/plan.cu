// Plan kernel: checks a launch's grouped candidate lists and drops the pairs
// that their sets' signatures prove dissimilar; what is left is queued for
// the verify kernel.
//
// The signature test is the bitmap filter of Sandes, Teodoro and Melo
// ("Bitmap filter: speeding up exact set similarity joins with bitwise
// operations", 2020): a set's record (layout.cu) holds its length, a bitmap
// of its tokens' hash values, and its loss, the number of tokens that share
// a bit with another token of the set.  With a the common bits of two
// bitmaps, |r n s| <= a + min(loss_r, loss_s): every common token sets a
// common bit, and of the tokens of x on common bits at most loss_x are not
// the first on their bit.  The bound is tested with the exact integer form of
// the similarity function, which is monotone in the overlap, so a pair that
// passes the join is never dropped.  (The bound never exceeds min(|r|, |s|),
// so the test includes the length filter of Section 2.2.3.)
//
// Two levels: a short record first (about one bit per token), and for the
// pairs that it leaves, a few percent, a long one.
//
// What bounds it: the records gathered from L2 (32 to 256 bytes a candidate,
// by the collections' set sizes, instead of the tokens the merge would read:
// 4 bytes each, of both sets, up to the positional filter's stop) and the
// instructions that count their common bits, about three per four bytes.
// Verification of 9.2e7 candidates of long sets (about 300 tokens, t = 0.6)
// took 5.2 ms when every candidate was walked against a bitmap of its probe;
// the test takes 1.10 ms (64 bytes per candidate, 6e9 bytes from L2) and
// leaves 47 us of merging.  On 5.7e6 candidates of short sets (about 20
// tokens) 55 us, leaving 18 us, instead of 195 us of merging.
#include <cstdint>
#include <cuda_runtime.h>

#include "arith.h"
#include "checked.cuh"
#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kPlanThreads = 256;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr uint32_t kPlanBuf = kPlanFlush + 32;  // survivors buffered per warp
constexpr int kSectors = 2;                     // 32-byte record loads in flight per lane, at most (4: 2% slower)
constexpr uint32_t kOneProbe = 64;              // candidates of a list worth rounds of their own (32: the same)
// CTAs per SM the registers are budgeted for (64 each).  With 3 and 4 loads in flight the long sets
// take 1.25 ms instead of 1.10, with 5 the spills cost more than the warps gain (1.32).
constexpr int kPlanCtas = 4;

// Instance fields read by the plan kernel (from the kernel parameters for a
// one-batch launch, else from the device table).
struct PlanInst {
    const uint32_t* probe_ids;
    const uint64_t* cand_offsets;
    const uint32_t* cand_ids;
    const uint4* r_rec[2];
    const uint4* s_rec[2];
    const uint2* r_desc;
    const uint2* s_desc;
    uint64_t n_cands, chunk_base;
    uint32_t r_n_sets, s_n_sets, n_probes, tile_base, flags, sim, p, den;
    uint32_t rec_sectors[2];
};

__device__ __forceinline__ PlanInst plan_inst(const Instance& I) {
    PlanInst q;
    q.probe_ids = I.probe_ids;
    q.cand_offsets = I.cand_offsets;
    q.cand_ids = I.cand_ids;
    q.r_desc = I.r_desc;
    q.s_desc = I.s_desc;
    q.n_cands = I.n_cands;
    q.chunk_base = I.chunk_base;
    q.r_n_sets = I.r_n_sets;
    q.s_n_sets = I.s_n_sets;
    q.n_probes = I.n_probes;
    q.tile_base = I.tile_base;
    q.flags = I.flags;
    q.sim = I.sim;
    q.p = I.p;
    q.den = I.den;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        q.r_rec[l] = I.r_rec[l];
        q.s_rec[l] = I.s_rec[l];
        q.rec_sectors[l] = I.rec_sectors[l];
    }
    return q;
}

// Does overlap o reach the threshold (Table "Similarity Functions", exact
// integer forms)?  Empty sets never match.
__device__ __forceinline__ bool overlap_passes(const PlanInst& I, uint32_t o, uint32_t nr, uint32_t ns) {
    if (nr == 0 || ns == 0) return false;
    if (I.sim == SIM_COSINE) return cosine_pass(o, I.p, I.den, nr, ns);
    if (I.sim == SIM_OVERLAP) return o >= I.den;
    return (uint64_t)o * I.den >= (uint64_t)I.p * ((uint64_t)nr + ns);  // Jaccard: den = p + q, Dice: 2q
}

// One 32-byte sector of a record.
struct Sector {
    uint32_t w[8];
};

__device__ __forceinline__ Sector ld_sector(const uint4* p) {
    Sector x;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3]), "=r"(x.w[4]), "=r"(x.w[5]), "=r"(x.w[6]), "=r"(x.w[7])
        : "l"(p));
    return x;
}

// Common bits of two sectors, the first word only where `first` has bits:
// full adders (a sum and a carry of three words, one logic operation each)
// turn eight words into four to count, since counting runs at a fraction of
// the rate of logic.
__device__ __forceinline__ uint32_t common_bits(const Sector& x, const Sector& y, uint32_t first) {
    uint32_t v[8];
    v[0] = x.w[0] & y.w[0] & first;
#pragma unroll
    for (int i = 1; i < 8; ++i) v[i] = x.w[i] & y.w[i];
    auto sum = [](uint32_t p, uint32_t q, uint32_t r) { return p ^ q ^ r; };
    auto carry = [](uint32_t p, uint32_t q, uint32_t r) { return (p & q) | (p & r) | (q & r); };
    const uint32_t s1 = sum(v[0], v[1], v[2]), c1 = carry(v[0], v[1], v[2]);
    const uint32_t s2 = sum(v[3], v[4], v[5]), c2 = carry(v[3], v[4], v[5]);
    const uint32_t s3 = sum(s1, s2, v[6]), c3 = carry(s1, s2, v[6]);
    const uint32_t s4 = sum(c1, c2, c3), c4 = carry(c1, c2, c3);
    return __popc(s3) + __popc(v[7]) + 2 * __popc(s4) + 4 * __popc(c4);
}

// Sum over the G lanes of a group of their part[i], i the lane's place in the
// group: a butterfly that halves the values at each step.
template <int G>
__device__ __forceinline__ uint32_t sum_of_group(uint32_t (&part)[G], uint32_t sub) {
#pragma unroll
    for (int m = G / 2; m > 0; m /= 2) {
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const bool up = (sub & m) != 0;
            const uint32_t give = up ? part[i] : part[i + m], keep = up ? part[i + m] : part[i];
            part[i] = keep + __shfl_xor_sync(kFull, give, m);
        }
    }
    return part[0];
}

// For the lane's own pair (any valid ids s, r): |s| in the upper half, the
// bound on the overlap in the lower half (see the record header, rec_bits).
// G lanes read a record, a sector each, so that a load takes whole lines (a
// lane reading its own record 16 bytes at a time costs one L1 wavefront per
// lane and load: with 128-byte records 90% of the L1's wavefronts and twice
// the time); the partial counts of the group's G pairs are then summed across
// it.  kSame: every lane's probe is the one whose sector of this lane is rs.
template <int G, bool kSame>
__device__ __forceinline__ uint32_t bound_of_pair(const uint4* s_rec, const uint4* r_rec, uint32_t s, uint32_t r,
                                                  const Sector& rs, int lane, uint32_t* r_head = nullptr) {
    const uint32_t sub = lane % G;
    const uint32_t first = sub == 0 ? 0u : kFull;  // the first sector's first word is the header
    constexpr int kBatch = G < kSectors ? G : kSectors;  // loads in flight
    uint32_t part[G];
#pragma unroll
    for (int b = 0; b < G; b += kBatch) {
        Sector x[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const uint32_t sj = G == 1 ? s : __shfl_sync(kFull, s, b + i, G);
            x[i] = ld_sector(s_rec + ((uint64_t)sj * G + sub) * 2);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            uint32_t hr;
            if (kSame) {
                part[b + i] = common_bits(x[i], rs, first);
                hr = rs.w[0];
            } else {
                const uint32_t rj = G == 1 ? r : __shfl_sync(kFull, r, b + i, G);
                const Sector y = ld_sector(r_rec + ((uint64_t)rj * G + sub) * 2);
                part[b + i] = common_bits(x[i], y, first);
                hr = y.w[0];
                if (G == 1) *r_head = hr;
            }
            if (G == 1 || sub == 0) part[b + i] += (x[i].w[0] & 0xFFFF0000u) + min(x[i].w[0] & 0xFFFFu, hr & 0xFFFFu);
        }
    }
    return sum_of_group<G>(part, sub);
}

// The signature test of a pair from its bound_of_pair value and |r| (65535 in
// a header: 65535 tokens or more, not tested).
__device__ __forceinline__ bool bound_passes(const PlanInst& I, uint32_t v, uint32_t nr) {
    const uint32_t ns = v >> 16;
    return ns == 0xFFFFu || nr == 0xFFFFu || overlap_passes(I, v & 0xFFFFu, nr, ns);
}

// Second level: the n buffered pairs tested with the long records; the ones
// left stay in the buffer, in order.  Returns their number.
template <int G>
__device__ __noinline__ uint32_t second_level(const PlanInst& I, uint2* buf, uint32_t n, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    uint32_t left = 0;
    for (uint32_t t = 0; t < n; t += 32) {
        const bool have = t + lane < n;
        const uint2 e = buf[have ? t + lane : t];
        const uint32_t r = __ldg(I.probe_ids + (e.x - 32u * I.tile_base));
        const uint32_t r_head = __ldg(&I.r_rec[1][(uint64_t)r * G * 2].x);
        const uint32_t v = bound_of_pair<G, false>(I.s_rec[1], I.r_rec[1], e.y, r, Sector(), lane);
        const bool pass = have && bound_passes(I, v, r_head >> 16);
        const uint32_t m = __ballot_sync(kFull, pass);  // (every lane has read its entry)
        if (pass) buf[left + __popc(m & lt_mask)] = e;
        left += __popc(m);
        __syncwarp();
    }
    return left;
}

// Granularity of a probe with |r| = nr and n candidates left: 0 thread per
// pair, 1 warp per pair, 2 block per pair, 3 lane per pair with r in the
// warp's shared memory (Alternative B; needs r to fit and enough candidates
// to occupy the lanes), 4 index items (many candidates, when the launch's
// token values fit the probe bitmap).
__device__ __forceinline__ uint32_t probe_bin(const VerifyArgs& a, uint32_t flags, uint32_t nr, uint32_t n) {
    const bool lane_ok = nr + 4 <= kWarpRCap;
    if (flags & VF_FORCE_INDEX) return a.index_words ? 4u : (lane_ok ? 3u : 1u);
    if (flags & VF_FORCE_BLOCK) return 2;
    if (flags & VF_FORCE_WARP) return 1;
    if (flags & VF_FORCE_THREAD) return 0;
    if (flags & VF_FORCE_LANE) return lane_ok ? 3u : 1u;
    if (a.index_words && a.index_min_cands && n >= min(a.index_min_cands, kPlanFlush)) return 4;
    const uint64_t key = 2ull * nr;  // |r|+|s| at |s| = |r|
    if (key <= a.thread_max_key) return 0;
    if (key <= a.lane_max_key && lane_ok && n >= kLaneMinCands) return 3;
    return key <= a.warp_max_key ? 1u : 2u;
}

// Queue the pairs that the second level leaves of the warp's n buffered ones
// (probe slot, candidate id), in candidate order.  Short pairs go to the front of the pair list, the others
// to its back, a probe's pairs side by side; lane, block and index items
// refer to such a run, and its pairs are marked (kInItem) so that the
// warp-per-pair phase passes over them.
__device__ __noinline__ void flush_survivors(const VerifyArgs& a, const PlanInst& I, uint32_t inst, uint2* buf,
                                             uint32_t n, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    switch (I.rec_sectors[1]) {
        case 2: n = second_level<2>(I, buf, n, lane); break;
        case 4: n = second_level<4>(I, buf, n, lane); break;
        case 8: n = second_level<8>(I, buf, n, lane); break;
        default: break;
    }
    if (n == 0) return;
    uint32_t* err = &a.ctr->err;
    // bin of entry i and the run [h, e) of its probe's entries
    auto classify = [&](uint32_t i, uint32_t* h, uint32_t* e, uint32_t* r) -> uint32_t {
        const uint32_t slot = buf[i].x;
        uint32_t lo = 0, hi = i;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (buf[mid].x < slot) lo = mid + 1; else hi = mid;
        }
        *h = lo;
        lo = i + 1;
        hi = n;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (buf[mid].x <= slot) lo = mid + 1; else hi = mid;
        }
        *e = lo;
        *r = I.probe_ids[slot - 32u * I.tile_base];
        return probe_bin(a, I.flags, I.r_desc[*r].y, *e - *h);
    };
    uint32_t n_long = 0;
    for (uint32_t t = 0; t < n; t += 32) {
        uint32_t h, e, r;
        const bool is_long = t + lane < n && classify(t + lane, &h, &e, &r) != 0;
        n_long += __popc(__ballot_sync(kFull, is_long));
    }
    unsigned long long base_s = 0, base_l = 0;
    if (lane == 0) {
        if (n > n_long) base_s = atomicAdd(&a.ctr->thread_pairs, (unsigned long long)(n - n_long));
        if (n_long) base_l = atomicAdd(&a.ctr->long_pairs, (unsigned long long)n_long);
    }
    base_s = __shfl_sync(kFull, base_s, 0);
    base_l = __shfl_sync(kFull, base_l, 0);
    // every candidate is queued at most once, so the lists never meet
    if (base_s + (n - n_long) > a.pair_cap || base_l + n_long > a.pair_cap) {
        if (lane == 0) atomicOr(err, ERR_GUARD);
        return;
    }
    unsigned long long at_s = base_s, at_l = a.pair_cap - base_l - n_long;
    for (uint32_t t = 0; t < n; t += 32) {
        const uint32_t i = t + lane;
        uint32_t h = 0, e = 0, r = 0, bin = 5;
        if (i < n) bin = classify(i, &h, &e, &r);
        const uint32_t ms = __ballot_sync(kFull, bin == 0), ml = __ballot_sync(kFull, bin >= 1 && bin <= 4);
        const unsigned long long pos = bin == 0 ? at_s + __popc(ms & lt_mask) : at_l + __popc(ml & lt_mask);
        at_s += __popc(ms);
        at_l += __popc(ml);
        if (bin <= 4 && in_bounds(pos, a.pair_cap, err)) {
            PairRef pr;
            pr.k = buf[i].x;
            pr.s = buf[i].y | (bin >= 2 ? kInItem : 0u);
            a.pairs[pos] = pr;
        }
        // items, by the first entry of a run
        const bool head = i < n && i == h;
        const uint32_t per = bin == 3 ? a.lane_item_cands : (bin == 4 ? a.index_item_cands : a.block_item_cands);
        const uint32_t items = head && bin >= 2 ? (e - h + per - 1) / per : 0u;
        uint32_t wn = bin == 3 ? items : 0u, bn = bin == 3 ? 0u : items;
        if (__any_sync(kFull, items != 0)) {
            uint32_t wincl = wn, bincl = bn;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t yw = __shfl_up_sync(kFull, wincl, off), yb = __shfl_up_sync(kFull, bincl, off);
                if (lane >= off) { wincl += yw; bincl += yb; }
            }
            unsigned long long wbase = 0, bbase = 0;
            if (lane == 31) {
                if (wincl) wbase = atomicAdd(&a.ctr->warp_items, (unsigned long long)wincl);
                if (bincl) bbase = atomicAdd(&a.ctr->block_items, (unsigned long long)bincl);
            }
            wbase = __shfl_sync(kFull, wbase, 31) + (wincl - wn);
            bbase = __shfl_sync(kFull, bbase, 31) + (bincl - bn);
            for (uint32_t it = 0; it < items; ++it) {
                WorkItem wi;
                wi.r = r;
                wi.n = min(per, e - h - it * per);
                wi.c0 = pos + (uint64_t)it * per;
                wi.inst = inst;
                wi.pad = bin >= 3 ? 1u : 0u;
                const unsigned long long q = (bin == 3 ? wbase : bbase) + it;
                if (q >= (bin == 3 ? a.warp_item_cap : a.block_item_cap)) {
                    atomicOr(err, ERR_GUARD);
                    break;
                }
                (bin == 3 ? a.warp_items : a.block_items)[q] = wi;
            }
        }
    }
    __syncwarp();
}

// Largest k with offs[k] <= f, by the whole warp: each step narrows the range
// [lo, hi) of candidate answers 32-fold with one load per lane.  (Offsets that
// are not nondecreasing give some k below n_probes.)
__device__ __forceinline__ uint32_t find_probe(const uint64_t* offs, uint32_t n_probes, uint64_t f, int lane) {
    uint32_t lo = 0, hi = n_probes;
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32;
        const uint64_t at = (uint64_t)lo + (uint64_t)step * lane;
        const bool le = lane == 0 || (at < hi && __ldg(offs + at) <= f);
        const uint32_t m = __ballot_sync(kFull, le);
        const uint32_t last = 31 - __clz(m);
        const uint64_t end = (uint64_t)lo + (uint64_t)step * (last + 1);
        lo += step * last;
        if (end < hi) hi = (uint32_t)end;
    }
    return lo;
}

// Candidates [f0, f1) of an instance, by one warp, 32 at a time; the pairs
// left go to buf, *n of them, and the position up to which candidates are done
// is returned: f1, or less when the buffer is full.  (The caller queues them:
// a call in here would cost the loops their registers.)  The warp holds a window of 32 list ends; rounds within one probe's list keep the
// probe's record in registers, in the others each lane finds its candidate's
// probe in the window and reads its record.  G: sectors per record of the
// first level, 0 without signatures (the length filter alone).
template <int G>
__device__ __forceinline__ uint64_t filter_chunk(const PlanInst& I, uint64_t f0, uint64_t f1, uint2* buf,
                                                 uint32_t* n_out, uint32_t* err, int lane) {
    constexpr int kG = G > 0 ? G : 1;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool emit_all = (I.flags & VF_EMIT_ALL) != 0, self_join = (I.flags & VF_SELF_JOIN) != 0;
    const uint32_t len = (uint32_t)(f1 - f0), slot0 = 32u * I.tile_base, s_n_sets = I.s_n_sets;
    const uint32_t* cands = I.cand_ids + f0;
    // lane l of the window holds probe kb + l: its id, and the end of its list relative to f0 (saturated;
    // the last probe's list ends the batch)
    uint32_t kb = find_probe(I.cand_offsets, I.n_probes, f0, lane), ends, ids;
    auto list_end = [&](uint32_t k) -> uint32_t {
        const uint64_t at = (uint64_t)k + 1 + lane;
        if (at >= I.n_probes) return 0xFFFFFFFFu;
        const uint64_t v = __ldg(I.cand_offsets + at);
        return v <= f0 ? 0u : (uint32_t)min(v - f0, (uint64_t)0xFFFFFFFFu);
    };
    auto window = [&](uint32_t k) {
        kb = k;
        ends = list_end(k);
        ids = (uint64_t)k + lane < I.n_probes ? __ldg(I.probe_ids + k + lane) : 0xFFFFFFFFu;
    };
    window(kb);
    uint32_t n = 0;  // buffered pairs (warp-uniform)
    auto keep = [&](bool pass, uint32_t slot, uint32_t s) {
        const uint32_t m = __ballot_sync(kFull, pass);
        if (m == 0) return;
        const uint32_t q = n + __popc(m & lt_mask);
        if (pass && in_bounds(q, kPlanBuf, err)) buf[q] = make_uint2(slot, s);
        n += __popc(m);
    };
    uint32_t s_next = (uint32_t)lane < len ? __ldg(cands + lane) : 0u;  // the lane's candidate of the next round
    auto next = [&](uint32_t f) -> uint32_t {  // the round at f's candidate; asks for the one after
        const uint32_t s = s_next;
        if (f + 32 + lane < len) s_next = __ldg(cands + f + 32 + lane);
        return s;
    };
    uint32_t f = 0;
    while (f < len && n < kPlanFlush) {
        uint32_t passed = __popc(__ballot_sync(kFull, ends <= f));  // lists of the window that end by f
        while (passed == 32) {
            window(kb + 32);
            passed = __popc(__ballot_sync(kFull, ends <= f));
        }
        const uint32_t end = min(__shfl_sync(kFull, ends, passed), len);
        if (end - f >= kOneProbe || end == len) {
            // ---- rounds of one probe
            const uint32_t k = kb + passed, r = __shfl_sync(kFull, ids, passed);
            const bool r_ok = r < I.r_n_sets;  // (the probe check reports a bad probe id)
            const uint32_t rk = r_ok ? r : 0u;
            Sector rs;
            uint32_t nr;
            if (G == 0) {
                nr = r_ok ? I.r_desc[rk].y : 0u;
            } else {
                rs = ld_sector(I.r_rec[0] + ((uint64_t)rk * kG + lane % kG) * 2);
                nr = __ldg(&I.r_rec[0][(uint64_t)rk * kG * 2].x) >> 16;
            }
            for (; f < end && (end - f >= 32 || end == len) && n < kPlanFlush; f += 32) {
                const uint32_t s = next(f);
                const bool have = r_ok && f + lane < end, ok = have && s < s_n_sets;
                if (have && !ok) atomicOr(err, ERR_CAND_ID);
                bool pass = ok && !(self_join && s == r);
                if (G == 0) {
                    if (pass && !emit_all) {
                        const uint32_t ns = I.s_desc[s].y;
                        pass = overlap_passes(I, min(nr, ns), nr, ns);
                    }
                } else {
                    const uint32_t v = bound_of_pair<kG, true>(I.s_rec[0], nullptr, ok ? s : 0u, 0u, rs, lane);
                    pass = pass && bound_passes(I, v, nr);
                }
                keep(pass, slot0 + k, s);
            }
        } else {
            // ---- a round of several probes
            if (passed && __shfl_sync(kFull, ends, 31) <= f + 31) {  // the window may end before the round does
                window(kb + passed);
                passed = 0;
            }
            const uint32_t my = f + lane;
            const uint32_t rel = ends - f;  // (ends <= f wraps)
            const bool in_round = ends > f && rel < 32;
            const uint32_t starts = __reduce_or_sync(kFull, in_round ? 1u << rel : 0u);
            const uint32_t lists = __popc(__ballot_sync(kFull, in_round));
            uint32_t k, r;
            if (__popc(starts) == lists && passed + lists < 32) {  // no empty lists, and the window covers the round
                const uint32_t at = passed + __popc(starts & ((2u << lane) - 1u));
                k = kb + at;
                r = __shfl_sync(kFull, ids, at);
            } else {
                k = kb;
                for (uint32_t kw = kb, w = ends;;) {
                    uint32_t lo = 0;  // lists of window kw that end by my
#pragma unroll
                    for (int step = 16; step >= 1; step >>= 1) {
                        const uint32_t v = __shfl_sync(kFull, w, lo + step - 1);
                        if (v <= my) lo += step;
                    }
                    const uint32_t v = __shfl_sync(kFull, w, 31);
                    if (lo == 31 && v <= my) lo = 32;
                    if (k == kw) k = kw + lo;
                    kw += 32;
                    if (!__any_sync(kFull, my < len && k == kw)) break;  // no lane is past this window
                    w = list_end(kw);
                }
                r = k < I.n_probes ? __ldg(I.probe_ids + k) : 0xFFFFFFFFu;
            }
            const uint32_t s = next(f);
            const bool have = r < I.r_n_sets && my < len, ok = have && s < s_n_sets;
            if (have && !ok) atomicOr(err, ERR_CAND_ID);
            bool pass = ok && !(self_join && s == r);
            if (G == 0) {
                if (pass && !emit_all) {
                    const uint32_t nr = I.r_desc[r].y, ns = I.s_desc[s].y;
                    pass = overlap_passes(I, min(nr, ns), nr, ns);
                }
            } else {
                const uint32_t rk = r < I.r_n_sets ? r : 0u;
                uint32_t r_head = G > 1 ? __ldg(&I.r_rec[0][(uint64_t)rk * kG * 2].x) : 0u;
                const uint32_t v =
                    bound_of_pair<kG, false>(I.s_rec[0], I.r_rec[0], ok ? s : 0u, rk, Sector(), lane, &r_head);
                pass = pass && bound_passes(I, v, r_head >> 16);
            }
            keep(pass, slot0 + k, s);
            f += 32;
        }
    }
    *n_out = n;
    return f0 + min(f, len);
}

// Instance owning unit g of a partition whose first units are the instances'
// `base` fields: the last one whose base is <= g.
template <class T>
__device__ __forceinline__ uint32_t owner(const Instance* table, uint32_t n_inst, T Instance::*base, T g) {
    uint32_t lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (table[mid].*base <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace

// -------------------------------------------------------------------------
// Every probe's offsets and id are checked once (tiles of 32 probes, a warp
// each); the candidates of every instance are cut into chunks of a.chunk,
// a warp each, so the work is even whatever the probes' list lengths.
// -------------------------------------------------------------------------
__global__ void __launch_bounds__(kPlanThreads, kPlanCtas) plan_kernel(const __grid_constant__ VerifyArgs a) {
    __shared__ uint2 s_buf[kPlanWarps][kPlanBuf];
    __shared__ PlanInst s_inst[kPlanWarps];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    if (blockIdx.x == 0) {
        if (!a.table && threadIdx.x == 0) a.table_out[0] = a.single;
        for (uint32_t i = threadIdx.x; i < a.n_inst; i += blockDim.x)
            *(a.table ? a.table[i].count : a.single.count) = 0ull;
    }
    const uint32_t n_warps = gridDim.x * kPlanWarps;
    const uint32_t gwarp = blockIdx.x * kPlanWarps + warp;
    uint32_t held = 0xFFFFFFFFu;  // instance whose fields are in s_inst
    const PlanInst& I = s_inst[warp];
    for (uint64_t c = gwarp; c < a.n_chunks; c += n_warps) {
        const uint32_t inst = a.table ? owner(a.table, a.n_inst, &Instance::chunk_base, c) : 0u;
        if (inst != held) {
            __syncwarp();
            if (lane == 0) s_inst[warp] = plan_inst(a.table ? a.table[inst] : a.single);
            __syncwarp();
            held = inst;
        }
        uint64_t f = (c - I.chunk_base) * a.chunk;
        const uint64_t f1 = min(f + a.chunk, I.n_cands);
        if (I.n_probes == 0) continue;
        while (f < f1) {
            uint32_t n = 0;
            switch (I.rec_sectors[0]) {
                case 1: f = filter_chunk<1>(I, f, f1, s_buf[warp], &n, &a.ctr->err, lane); break;
                case 2: f = filter_chunk<2>(I, f, f1, s_buf[warp], &n, &a.ctr->err, lane); break;
                case 4: f = filter_chunk<4>(I, f, f1, s_buf[warp], &n, &a.ctr->err, lane); break;
                case 8: f = filter_chunk<8>(I, f, f1, s_buf[warp], &n, &a.ctr->err, lane); break;
                default: f = filter_chunk<0>(I, f, f1, s_buf[warp], &n, &a.ctr->err, lane); break;
            }
            __syncwarp();
            if (n) flush_survivors(a, I, inst, s_buf[warp], n, lane);
        }
    }
    for (uint32_t g = n_warps - 1 - gwarp; g < a.n_tiles; g += n_warps) {
        const uint32_t inst = a.table ? owner(a.table, a.n_inst, &Instance::tile_base, g) : 0u;
        const PlanInst I = plan_inst(a.table ? a.table[inst] : a.single);
        const uint32_t k = 32u * (g - I.tile_base) + (uint32_t)lane;
        if (k < I.n_probes) {
            const uint64_t c0 = I.cand_offsets[k], c1 = I.cand_offsets[k + 1];
            if ((k == 0 && c0 != 0) || (k + 1 == I.n_probes && c1 != I.n_cands) || c1 < c0 || c1 > I.n_cands)
                atomicOr(&a.ctr->err, ERR_OFFSETS);
            else if (c1 > c0 && I.probe_ids[k] >= I.r_n_sets)
                atomicOr(&a.ctr->err, ERR_PROBE_ID);
        }
    }
}

cudaError_t launch_plan(const VerifyArgs& a, cudaStream_t st, int num_sms) {
    static int ctas_per_sm = 0;  // resident CTAs per SM (same value from every thread)
    if (ctas_per_sm == 0) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, plan_kernel, kPlanThreads, 0) != cudaSuccess || n < 1) n = 4;
        ctas_per_sm = n;
    }
    // at most one wave; the kernel also runs for empty batches, to clear the instances' counts
    const uint64_t units = a.n_chunks > a.n_tiles ? a.n_chunks : a.n_tiles;
    uint64_t blocks = (units + kPlanWarps - 1) / kPlanWarps;
    const uint64_t most = (uint64_t)num_sms * (uint64_t)ctas_per_sm;
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    plan_kernel<<<(unsigned)blocks, kPlanThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ssj
