// The signature test of candidate pairs and the queueing of the pairs that it
// leaves, shared by the plan kernel (plan.cu) and the join kernel
// (candgen.cu).
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
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "arith.h"
#include "checked.cuh"
#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kPlanBuf = kPlanFlush + 32;  // pairs buffered per warp
constexpr int kSectors = 2;                     // 32-byte record loads in flight per lane, at most (4: 2% slower)

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

// Sector i of an array of n.
__device__ __forceinline__ Sector ld_sector(const uint4* rec, uint64_t i, uint64_t n, uint32_t* err) {
    Sector x = {};
    if (!in_bounds(i, n, err)) return x;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3]), "=r"(x.w[4]), "=r"(x.w[5]), "=r"(x.w[6]), "=r"(x.w[7])
        : "l"(rec + 2 * i));
    return x;
}

// Header of set r's record, of n sets' records of `sectors` each.
__device__ __forceinline__ uint32_t ld_header(const uint4* rec, uint32_t r, uint32_t sectors, uint32_t n, uint32_t* err) {
    return ld_at(reinterpret_cast<const uint32_t*>(rec), (uint64_t)r * sectors * 8, (uint64_t)n * sectors * 8, err);
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
// s_n, r_n: sets of both collections (bounds of the checked build).
template <int G, bool kSame>
__device__ __forceinline__ uint32_t bound_of_pair(const uint4* s_rec, const uint4* r_rec, uint32_t s, uint32_t r,
                                                  const Sector& rs, int lane, uint32_t s_n, uint32_t r_n, uint32_t* err,
                                                  uint32_t* r_head = nullptr) {
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
            x[i] = ld_sector(s_rec, (uint64_t)sj * G + sub, (uint64_t)s_n * G, err);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            uint32_t hr;
            if (kSame) {
                part[b + i] = common_bits(x[i], rs, first);
                hr = rs.w[0];
            } else {
                const uint32_t rj = G == 1 ? r : __shfl_sync(kFull, r, b + i, G);
                const Sector y = ld_sector(r_rec, (uint64_t)rj * G + sub, (uint64_t)r_n * G, err);
                part[b + i] = common_bits(x[i], y, first);
                hr = y.w[0];
                if (G == 1) *r_head = hr;
            }
            if (G == 1 || sub == 0) part[b + i] += (x[i].w[0] & 0xFFFF0000u) + min(x[i].w[0] & 0xFFFFu, hr & 0xFFFFu);
        }
    }
    return sum_of_group<G>(part, sub);
}

// The similarity test of an instance as ub * a >= c * (|r| + |s|) + k in 32
// bits, if it has that form: Jaccard and Dice while p and the divisor are
// small (sizes in a header are below 2^16), and the plain overlap.  (The
// branches on the function and 64-bit products cost the plan kernel a tenth of
// its time: 1.10 against 1.00 ms on 9.2e7 candidates.)
struct Threshold {
    uint32_t a, c, k;
    bool linear;
};

__device__ __forceinline__ Threshold threshold(const PlanInst& I) {
    Threshold t;
    t.linear = I.sim == SIM_OVERLAP || (I.sim != SIM_COSINE && I.den <= 32767u);  // 32767 * 131,070 < 2^32
    t.a = I.sim == SIM_OVERLAP ? 1u : I.den;
    t.c = I.sim == SIM_OVERLAP ? 0u : I.p;
    t.k = I.sim == SIM_OVERLAP ? I.den : 0u;
    return t;
}

// The signature test of a pair from its bound_of_pair value and |r| (65535 in
// a header: 65535 tokens or more, not tested).  In the linear form an empty s
// fails by itself (its bound is 0) unless r is empty too.
__device__ __forceinline__ bool bound_passes(const PlanInst& I, const Threshold& t, uint32_t v, uint32_t nr) {
    const uint32_t ns = v >> 16, ub = v & 0xFFFFu;
    if (t.linear) return (nr != 0 && ub * t.a >= t.c * (nr + ns) + t.k) || ns == 0xFFFFu || nr == 0xFFFFu;
    return ns == 0xFFFFu || nr == 0xFFFFu || overlap_passes(I, ub, nr, ns);
}

// Second level: the n buffered pairs tested with the long records; the ones
// left stay in the buffer, in order.  Returns their number.
template <int G>
__device__ __noinline__ uint32_t second_level(const PlanInst& I, uint2* buf, uint32_t n, uint32_t* err, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    const Threshold th = threshold(I);
    uint32_t left = 0;
    for (uint32_t t = 0; t < n; t += 32) {
        const bool have = t + lane < n;
        const uint2 e = buf[have ? t + lane : t];
        const uint32_t r = ld_at(I.probe_ids, e.x - 32u * I.tile_base, I.n_probes, err);
        const uint32_t r_head = ld_header(I.r_rec[1], r, G, I.r_n_sets, err);
        const uint32_t v = bound_of_pair<G, false>(I.s_rec[1], I.r_rec[1], e.y, r, Sector(), lane, I.s_n_sets, I.r_n_sets, err);
        const bool pass = have && bound_passes(I, th, v, r_head >> 16);
        const uint32_t m = __ballot_sync(kFull, pass);  // (every lane has read its entry)
        if (pass && in_bounds(left + __popc(m & lt_mask), n, err)) buf[left + __popc(m & lt_mask)] = e;
        left += __popc(m);
        __syncwarp();
    }
    return left;
}

// Granularity of a run, n pairs left of a probe with |r| = nr: 0 thread per
// pair, 1 warp per pair, 2 block per pair, 3 lane per pair with r in the
// warp's shared memory (Alternative B; needs r to fit and enough candidates
// to occupy the lanes), 4 an index item (many candidates, when the launch's
// token values fit the probe bitmap).
//
// A list is cut into runs where a warp's candidates or its buffer end, so its
// last run is often much shorter than the list.  Beyond the thread bin an index
// item is the better choice from about 60 pairs on (300 tokens; 18 us an item
// and 0.14 a pair of a CTA's time, one lane per pair 0.45) or 20 (1,500 tokens;
// 90 and 0.6, one block per pair 5.8), within it from about 270 (60 tokens): a
// quarter of the threshold for the former.  Lists of 1,000 pairs of 1,500 tokens
// that all pass took 4.7 ms with one threshold for both, now 2.8.
// (The line holds with the largest bitmaps: 780,000 token values, lists of 130
// pairs of 300 tokens 1.29 ms, 1.48 with the full threshold.)
__device__ __forceinline__ uint32_t probe_bin(const VerifyArgs& a, uint32_t flags, uint32_t nr, uint32_t n) {
    const bool lane_ok = nr + 4 <= kWarpRCap;
    if (flags & VF_FORCE_INDEX) return a.index_words ? 4u : (lane_ok ? 3u : 1u);
    if (flags & VF_FORCE_BLOCK) return 2;
    if (flags & VF_FORCE_WARP) return 1;
    if (flags & VF_FORCE_THREAD) return 0;
    if (flags & VF_FORCE_LANE) return lane_ok ? 3u : 1u;
    const uint64_t key = 2ull * nr;  // |r|+|s| at |s| = |r|
    const uint32_t index_min = min(a.index_min_cands, kPlanFlush);
    if (a.index_words && index_min && n >= (key <= a.thread_max_key ? index_min : max(index_min / 4, 1u))) return 4;
    if (key <= a.thread_max_key) return 0;
    if (key <= a.lane_max_key && lane_ok && n >= kLaneMinCands) return 3;
    return key <= a.warp_max_key ? 1u : 2u;
}

// Work items of one run: n pairs of probe r from pos on in the pair list, of
// granularity bin (2 to 4), as items first, first + 1, ... of its list.
__device__ __forceinline__ uint32_t item_pairs(const VerifyArgs& a, uint32_t bin) {
    return bin == 3 ? a.lane_item_cands : (bin == 4 ? kPlanBuf : a.block_item_cands);  // (an index item is a run)
}
__device__ __forceinline__ void write_item(const VerifyArgs& a, uint32_t bin, uint32_t inst, uint32_t r, uint32_t n,
                                           unsigned long long pos, unsigned long long first, uint32_t it) {
    const uint32_t per = item_pairs(a, bin);
    if (first + it >= (bin == 3 ? a.warp_item_cap : a.block_item_cap)) {
        atomicOr(&a.ctr->err, ERR_GUARD);
        return;
    }
    WorkItem wi;
    wi.r = r;
    wi.n = min(per, n - it * per);
    wi.c0 = pos + (uint64_t)it * per;
    wi.inst = inst;
    wi.pad = bin >= 3 ? 1u : 0u;
    (bin == 3 ? a.warp_items : a.block_items)[first + it] = wi;
}

// Queue the warp's n buffered pairs (probe slot, candidate id; n > 0) in
// candidate order, a probe's pairs side by side.  Short pairs go to the front
// of the pair list, the others to its back; lane, block and index items refer
// to a run of one probe's pairs, and those pairs are marked (kInItem) so that
// the warp-per-pair phase passes over them.
//
// Bound by its instructions where many pairs are left, so a buffer of one run
// (long lists) is copied straight out, and of several runs the ends come from
// the windows' head masks and each entry's granularity is looked up once and
// kept.  (With two binary searches and two dependent loads per entry, twice, the
// plan kernel took 260 us where 1e7 pairs of lists of 10,000 all pass, now 102,
// and 178 on 5.6e6 pairs in lists of 30, all kept, now 117.)
__device__ __noinline__ void queue_pairs(const VerifyArgs& a, const PlanInst& I, uint32_t inst, const uint2* buf,
                                         uint32_t n, int lane) {
    static_assert(kPlanBuf <= 16 * 32, "granularities and head masks of 16 windows");
    const unsigned lt_mask = (1u << lane) - 1u;
    uint32_t* err = &a.ctr->err;
    auto probe_of = [&](uint32_t i) -> uint32_t { return ld_at(I.probe_ids, buf[i].x - 32u * I.tile_base, I.n_probes, err); };
    auto size_of = [&](uint32_t r) -> uint32_t { return ld_at(I.r_desc, r, I.r_n_sets, err).y; };
    // lane 0 takes room for ns short and nl long pairs (nw of them without an item); false if there is none
    unsigned long long base_s = 0, base_l = 0;
    auto reserve = [&](uint32_t ns, uint32_t nl, uint32_t nw) -> bool {
        if (lane == 0) {
            if (ns) base_s = atomicAdd(&a.ctr->thread_pairs, (unsigned long long)ns);
            if (nl) base_l = atomicAdd(&a.ctr->long_pairs, (unsigned long long)nl);
            if (nw) atomicAdd(&a.ctr->warp_pairs, (unsigned long long)nw);
        }
        base_s = __shfl_sync(kFull, base_s, 0);
        base_l = __shfl_sync(kFull, base_l, 0);
        // every candidate is queued at most once, so the lists never meet
        if (base_s + ns <= a.pair_cap && base_l + nl <= a.pair_cap) return true;
        if (lane == 0) atomicOr(err, ERR_GUARD);
        return false;
    };
    auto write_pair = [&](unsigned long long pos, uint2 e, uint32_t bin) {
        if (!in_bounds(pos, a.pair_cap, err)) return;
        PairRef pr;
        pr.k = e.x;
        pr.s = e.y | (bin >= 2 ? kInItem : 0u);
        a.pairs[pos] = pr;
    };
    if (buf[0].x == buf[n - 1].x) {  // one run (slots ascend)
        const uint32_t r = probe_of(0), bin = probe_bin(a, I.flags, size_of(r), n);
        if (!reserve(bin ? 0u : n, bin ? n : 0u, bin == 1 ? n : 0u)) return;
        const unsigned long long pos = bin ? a.pair_cap - base_l - n : base_s;
        for (uint32_t i = lane; i < n; i += 32) write_pair(pos + i, buf[i], bin);
        if (bin >= 2) {
            const uint32_t items = (n + item_pairs(a, bin) - 1) / item_pairs(a, bin);
            unsigned long long first = 0;
            if (lane == 0) first = atomicAdd(bin == 3 ? &a.ctr->warp_items : &a.ctr->block_items, (unsigned long long)items);
            first = __shfl_sync(kFull, first, 0);
            for (uint32_t it = lane; it < items; it += 32) write_item(a, bin, inst, r, n, pos, first, it);
        }
        __syncwarp();
        return;
    }
    uint32_t heads = 0;  // lane w: the entries of window w (32 entries) that begin a run
    for (uint32_t w = 0; 32 * w < n; ++w) {
        const uint32_t i = 32 * w + lane;
        const uint32_t m = __ballot_sync(kFull, i < n && (i == 0 || buf[i - 1].x != buf[i].x));
        if (lane == (int)w) heads = m;
    }
    const uint32_t headed = __ballot_sync(kFull, heads != 0);  // windows with heads (the first is one)
    // the run [h, e) of entry 32 * w + lane
    auto run_of = [&](uint32_t w, uint32_t* h, uint32_t* e) {
        const uint32_t m = __shfl_sync(kFull, heads, w);
        const uint32_t earlier = (headed & ((1u << w) - 1u)) | 1u, later = headed & (kFull << w << 1);
        const uint32_t we = 31 - __clz(earlier), wl = later ? __ffs(later) - 1 : 0u;
        const uint32_t me = __shfl_sync(kFull, heads, we), ml = __shfl_sync(kFull, heads, wl);
        const uint32_t upto = m & (lt_mask | 1u << lane), past = m & (kFull << lane << 1);
        *h = upto ? 32 * w + 31 - __clz(upto) : 32 * we + 31 - __clz(me);
        *e = past ? 32 * w + __ffs(past) - 1 : (later ? 32 * wl + __ffs(ml) - 1 : n);
    };
    uint64_t bins = 0;  // 3 bits a window
    uint32_t n_long = 0, n_warp = 0;
#pragma unroll 2
    for (uint32_t w = 0; 32 * w < n; ++w) {
        const uint32_t i = 32 * w + lane;
        uint32_t h, e, bin = 0;
        run_of(w, &h, &e);
        if (i < n) bin = probe_bin(a, I.flags, size_of(probe_of(i)), e - h);
        bins |= (uint64_t)bin << (3 * w);
        n_long += __popc(__ballot_sync(kFull, bin != 0));
        n_warp += __popc(__ballot_sync(kFull, bin == 1));
    }
    if (!reserve(n - n_long, n_long, n_warp)) return;
    unsigned long long at_s = base_s, at_l = a.pair_cap - base_l - n_long;
    for (uint32_t w = 0; 32 * w < n; ++w) {
        const uint32_t i = 32 * w + lane;
        uint32_t h, e;
        run_of(w, &h, &e);
        const uint32_t bin = i < n ? (uint32_t)(bins >> (3 * w)) & 7u : 5u;
        const uint32_t ms = __ballot_sync(kFull, bin == 0), ml = __ballot_sync(kFull, bin >= 1 && bin <= 4);
        const unsigned long long pos = bin == 0 ? at_s + __popc(ms & lt_mask) : at_l + __popc(ml & lt_mask);
        at_s += __popc(ms);
        at_l += __popc(ml);
        if (bin <= 4) write_pair(pos, buf[i], bin);
        // items, by the first entry of a run
        const uint32_t items = i < n && i == h && bin >= 2 ? (e - h + item_pairs(a, bin) - 1) / item_pairs(a, bin) : 0u;
        if (__any_sync(kFull, items != 0)) {
            const uint32_t r = items ? probe_of(i) : 0u;
            const uint32_t wn = bin == 3 ? items : 0u, bn = bin == 3 ? 0u : items;
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
            for (uint32_t it = 0; it < items; ++it) write_item(a, bin, inst, r, e - h, pos, bin == 3 ? wbase : bbase, it);
        }
    }
    __syncwarp();
}

// Queue what the second level leaves of the n buffered pairs.  Mostly that is
// nothing, so only the queueing is a call (9.2e7 candidates of long sets: plan
// kernel 961 us; 991 with a function around both, which saves its registers
// every time).
__device__ __forceinline__ void flush_survivors(const VerifyArgs& a, const PlanInst& I, uint32_t inst, uint2* buf,
                                                uint32_t n, int lane) {
    switch (I.rec_sectors[1]) {
        case 2: n = second_level<2>(I, buf, n, &a.ctr->err, lane); break;
        case 4: n = second_level<4>(I, buf, n, &a.ctr->err, lane); break;
        case 8: n = second_level<8>(I, buf, n, &a.ctr->err, lane); break;
        default: break;
    }
    if (n) queue_pairs(a, I, inst, buf, n, lane);
}

}  // namespace

}  // namespace ssj
