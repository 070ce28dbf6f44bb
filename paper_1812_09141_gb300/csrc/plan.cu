// Plan kernel: checks a launch's grouped candidate lists and drops the pairs
// that their sets' signatures prove dissimilar (signature.cuh); what is left
// is queued for the verify kernel.
//
// What bounds it: the records gathered from L2 (32 to 256 bytes a candidate,
// by the collections' set sizes, instead of the tokens the merge would read:
// 4 bytes each, of both sets, up to the positional filter's stop).  On long
// sets their loads take 75% of the L1 data pipe's wavefronts and half of a
// warp's waiting is for them; the issue slots are busy 58% of the time with
// counting common bits (about three instructions per four bytes), L2 40%.
// Verification of 9.2e7 candidates of long sets (about 300 tokens, t = 0.6)
// took 5.2 ms when every candidate was walked against a bitmap of its probe;
// the test takes 0.95 ms (64 bytes per candidate, 6e9 bytes from L2) and
// leaves 50 us of verification.  On 5.7e6 candidates of short sets (about 20
// tokens) 48 us, leaving 10 us, instead of 195 us of merging.
#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

#include "checked.cuh"
#include "signature.cuh"
#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr int kPlanThreads = 256;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr uint32_t kOneProbe = 64;              // candidates of a list worth rounds of their own (32: the same)
constexpr uint32_t kWalkWindows = 4;            // windows that a round of several probes walks before it searches
// CTAs per SM the registers are budgeted for (64 each).  With 3 the long sets took 1.09 ms instead of
// 1.00; with 5 the spills cost more than the warps gain (1.20).  Asking for the next round's records
// before these are counted cost more registers than it hid latency (1.16 ms with 3 CTAs); more
// candidate ids asked for ahead changed nothing (2 rounds) or cost registers (4: 1.02 ms).
constexpr int kPlanCtas = 4;

// Largest k of [lo, hi) with offs[k] <= f (lo < hi; lo, if offs[lo] is beyond
// f), by the whole warp: each step narrows the range of candidate answers
// 32-fold with one load per lane.  (Offsets that are not nondecreasing give
// some k of the range.)
__device__ __forceinline__ uint32_t find_probe(const uint64_t* offs, uint32_t lo, uint32_t hi, uint64_t f, uint32_t* err,
                                               int lane) {
    const uint32_t n = hi;
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32;
        const uint64_t at = (uint64_t)lo + (uint64_t)step * lane;
        const bool le = lane == 0 || (at < hi && ld_at(offs, at, n, err) <= f);
        const uint32_t m = __ballot_sync(kFull, le);
        const uint32_t last = 31 - __clz(m);
        const uint64_t end = (uint64_t)lo + (uint64_t)step * (last + 1);
        lo += step * last;
        if (end < hi) hi = (uint32_t)end;
    }
    return lo;
}

// The same by one lane for its own f, in steps that double and then a binary
// search (it is near lo more often than not).
__device__ __forceinline__ uint32_t find_probe_lane(const uint64_t* offs, uint32_t lo, uint32_t hi, uint64_t f,
                                                    uint32_t* err) {
    const uint32_t n = hi;
    uint32_t step = 32;
    while (step < hi - lo && ld_at(offs, lo + step, n, err) <= f) {
        lo += step;
        step = min(2 * step, 1u << 30);
    }
    hi = min(hi - lo, step) + lo;
    while (hi - lo > 1) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (ld_at(offs, mid, n, err) <= f) lo = mid; else hi = mid;
    }
    return lo;
}

// Candidates [f0, f1) of an instance, by one warp, 32 at a time; the pairs
// left go to buf, *n of them, and the position up to which candidates are done
// is returned: f1, or less when the buffer is full.  (The caller queues them:
// a call in here would cost the loops their registers.)  The warp holds a
// window of 32 list ends; rounds within one probe's list keep the probe's
// record in registers, in the others each lane finds its candidate's probe in
// the window and reads its record.  G: sectors per record of the
// first level, 0 without signatures (the length filter alone).
//
// The next list is mostly in the window or the one after it.  Beyond those the
// warp searches for it: a batch may list any number of probes without
// candidates, and walked window by window 1e7 probes with 1,000 candidates took
// 6.1 ms a call (now 0.07).
template <int G>
__device__ __forceinline__ uint64_t filter_chunk(const PlanInst& I, uint64_t f0, uint64_t f1, uint2* buf,
                                                 uint32_t* n_out, uint32_t* err, int lane) {
    constexpr int kG = G > 0 ? G : 1;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool emit_all = (I.flags & VF_EMIT_ALL) != 0, self_join = (I.flags & VF_SELF_JOIN) != 0;
    const uint32_t len = (uint32_t)(f1 - f0), slot0 = 32u * I.tile_base, s_n_sets = I.s_n_sets;
    const uint32_t* cands = I.cand_ids + f0;
    auto cand = [&](uint32_t at) -> uint32_t { return ld_at(cands, at, I.n_cands - f0, err); };
    // lane l of the window holds probe kb + l: its id, and the end of its list relative to f0 (saturated;
    // the last probe's list ends the batch)
    uint32_t kb = find_probe(I.cand_offsets, 0, I.n_probes, f0, err, lane), ends, ids;
    auto list_end = [&](uint32_t k) -> uint32_t {
        const uint64_t at = (uint64_t)k + 1 + lane;
        if (at >= I.n_probes) return 0xFFFFFFFFu;
        const uint64_t v = ld_at(I.cand_offsets, at, I.n_probes + 1ull, err);
        return v <= f0 ? 0u : (uint32_t)min(v - f0, (uint64_t)0xFFFFFFFFu);
    };
    auto window = [&](uint32_t k) {
        kb = k;
        ends = list_end(k);
        ids = (uint64_t)k + lane < I.n_probes ? ld_at(I.probe_ids, (uint64_t)k + lane, I.n_probes, err) : 0xFFFFFFFFu;
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
    uint32_t s_next = (uint32_t)lane < len ? cand(lane) : 0u;  // the lane's candidate of the next round
    auto next = [&](uint32_t f) -> uint32_t {  // the round at f's candidate; asks for the one after
        const uint32_t s = s_next;
        if (f + 32 + lane < len) s_next = cand(f + 32 + lane);
        return s;
    };
    const Threshold th = threshold(I);
    bool bad = false;  // a candidate id is out of range
    uint32_t f = 0;
    while (f < len && n < kPlanFlush) {
        // Lists of the window before the first that ends after f.  (Not the number that end by f: with
        // offsets that are not nondecreasing, which the probe check reports, the list at that number may
        // end before f, and no round would be made.)
        uint32_t m = __ballot_sync(kFull, ends > f);
        for (bool near = true; m == 0; near = false) {  // (kb + 32 < n_probes: the last list's end is beyond every f)
            window(near ? kb + 32 : find_probe(I.cand_offsets, kb + 32, I.n_probes, f0 + f, err, lane));
            m = __ballot_sync(kFull, ends > f);
        }
        const uint32_t passed0 = __ffs(m) - 1;
        const uint32_t end = min(__shfl_sync(kFull, ends, passed0), len);
        if (end - f >= kOneProbe || end == len) {
            // ---- rounds of one probe
            const uint32_t k = kb + passed0, r = __shfl_sync(kFull, ids, passed0);
            const bool r_ok = r < I.r_n_sets;  // (the probe check reports a bad probe id)
            const uint32_t rk = r_ok ? r : 0u;
            Sector rs;
            uint32_t nr;
            if (G == 0) {
                nr = r_ok ? ld_at(I.r_desc, rk, I.r_n_sets, err).y : 0u;
            } else {
                rs = ld_sector(I.r_rec[0], (uint64_t)rk * kG + lane % kG, (uint64_t)I.r_n_sets * kG, err);
                nr = ld_header(I.r_rec[0], rk, kG, I.r_n_sets, err) >> 16;
            }
            for (; f < end && (end - f >= 32 || end == len) && n < kPlanFlush; f += 32) {
                const uint32_t s = next(f);
                const bool have = r_ok && f + lane < end, ok = have && s < s_n_sets;
                bad = bad || (have && !ok);
                bool pass = ok && !(self_join && s == r);
                if (G == 0) {
                    if (pass && !emit_all) {
                        const uint32_t ns = ld_at(I.s_desc, s, s_n_sets, err).y;
                        pass = overlap_passes(I, min(nr, ns), nr, ns);
                    }
                } else {
                    const uint32_t v = bound_of_pair<kG, true>(I.s_rec[0], nullptr, ok ? s : 0u, 0u, rs, lane, s_n_sets, 0u, err);
                    pass = pass && bound_passes(I, th, v, nr);
                }
                keep(pass, slot0 + k, s);
            }
        } else {
            // ---- a round of several probes
            uint32_t passed = passed0;
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
                for (uint32_t kw = kb, w = ends, windows = 1;; ++windows) {
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
                    const bool beyond = my < len && k == kw;
                    if (!__any_sync(kFull, beyond)) break;  // no lane is past this window
                    if (windows == kWalkWindows) {
                        if (beyond) k = find_probe_lane(I.cand_offsets, kw, I.n_probes, f0 + my, err);
                        if (f + 32 < len) window(__shfl_sync(kFull, k, 31));
                        break;
                    }
                    w = list_end(kw);
                }
                r = k < I.n_probes ? ld_at(I.probe_ids, k, I.n_probes, err) : 0xFFFFFFFFu;
            }
            const uint32_t s = next(f);
            const bool have = r < I.r_n_sets && my < len, ok = have && s < s_n_sets;
            bad = bad || (have && !ok);
            bool pass = ok && !(self_join && s == r);
            if (G == 0) {
                if (pass && !emit_all) {
                    const uint32_t nr = ld_at(I.r_desc, r, I.r_n_sets, err).y, ns = ld_at(I.s_desc, s, s_n_sets, err).y;
                    pass = overlap_passes(I, min(nr, ns), nr, ns);
                }
            } else {
                const uint32_t rk = r < I.r_n_sets ? r : 0u;
                uint32_t r_head = G > 1 ? ld_header(I.r_rec[0], rk, kG, I.r_n_sets, err) : 0u;
                const uint32_t v = bound_of_pair<kG, false>(I.s_rec[0], I.r_rec[0], ok ? s : 0u, rk, Sector(), lane, s_n_sets,
                                                            I.r_n_sets, err, &r_head);
                pass = pass && bound_passes(I, th, v, r_head >> 16);
            }
            keep(pass, slot0 + k, s);
            f += 32;
        }
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(err, ERR_CAND_ID);
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
    if (blockIdx.x == 0 && a.chunk_begin == 0) {
        if (!a.table && threadIdx.x == 0) a.table_out[0] = a.single;
        for (uint32_t i = threadIdx.x; i < a.n_inst; i += blockDim.x)
            *(a.table ? a.table[i].count : a.single.count) = 0ull;
    }
    const uint32_t n_warps = gridDim.x * kPlanWarps;
    const uint32_t gwarp = blockIdx.x * kPlanWarps + warp;
    uint32_t held = 0xFFFFFFFFu;  // instance whose fields are in s_inst
    const PlanInst& I = s_inst[warp];
    for (uint64_t c = a.chunk_begin + gwarp; c < a.n_chunks; c += n_warps) {
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
    if (a.chunk_begin) return;  // (the first piece checks the probes)
    for (uint32_t g = n_warps - 1 - gwarp; g < a.n_tiles; g += n_warps) {
        const uint32_t inst = a.table ? owner(a.table, a.n_inst, &Instance::tile_base, g) : 0u;
        const PlanInst I = plan_inst(a.table ? a.table[inst] : a.single);
        const uint32_t k = 32u * (g - I.tile_base) + (uint32_t)lane;
        if (k < I.n_probes) {
            const uint64_t n_offs = I.n_probes + 1ull;
            const uint64_t c0 = ld_at(I.cand_offsets, k, n_offs, &a.ctr->err), c1 = ld_at(I.cand_offsets, k + 1, n_offs, &a.ctr->err);
            if ((k == 0 && c0 != 0) || (k + 1 == I.n_probes && c1 != I.n_cands) || c1 < c0 || c1 > I.n_cands)
                atomicOr(&a.ctr->err, ERR_OFFSETS);
            else if (c1 > c0 && ld_at(I.probe_ids, k, I.n_probes, &a.ctr->err) >= I.r_n_sets)
                atomicOr(&a.ctr->err, ERR_PROBE_ID);
        }
    }
}

cudaError_t launch_plan(const VerifyArgs& a, cudaStream_t st, int num_sms) {
    // resident CTAs per SM: the same value from every thread that submits (all devices are alike)
    static std::atomic<int> cached{0};
    int ctas_per_sm = cached.load(std::memory_order_relaxed);
    if (ctas_per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas_per_sm, plan_kernel, kPlanThreads, 0) != cudaSuccess ||
            ctas_per_sm < 1)
            ctas_per_sm = kPlanCtas;
        cached.store(ctas_per_sm, std::memory_order_relaxed);
    }
    // at most one wave; the kernel also runs for empty batches, to clear the instances' counts
    const uint64_t chunks = a.n_chunks - a.chunk_begin, tiles = a.chunk_begin ? 0 : a.n_tiles;
    const uint64_t units = chunks > tiles ? chunks : tiles;
    uint64_t blocks = (units + kPlanWarps - 1) / kPlanWarps;
    const uint64_t most = (uint64_t)num_sms * (uint64_t)ctas_per_sm;
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    plan_kernel<<<(unsigned)blocks, kPlanThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace ssj
