// Self-join on the device: the prefix filter and inverted-index probing of
// algorithm ALL (Sections 2.2.3, 2.2.4, 3.1), which the paper leaves on the
// CPU and names as future work (Section 6), and the signature test of every
// candidate as it is found; the pairs left go straight to the verify
// kernel's lists.
//
// Steps, on one stream:
//   1. order the sets by size (counting sort; ties in any order: the set of
//      unordered candidate pairs does not depend on it);
//   2. index every set's prefix: per token and range of positions (cell), the
//      entries (position in that order, set id; for the positional bound also the token's position in
//      the set and the set's size), by a count / scan / scatter over the
//      prefix tokens;
//   3. one warp per probe walks its prefix tokens' entries, keeps those of
//      earlier sets that pass the length filter (positions [lo, its own), and
//      optionally the positional bound of the matching token, PPJoin-style),
//      drops repeated ones by a set in shared memory, and tests the others'
//      short records 32 at a time;
//   4. a warp per run of pairs left tests their long records and queues what
//      remains for the verify kernel (signature.cuh).
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

#include "arith.h"
#include "signature.cuh"
#include "ssj_internal.h"

namespace ssj {
namespace {

constexpr int kJoinWarps = 8;             // warps per CTA of the join kernel
constexpr uint32_t kSeenWords = 1024;    // a warp's set of candidates seen: a bitmap of 32,768 positions, or a
constexpr uint32_t kSeenBits = 32 * kSeenWords;  // hash set of up to half as many as it has words
constexpr uint32_t kJoinFlush = kJoinRun - 32;  // pairs left that a warp hands over at once (room for 32 more)
constexpr uint64_t kLongList = 1u << 26;  // 32 lists below this add up in 32 bits
constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr uint32_t kFree = 0xFFFFFFFFu;

struct Params {
    const uint4* toks4;
    const uint2* desc;
    uint32_t cells_log2, cell_shift;  // a token's list is cut into 1 << cells_log2 cells, by position >> cell_shift
    uint32_t n;
    uint32_t sim, p, q;     // sim: SIM_*; t = p/q
    uint32_t positional;    // apply the positional bound at the matching token
};

__device__ __forceinline__ const uint32_t* set_tokens(const Params& P, uint2 d) {
    return reinterpret_cast<const uint32_t*>(P.toks4 + d.x);
}

// Least overlap a set of size len shares with any partner that can reach t
// (Jaccard t|x|, Dice t|x|/(2-t), Cosine t^2|x|, plain overlap t, rounded
// up); also the smallest partner size the length filter admits.
__device__ __forceinline__ uint64_t min_overlap(const Params& P, uint32_t len) {
    const uint64_t p = P.p, q = P.q;
    switch (P.sim) {
        case SIM_DICE: return ((uint64_t)len * p + (2 * q - p) - 1) / (2 * q - p);
        case SIM_COSINE: {  // p^2 len needs 128 bits
            const unsigned __int128 d = (unsigned __int128)q * q;
            return (uint64_t)(((unsigned __int128)p * p * len + d - 1) / d);
        }
        case SIM_OVERLAP: return (p + q - 1) / q;
        default: return ((uint64_t)len * p + q - 1) / q;
    }
}

// Prefix of len - min_overlap + 1 tokens (none if no partner can reach t).
__device__ __forceinline__ uint32_t prefix_len(const Params& P, uint32_t len) {
    if (len == 0) return 0;
    const uint64_t need = min_overlap(P, len);
    if (need > len) return 0;
    const uint64_t pl = (uint64_t)len + 1 - need;
    return pl > len ? len : (uint32_t)pl;
}

// Equivalent overlap of a pair (for the positional bound).
__device__ __forceinline__ uint32_t pair_required(const Params& P, uint32_t nr, uint32_t ns) {
    switch (P.sim) {
        case SIM_DICE: return required_overlap_magic(nr, ns, P.p, 2 * P.q, div_magic(2ull * P.q));
        case SIM_COSINE: return required_overlap_cosine(P.p, P.q, nr, ns);
        case SIM_OVERLAP: return (uint32_t)(((uint64_t)P.p + P.q - 1) / P.q);
        default: return required_overlap_magic(nr, ns, P.p, P.p + P.q, div_magic((uint64_t)P.p + P.q));
    }
}

// Counting sort by size.  A CTA takes one run of sets and counts them in shared
// memory first, so that the global counters see one atomic per size and CTA
// (200,000 sets of about 100 sizes: 54 + 56 us with one atomic per set).
constexpr uint32_t kSizeBins = 4096;  // sizes counted in shared memory; longer sets one by one
constexpr int kSizeThreads = 256;

__global__ void __launch_bounds__(kSizeThreads) size_hist_kernel(Params P, uint32_t per_cta, uint64_t* hist) {
    __shared__ uint32_t cnt[kSizeBins];
    for (uint32_t b = threadIdx.x; b < kSizeBins; b += kSizeThreads) cnt[b] = 0;
    __syncthreads();
    const uint32_t lo = blockIdx.x * per_cta, hi = min(lo + per_cta, P.n);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kSizeThreads) {
        const uint32_t L = P.desc[i].y;
        if (L < kSizeBins) atomicAdd(cnt + L, 1u);
        else atomicAdd(reinterpret_cast<unsigned long long*>(hist + L), 1ull);
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < kSizeBins; b += kSizeThreads)
        if (cnt[b]) atomicAdd(reinterpret_cast<unsigned long long*>(hist + b), (unsigned long long)cnt[b]);
}

// cursor: the sizes' first positions; afterwards the positions after their
// last.  probes: the sets from the last position down.
__global__ void __launch_bounds__(kSizeThreads) place_kernel(Params P, uint32_t per_cta, uint64_t* cursor,
                                                             uint32_t* probes, uint32_t* rank) {
    __shared__ uint32_t cnt[kSizeBins], at[kSizeBins];
    for (uint32_t b = threadIdx.x; b < kSizeBins; b += kSizeThreads) cnt[b] = 0;
    __syncthreads();
    const uint32_t lo = blockIdx.x * per_cta, hi = min(lo + per_cta, P.n);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kSizeThreads) {
        const uint32_t L = P.desc[i].y;
        if (L < kSizeBins) atomicAdd(cnt + L, 1u);
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < kSizeBins; b += kSizeThreads)
        if (cnt[b]) at[b] = (uint32_t)atomicAdd(reinterpret_cast<unsigned long long*>(cursor + b), (unsigned long long)cnt[b]);
    __syncthreads();
    for (uint32_t i = lo + threadIdx.x; i < hi; i += kSizeThreads) {
        const uint32_t L = P.desc[i].y;
        const uint32_t pos = L < kSizeBins ? atomicAdd(at + L, 1u)
                                           : (uint32_t)atomicAdd(reinterpret_cast<unsigned long long*>(cursor + L), 1ull);
        probes[P.n - 1 - pos] = i;
        rank[i] = pos;
    }
}

// Prefix tokens of every set, by kSetLanes lanes a set (prefixes are mostly
// shorter than a warp): f(set, its size, token's position, token).
constexpr uint32_t kSetLanes = 8;
template <class F>
__device__ __forceinline__ void for_prefix_tokens(const Params& P, F&& f) {
    const uint32_t sub = threadIdx.x % kSetLanes;
    const uint32_t groups = (gridDim.x * blockDim.x) / kSetLanes;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) / kSetLanes; i < P.n; i += groups) {
        const uint2 d = P.desc[i];
        const uint32_t* t = set_tokens(P, d);
        const uint32_t pl = prefix_len(P, d.y);
        for (uint32_t a = sub; a < pl; a += kSetLanes) f(i, d.y, a, t[a]);
    }
}

// Cell of a token's index entries at a position.  A probe admits a range of
// positions only (the length filter), about a sixth of them for long sets at
// t = 0.8, so it reads the cells of that range instead of the whole list.
__device__ __forceinline__ uint64_t cell_of(const Params& P, uint32_t tok, uint32_t pos) {
    return ((uint64_t)tok << P.cells_log2) + (pos >> P.cell_shift);
}

__global__ void token_count_kernel(Params P, const uint32_t* rank, uint64_t* tcnt) {
    for_prefix_tokens(P, [&](uint32_t i, uint32_t, uint32_t, uint32_t tok) {
        atomicAdd(reinterpret_cast<unsigned long long*>(tcnt + cell_of(P, tok, rank[i])), 1ull);
    });
}

// An index entry: position and id of the set; with the positional bound also
// the token's position in the set and the set's size.
template <bool POS>
struct Entry {
    uint32_t rank, id;
};
template <>
struct Entry<true> {
    uint32_t rank, id, at, size;
};
__device__ __forceinline__ Entry<false> ld_entry(const Entry<false>* post, uint64_t e, uint64_t n, uint32_t* err) {
    const uint2 x = ld_at(reinterpret_cast<const uint2*>(post), e, n, err);
    return {x.x, x.y};
}
__device__ __forceinline__ Entry<true> ld_entry(const Entry<true>* post, uint64_t e, uint64_t n, uint32_t* err) {
    const uint4 x = ld_at(reinterpret_cast<const uint4*>(post), e, n, err);
    return {x.x, x.y, x.z, x.w};
}

// every set's prefix entries into the token lists
template <bool POS>
__global__ void postings_kernel(Params P, const uint32_t* rank, uint64_t* tcur, void* post) {
    for_prefix_tokens(P, [&](uint32_t i, uint32_t size, uint32_t a, uint32_t tok) {
        const uint32_t pos = rank[i];
        const uint64_t slot = atomicAdd(reinterpret_cast<unsigned long long*>(tcur + cell_of(P, tok, pos)), 1ull);
        if constexpr (POS) reinterpret_cast<uint4*>(post)[slot] = make_uint4(pos, i, a, size);
        else reinterpret_cast<uint2*>(post)[slot] = make_uint2(pos, i);
    });
}

// Positional bound of an index entry matched at probe token position a: at
// most min(a, j) matches before this one, one here, min(|r|-a-1, |s|-j-1)
// after.
__device__ __forceinline__ bool position_ok(const Params&, const Entry<false>&, uint32_t, uint32_t) { return true; }
__device__ __forceinline__ bool position_ok(const Params& P, const Entry<true>& e, uint32_t L, uint32_t a) {
    const uint32_t ub = min(a, e.at) + 1 + min(L - a - 1, e.size - e.at - 1);
    return ub >= pair_required(P, L, e.size);
}

// The 32-bit finaliser of MurmurHash3 (Appleby).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85ebca6bu;
    x ^= x >> 13;
    x *= 0xc2b2ae35u;
    x ^= x >> 16;
    return x;
}

struct JoinArgs {
    const uint32_t* probes;    // the sets in the order in which they probe: from the last position down
    const uint64_t* size_end;  // size -> position after its last set
    const uint64_t* toff;      // cell -> first index entry (and one past the last cell)
    const void* post;          // index entries (Entry<POS>)
    uint64_t sizes, cells, entries;  // of size_end, toff (without the closing one) and post
    uint32_t* cursor;          // next probe (from the last position down)
    uint32_t grab;             // probes per grab
    JoinQueue out;             // pairs left
};

struct JoinWarp {
    uint32_t seen[kSeenWords];
    uint2 buf[kJoinRun];
    uint2 fresh[64];  // candidates to be tested: index of the probe, set
};

// The join of the sets in size order: a warp takes a few probes at a time, the
// largest first (they have the most candidates).  The index entries of 32
// tokens are read as one list, 32 at a time.
// A candidate found through several tokens is kept once, by a bitmap over the
// positions that the length filter admits; when these are more than the
// bitmap holds, by a hash set if there are few entries, else window by window
// of positions.  G: sectors per record of the first level of the signature
// test, 0: every candidate is handed over.  POS: the positional bound.
//
// Bound by latency: a probe is a chain of dependent loads (set, size, tokens,
// list bounds, entries, records).  The sets and sizes are therefore loaded for
// all probes of a grab at once, the tokens and list bounds of the next 32
// tokens while the entries of these are read, the next entries before these
// are taken, and with one-sector records the candidates of several probes are
// tested together.
template <int G, bool POS>
__global__ void __launch_bounds__(kJoinWarps * 32, 4) join_kernel(const __grid_constant__ VerifyArgs a, Params P,
                                                                  JoinArgs J) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PlanInst s_inst;
    constexpr int kG = G > 0 ? G : 1;
    const int lane = threadIdx.x & 31;
    JoinWarp& W = reinterpret_cast<JoinWarp*>(smem)[threadIdx.x >> 5];
    const unsigned lt = (1u << lane) - 1u;
    if (threadIdx.x == 0) {
        s_inst = plan_inst(a.single);
        if (blockIdx.x == 0) {
            a.table_out[0] = a.single;
            *a.single.count = 0ull;
        }
    }
    __syncthreads();
    const PlanInst& I = s_inst;
    const Entry<POS>* post = static_cast<const Entry<POS>*>(J.post);
    uint32_t* err = &a.ctr->err;
    const uint32_t* all_tokens = reinterpret_cast<const uint32_t*>(P.toks4);
    auto token = [&](uint32_t first_block, uint32_t k) -> uint32_t {
        return ld_at(all_tokens, 4ull * first_block + k, 4ull * a.single.r_n_chunks, err);
    };
    auto cell_start = [&](uint64_t c) -> uint64_t { return ld_at(J.toff, c, J.cells + 1, err); };
    unsigned long long found = 0;  // candidates (warp-uniform)
    uint32_t n = 0, q = 0;         // pairs in buf, candidates waiting for the test (warp-uniform)
    auto hand_over = [&]() {       // buf as one run
        unsigned long long at = 0, run = 0;
        if (lane == 0) {
            at = atomicAdd(&a.ctr->join_pairs, (unsigned long long)n);
            if (at + n <= J.out.pair_cap) run = atomicAdd(&a.ctr->join_runs, 1ull);
        }
        at = __shfl_sync(kAll, at, 0);
        if (at + n <= J.out.pair_cap) {  // (else the host sees the count and asks again with more room)
            if (lane == 0) {
                if (run < J.out.run_cap) J.out.runs[run] = make_ulonglong2(at, n);
                else atomicOr(&a.ctr->err, ERR_GUARD);  // cannot happen with a sized workspace
            }
            for (uint32_t k = lane; k < n; k += 32) J.out.pairs[at + k] = W.buf[k];
        }
        __syncwarp();
        n = 0;
    };
    const Threshold th = threshold(I);
    Sector rs;        // G > 1: the probe's record
    uint32_t nr = 0;
    auto test = [&](uint32_t m) {  // the first m waiting candidates
        if (n >= kJoinFlush) hand_over();
        const uint2 e = W.fresh[(uint32_t)lane < m ? lane : 0];
        bool pass = (uint32_t)lane < m;
        if (G == 1) {
            uint32_t r_head;
            const uint32_t r = ld_at(J.probes, e.x, P.n, err);
            const uint32_t v = bound_of_pair<1, false>(I.s_rec[0], I.r_rec[0], e.y, r, rs, lane, P.n, P.n, err, &r_head);
            pass = pass && bound_passes(I, th, v, r_head >> 16);
        } else if (G > 1) {
            const uint32_t v = bound_of_pair<kG, true>(I.s_rec[0], nullptr, e.y, 0u, rs, lane, P.n, 0u, err);
            pass = pass && bound_passes(I, th, v, nr);
        }
        const uint32_t pm = __ballot_sync(kAll, pass);
        if (pass && in_bounds(n + __popc(pm & lt), kJoinRun, err)) W.buf[n + __popc(pm & lt)] = e;
        n += __popc(pm);
        __syncwarp();
    };
    for (;;) {
        uint32_t g0 = 0;
        if (lane == 0) g0 = atomicAdd(J.cursor, J.grab);
        g0 = __shfl_sync(kAll, g0, 0);
        if (g0 >= P.n) break;
        const uint32_t probes = min(J.grab, P.n - g0);  // (at most 32)
        // lane i: probe g0 + i, its set, prefix length (0: no candidates) and the first position admitted
        uint32_t my_r = 0, my_pl = 0, my_lo = 0;
        uint2 my_d = make_uint2(0u, 0u);
        if ((uint32_t)lane < probes) {
            my_r = ld_at(J.probes, g0 + lane, P.n, err);
            my_d = ld_at(P.desc, my_r, P.n, err);
            my_pl = prefix_len(P, my_d.y);
            if (my_pl) {
                my_lo = (uint32_t)ld_at(J.size_end, min_overlap(P, my_d.y) - 1, J.sizes, err);  // (at least 1, at most the size)
                if (my_lo >= P.n - 1 - (g0 + lane)) my_pl = 0;
            }
        }
        uint32_t left = __ballot_sync(kAll, my_pl != 0);
        // bounds of the lists of tokens k .. k + 31 of probe p, in the cells of the positions it admits,
        // asked for ahead of their use
        uint64_t next_start = 0, next_end = 0;
        auto bounds = [&](uint32_t tok, bool have, int p) {
            const uint32_t first = __shfl_sync(kAll, my_lo, p), last = P.n - 2 - (g0 + p);
            next_start = have ? cell_start(cell_of(P, tok, first)) : 0;
            next_end = have ? cell_start(cell_of(P, tok, last) + 1) : 0;
        };
        if (left) {
            const int p = __ffs(left) - 1;
            const uint32_t t = __shfl_sync(kAll, my_d.x, p);
            const bool have = (uint32_t)lane < __shfl_sync(kAll, my_pl, p);
            bounds(have ? token(t, lane) : 0u, have, p);
        }
        while (left) {
            const int p = __ffs(left) - 1;
            left &= left - 1;
            const int p2 = left ? __ffs(left) - 1 : p;  // the probe after this
            const uint32_t g = g0 + p, rpos = P.n - 1 - g, lo = __shfl_sync(kAll, my_lo, p);
            const uint32_t L = __shfl_sync(kAll, my_d.y, p), pl = __shfl_sync(kAll, my_pl, p);
            const uint32_t pl2 = left ? __shfl_sync(kAll, my_pl, p2) : 0u;
            const uint32_t t = __shfl_sync(kAll, my_d.x, p), t2 = __shfl_sync(kAll, my_d.x, p2);  // first blocks
            if (G > 1) {
                const uint32_t r = __shfl_sync(kAll, my_r, p);
                rs = ld_sector(I.r_rec[0], (uint64_t)r * kG + lane % kG, (uint64_t)P.n * kG, err);
                nr = ld_header(I.r_rec[0], r, kG, P.n, err) >> 16;
            }
            // entries in all, if the positions are more than the bitmap holds
            uint32_t hash_mask = 0;
            if (rpos - lo > kSeenBits) {
                uint64_t e = next_end - next_start;
                for (uint32_t k = 32 + lane; k < pl; k += 32)
                    e += cell_start(cell_of(P, token(t, k), rpos - 1) + 1) - cell_start(cell_of(P, token(t, k), lo));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(kAll, e, o);
                if (e <= kSeenWords / 2) hash_mask = e <= 32 ? 63u : (2u << (31 - __clz((uint32_t)e * 2 - 1))) - 1;
            }
            const uint32_t window = hash_mask ? rpos - lo : kSeenBits;
            for (uint32_t w0 = lo; w0 < rpos; w0 += min(window, rpos - w0)) {
                const uint32_t w1 = w0 + min(window, rpos - w0);
                const uint32_t words = hash_mask ? hash_mask + 1 : (w1 - w0 + 31) / 32;
                for (uint32_t k = lane; k < words; k += 32) W.seen[k] = hash_mask ? kFree : 0u;
                __syncwarp();
                // one index entry per lane (if have), found at the probe's token k
                auto take = [&](bool have, const Entry<POS>& en, uint32_t k) {
                    bool is_new = false;
                    if (have && en.rank >= w0 && en.rank < w1 && position_ok(P, en, L, k)) {
                        if (hash_mask) {
                            uint32_t h = mix32(en.rank) & hash_mask;
                            for (;;) {  // (at most half of the slots are ever taken)
                                const uint32_t old = atomicCAS(W.seen + h, kFree, en.rank);
                                is_new = old == kFree;
                                if (is_new || old == en.rank) break;
                                h = (h + 1) & hash_mask;
                            }
                        } else {
                            const uint32_t b = en.rank - w0, bit = 1u << (b & 31u);
                            is_new = in_bounds(b >> 5, kSeenWords, err) && (atomicOr(W.seen + (b >> 5), bit) & bit) == 0;
                        }
                    }
                    const uint32_t m = __ballot_sync(kAll, is_new);
                    if (m == 0) return;
                    if (is_new && in_bounds(q + __popc(m & lt), 64, err)) W.fresh[q + __popc(m & lt)] = make_uint2(g, en.id);
                    q += __popc(m);
                    found += __popc(m);
                    __syncwarp();
                    if (q >= 32) {
                        test(32);
                        q -= 32;
                        const uint2 keep = W.fresh[32 + lane];
                        __syncwarp();
                        if ((uint32_t)lane < q) W.fresh[lane] = keep;
                        __syncwarp();
                    }
                };
                for (uint32_t k0 = 0; k0 < pl; k0 += 32) {
                    const uint64_t start = next_start, len = next_end - next_start;
                    // the tokens after these: this probe's, its first again (another window), or the next probe's
                    const bool more = k0 + 32 < pl, again = !more && w1 < rpos;
                    const uint32_t kn = more ? k0 + 32 + lane : (uint32_t)lane;
                    const bool have_n = kn < (more || again ? pl : pl2);
                    const uint32_t tok_n = have_n ? token(more || again ? t : t2, kn) : 0u;
                    // lists that do not add up in 32 bits, one by one
                    uint32_t longs = __ballot_sync(kAll, len >= kLongList);
                    while (longs) {
                        const int src = __ffs(longs) - 1;
                        longs &= longs - 1;
                        const uint64_t e0 = __shfl_sync(kAll, start, src), e1 = e0 + __shfl_sync(kAll, len, src);
                        for (uint64_t e = e0; e < e1; e += 32) {
                            const bool have = e + lane < e1;
                            take(have, ld_entry(post, have ? e + lane : e, J.entries, err), k0 + src);
                        }
                    }
                    const uint32_t mine = len >= kLongList ? 0u : (uint32_t)len;
                    uint32_t incl = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(kAll, incl, o);
                        if (lane >= o) incl += y;
                    }
                    const uint32_t total = __shfl_sync(kAll, incl, 31);
                    const uint64_t base = start - (incl - mine);  // entry e of the one list is base + e of its token
                    auto locate = [&](uint32_t e, uint32_t* k) -> uint64_t {
                        uint32_t x = 0;  // tokens whose entries end by e
#pragma unroll
                        for (int step = 16; step >= 1; step >>= 1) {
                            const uint32_t v = __shfl_sync(kAll, incl, x + step - 1);
                            if (v <= e) x += step;
                        }
                        *k = x;
                        return __shfl_sync(kAll, base, x) + e;
                    };
                    Entry<POS> en_n = {};
                    uint32_t k_n = 0;
                    if (total) {
                        const uint64_t at = locate(lane, &k_n);
                        if ((uint32_t)lane < total) en_n = ld_entry(post, at, J.entries, err);
                    }
                    bounds(tok_n, have_n, more || again ? p : p2);
                    for (uint32_t e0 = 0; e0 < total; e0 += 32) {
                        const Entry<POS> en = en_n;
                        const uint32_t k = k_n;
                        if (e0 + 32 < total) {
                            const uint32_t e = e0 + 32 + lane;
                            const uint64_t at = locate(e, &k_n);
                            if (e < total) en_n = ld_entry(post, at, J.entries, err);
                        }
                        take(e0 + lane < total, en, k0 + k);
                    }
                }
            }
            if (G > 1 && q) {  // (the record is this probe's)
                test(q);
                q = 0;
            }
        }
    }
    if (q) test(q);
    if (n) hand_over();
    if (lane == 0 && found) atomicAdd(&a.ctr->candidates, found);
}

// The runs' second level and queueing (a kernel of its own: a function call in
// the join kernel's loops would cost them their registers).
__global__ void __launch_bounds__(kJoinWarps * 32) queue_kernel(const __grid_constant__ VerifyArgs a, JoinQueue Q) {
    __shared__ PlanInst s_inst;
    __shared__ uint2 s_buf[kJoinWarps][kJoinRun];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_inst = plan_inst(a.single);
    __syncthreads();
    if (a.ctr->join_pairs > Q.pair_cap) return;  // not all of them are here: the host asks again
    const unsigned long long runs = min(a.ctr->join_runs, (unsigned long long)Q.run_cap);
    for (unsigned long long b = blockIdx.x * kJoinWarps + warp; b < runs; b += gridDim.x * kJoinWarps) {
        const ulonglong2 run = Q.runs[b];
        const uint32_t n = min((uint32_t)run.y, kJoinRun);
        for (uint32_t k = lane; k < n; k += 32)
            s_buf[warp][k] = in_bounds(run.x + k, Q.pair_cap, &a.ctr->err) ? Q.pairs[run.x + k] : make_uint2(0u, 0u);
        __syncwarp();
        flush_survivors(a, s_inst, 0, s_buf[warp], n, lane);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// GroupJoin expansion: entry k < n_probe_groups is a probe group with its
// candidate groups (every member of the probe group against every member of
// those groups); entry n_probe_groups + g is group g itself (each member
// against the later members, when the group's prefix is not empty).
// ---------------------------------------------------------------------------

struct GroupArgs {
    const uint64_t* group_offsets;
    const uint32_t* members;
    const uint32_t* probe_groups;
    const uint64_t* cand_offsets;
    const uint32_t* cand_groups;
    uint32_t n_groups, n_probe_groups;
};

// one warp per entry: probes, pairs and (inter entries) candidates per probe
__global__ void group_count_kernel(Params P, GroupArgs G, uint64_t* n_probes, uint64_t* n_pairs, uint64_t* per_probe) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_entries = G.n_probe_groups + G.n_groups;
    if (blockIdx.x == 0 && threadIdx.x == 0) n_probes[n_entries] = n_pairs[n_entries] = 0;  // the scans' closing entries
    for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n_entries; k += warps) {
        uint64_t probes = 0, pairs = 0, sum = 0;
        if (k < G.n_probe_groups) {
            const uint32_t g = G.probe_groups[k];
            const uint64_t m = G.group_offsets[g + 1] - G.group_offsets[g];
            for (uint64_t c = G.cand_offsets[k] + lane; c < G.cand_offsets[k + 1]; c += 32) {
                const uint32_t h = G.cand_groups[c];
                sum += G.group_offsets[h + 1] - G.group_offsets[h];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kAll, sum, o);
            probes = sum ? m : 0;
            pairs = m * sum;
        } else {
            const uint32_t g = k - G.n_probe_groups;
            const uint64_t b = G.group_offsets[g], m = G.group_offsets[g + 1] - b;
            if (m >= 2 && prefix_len(P, P.desc[G.members[b]].y) > 0) {
                probes = m - 1;
                pairs = m * (m - 1) / 2;
            }
        }
        if (lane == 0) {
            n_probes[k] = probes;
            n_pairs[k] = pairs;
            per_probe[k] = sum;
        }
    }
}

// one warp per entry: write the expanded probes, offsets and candidates
__global__ void group_write_kernel(GroupArgs G, const uint64_t* probe_off, const uint64_t* pair_off,
                                   const uint64_t* per_probe, uint32_t* probe_ids, uint64_t* cand_offsets,
                                   uint32_t* cand_ids) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_entries = G.n_probe_groups + G.n_groups;
    if (blockIdx.x == 0 && threadIdx.x == 0) cand_offsets[probe_off[n_entries]] = pair_off[n_entries];
    for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n_entries; k += warps) {
        const uint64_t p0 = probe_off[k], np = probe_off[k + 1] - p0, c0 = pair_off[k];
        if (np == 0) continue;
        if (k < G.n_probe_groups) {
            const uint32_t g = G.probe_groups[k];
            const uint64_t b = G.group_offsets[g], S = per_probe[k];
            for (uint64_t i = 0; i < np; ++i) {
                if (lane == 0) {
                    probe_ids[p0 + i] = G.members[b + i];
                    cand_offsets[p0 + i] = c0 + i * S;
                }
                uint64_t w = c0 + i * S;  // the candidate groups' members, in order
                for (uint64_t c = G.cand_offsets[k]; c < G.cand_offsets[k + 1]; ++c) {
                    const uint32_t h = G.cand_groups[c];
                    const uint64_t hb = G.group_offsets[h], hm = G.group_offsets[h + 1] - hb;
                    for (uint64_t j = lane; j < hm; j += 32) cand_ids[w + j] = G.members[hb + j];
                    w += hm;
                }
            }
        } else {
            const uint32_t g = k - G.n_probe_groups;
            const uint64_t b = G.group_offsets[g], m = G.group_offsets[g + 1] - b;
            for (uint64_t i = 0; i < np; ++i) {
                const uint64_t w = c0 + i * (2 * m - i - 1) / 2;  // pairs of the members before i
                if (lane == 0) {
                    probe_ids[p0 + i] = G.members[b + i];
                    cand_offsets[p0 + i] = w;
                }
                for (uint64_t j = i + 1 + lane; j < m; j += 32) cand_ids[w + (j - i - 1)] = G.members[b + j];
            }
        }
    }
}

unsigned grid_for(uint64_t work, unsigned per_block, int num_sms, unsigned per_sm) {
    const uint64_t want = (work + per_block - 1) / per_block;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)num_sms * per_sm));
}

}  // namespace

cudaError_t candgen_run(const CandgenInput& in, cudaStream_t st, int num_sms, CandgenIndex* ix, uint64_t* host_word) {
    Params P;
    P.toks4 = in.toks4;
    P.desc = in.desc;
    P.n = in.n;
    P.sim = in.sim;
    P.p = in.p;
    P.q = in.q;
    P.positional = in.positional;
    P.cells_log2 = candgen_cells_log2(in.vocab);
    P.cell_shift = candgen_cell_shift(in.n, P.cells_log2);
    const uint64_t cells = candgen_cells(in.vocab);
    cudaError_t e;
    const unsigned tb = 256;
    if (in.stage == 0) {
        // order by size, then count prefix tokens
        e = cudaMemsetAsync(ix->size_hist, 0, 8ull * (candgen_toff_at(in.max_len) + cells + 1), st);
        if (e != cudaSuccess) return e;
        if (in.n) {
            const uint32_t per = std::max<uint32_t>((in.n + 2 * (uint32_t)num_sms - 1) / (2 * (uint32_t)num_sms), 1024u);
            const unsigned blocks = (in.n + per - 1) / per;
            size_hist_kernel<<<blocks, kSizeThreads, 0, st>>>(P, per, ix->size_hist);
            e = exclusive_scan_u64(ix->size_hist, in.max_len + 2, ix->scan_scratch, ix->total, st);
            if (e != cudaSuccess) return e;
            place_kernel<<<blocks, kSizeThreads, 0, st>>>(P, per, ix->size_hist, ix->probes, ix->rank);
            token_count_kernel<<<grid_for((uint64_t)kSetLanes * in.n, tb, num_sms, 8), tb, 0, st>>>(P, ix->rank, ix->toff);
        }
        e = exclusive_scan_u64(ix->toff, cells + 1, ix->scan_scratch, ix->total, st, ix->tcnt);
        if (e == cudaSuccess) e = cudaMemcpyAsync(host_word, ix->total, 8, cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return e;
        return cudaStreamSynchronize(st);  // *host_word: index entries
    }
    // fill the token lists
    if (in.n) {
        const unsigned blocks = grid_for((uint64_t)kSetLanes * in.n, tb, num_sms, 8);
        if (in.positional) postings_kernel<true><<<blocks, tb, 0, st>>>(P, ix->rank, ix->tcnt, ix->post);
        else postings_kernel<false><<<blocks, tb, 0, st>>>(P, ix->rank, ix->tcnt, ix->post);
    }
    return cudaGetLastError();
}

template <int G, bool POS>
static cudaError_t launch_join(const VerifyArgs& a, const Params& P, JoinArgs J, int num_sms, cudaStream_t st) {
    constexpr size_t smem = kJoinWarps * sizeof(JoinWarp);
    cudaError_t e = cudaFuncSetAttribute(join_kernel<G, POS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)std::max<uint64_t>(
        1, std::min<uint64_t>(((uint64_t)P.n + kJoinWarps - 1) / kJoinWarps, 4ull * num_sms));
    J.grab = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(8, P.n / (16ull * blocks * kJoinWarps)));
    join_kernel<G, POS><<<blocks, kJoinWarps * 32, smem, st>>>(a, P, J);
    return cudaGetLastError();
}

template <bool POS>
static cudaError_t launch_join(const VerifyArgs& a, const Params& P, const JoinArgs& J, int num_sms, cudaStream_t st) {
    switch (a.single.rec_sectors[0]) {
        case 1: return launch_join<1, POS>(a, P, J, num_sms, st);
        case 2: return launch_join<2, POS>(a, P, J, num_sms, st);
        case 4: return launch_join<4, POS>(a, P, J, num_sms, st);
        case 8: return launch_join<8, POS>(a, P, J, num_sms, st);
        default: return launch_join<0, POS>(a, P, J, num_sms, st);
    }
}

cudaError_t join_probe(const CandgenInput& in, const CandgenIndex& ix, const VerifyArgs& a, const JoinQueue& out,
                       cudaStream_t st, int num_sms) {
    Params P;
    P.toks4 = in.toks4;
    P.desc = in.desc;
    P.n = in.n;
    P.sim = in.sim;
    P.p = in.p;
    P.q = in.q;
    P.positional = in.positional;
    P.cells_log2 = candgen_cells_log2(in.vocab);
    P.cell_shift = candgen_cell_shift(in.n, P.cells_log2);
    JoinArgs J;
    J.probes = ix.probes;
    J.size_end = ix.size_hist;
    J.toff = ix.toff;
    J.post = ix.post;
    J.sizes = (uint64_t)in.max_len + 2;
    J.cells = candgen_cells(in.vocab);
    J.entries = ix.entries;
    J.cursor = &a.ctr->probe_cursor;
    J.grab = 1;
    J.out = out;
    cudaError_t e = cudaMemsetAsync(a.ctr, 0, sizeof(Counters), st);
    if (e != cudaSuccess) return e;
    e = in.positional ? launch_join<true>(a, P, J, num_sms, st) : launch_join<false>(a, P, J, num_sms, st);
    if (e != cudaSuccess) return e;
    queue_kernel<<<(unsigned)(2 * num_sms), kJoinWarps * 32, 0, st>>>(a, out);
    return cudaGetLastError();
}

cudaError_t expand_groups(const GroupExpand& x, cudaStream_t st, int num_sms, uint64_t* host_words) {
    Params P;
    memset(&P, 0, sizeof(P));
    P.toks4 = x.toks4;
    P.desc = x.desc;
    P.sim = x.sim;
    P.p = x.p;
    P.q = x.q;
    GroupArgs G;
    G.group_offsets = x.group_offsets;
    G.members = x.members;
    G.probe_groups = x.probe_groups;
    G.cand_offsets = x.cand_offsets;
    G.cand_groups = x.cand_groups;
    G.n_groups = x.n_groups;
    G.n_probe_groups = x.n_probe_groups;
    const uint64_t n_entries = (uint64_t)x.n_groups + x.n_probe_groups;
    const unsigned tb = 256;
    const unsigned blocks = grid_for(32 * (n_entries + 1), tb, num_sms, 8);
    if (x.stage == 0) {
        group_count_kernel<<<blocks, tb, 0, st>>>(P, G, x.probe_off, x.pair_off, x.per_probe);
        cudaError_t e = exclusive_scan_u64(x.probe_off, n_entries + 1, x.scan_scratch, x.total, st, nullptr, 2,
                                           x.pair_off - x.probe_off);
        if (e == cudaSuccess) e = cudaMemcpyAsync(host_words, x.total, 16, cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return e;
        return cudaStreamSynchronize(st);  // host_words: expanded probes, expanded pairs
    }
    group_write_kernel<<<blocks, tb, 0, st>>>(G, x.probe_off, x.pair_off, x.per_probe, x.probe_ids, x.cand_offsets_out,
                                              x.cand_ids);
    return cudaGetLastError();
}

}  // namespace ssj
