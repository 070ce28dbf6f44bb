// Result triples sorted by (r, s) on the device (SSJ_SORTED), and the results of
// a launch's instances packed for one copy to the host.
//
// The number of results is known on the device only, so the sort of up to
// kSortTile triples an instance is queued right after the verify kernel, one
// CTA per instance, and the host reads count and triples back at once (2,034
// results: std::sort between two copies took about 100 us).  More results are
// sorted after the count has come back: small tiles by the same code, one pass
// that merges sixteen of them, then passes that merge two runs each.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr int kSortThreads = 1024;
constexpr int kMergeThreads = 256;
constexpr uint32_t kMergeTile = 1024;  // triples written by one CTA of a merge pass

__device__ __forceinline__ unsigned long long key_of(const ssj_triple& t) {
    return ((unsigned long long)t.r << 32) | t.s;
}

// n <= kSortTile triples from src to dst (may be the same), by one CTA of
// kSortThreads: runs of 32 sorted in registers (bitonic, by shuffles), then
// merged two by two between two buffers in shared memory, each triple finding
// its place by a binary search of the sibling run.  (Bound by latency: 2,034
// triples take 6 merge steps of at most 11 dependent shared-memory loads; a
// bitonic network in shared memory needs 66 steps with a barrier each and took
// 29 us.)  `smem` holds 2 * kSortTile keys, then as many overlaps.
constexpr size_t kSortSmem = 2 * kSortTile * (sizeof(unsigned long long) + sizeof(uint32_t));

__device__ void sort_tile(const ssj_triple* src, ssj_triple* dst, uint32_t n, unsigned long long* smem) {
    unsigned long long *key = smem, *key2 = smem + kSortTile;
    uint32_t *val = reinterpret_cast<uint32_t*>(smem + 2 * kSortTile), *val2 = val + kSortTile;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t i = threadIdx.x; i - lane < n; i += kSortThreads) {
        unsigned long long k = ~0ull;  // (past the end: last; set ids are below 2^31)
        uint32_t v = 0;
        if (i < n) {
            k = key_of(src[i]);
            v = src[i].overlap;
        }
#pragma unroll
        for (uint32_t size = 2; size <= 32; size <<= 1) {
#pragma unroll
            for (uint32_t j = size >> 1; j > 0; j >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xFFFFFFFFu, k, j);
                const uint32_t v2 = __shfl_xor_sync(0xFFFFFFFFu, v, j);
                // the lower lane of a pair keeps the smaller key in ascending runs
                const bool take = ((lane & j) == 0) == ((lane & size) == 0) ? k2 < k : k2 > k;
                if (take) {
                    k = k2;
                    v = v2;
                }
            }
        }
        key[i] = k;
        val[i] = v;
    }
    __syncthreads();
    for (uint32_t run = 32; run < n; run <<= 1) {
        for (uint32_t i = threadIdx.x; i < n; i += kSortThreads) {
            const unsigned long long k = key[i];
            const uint32_t mine = i / run, sib = (mine ^ 1u) * run;  // first triple of the sibling run
            const uint32_t end = min(sib + run, n);
            uint32_t lo = min(sib, end), hi = end;
            const bool left = (mine & 1u) == 0;
            while (lo < hi) {  // the sibling's triples that go before: smaller ones, and for the right run's also equal ones
                const uint32_t mid = (lo + hi) >> 1;
                if (left ? key[mid] < k : key[mid] <= k) lo = mid + 1; else hi = mid;
            }
            const uint32_t to = left ? i + (lo - min(sib, end)) : sib + (i - mine * run) + (lo - sib);
            key2[to] = k;
            val2[to] = val[i];
        }
        __syncthreads();
        unsigned long long* sk = key;
        key = key2;
        key2 = sk;
        uint32_t* sv = val;
        val = val2;
        val2 = sv;
    }
    for (uint32_t i = threadIdx.x; i < n; i += kSortThreads) {
        ssj_triple t;
        t.r = (uint32_t)(key[i] >> 32);
        t.s = (uint32_t)key[i];
        t.overlap = val[i];
        dst[i] = t;
    }
}

__global__ void __launch_bounds__(kSortThreads) sort_results_kernel(const Instance* table) {
    extern __shared__ unsigned long long smem[];
    const Instance& I = table[blockIdx.x];
    if (!(I.flags & VF_SORTED)) return;
    const unsigned long long n = min(*I.count, (unsigned long long)I.cap);
    if (n >= 2 && n <= kSortTile) sort_tile(I.out, I.out, (uint32_t)n, smem);
}

// Of more triples, tiles of kSmallTile (one a thread: a sort of few triples in one CTA is bound by its
// instructions, 2,034 take 17 us cold, 4,096 36).
constexpr uint32_t kSmallTile = kSortThreads;
constexpr uint32_t kManyRuns = 16;

__global__ void __launch_bounds__(kSortThreads) sort_tiles_kernel(const ssj_triple* src, ssj_triple* dst, uint64_t n) {
    extern __shared__ unsigned long long smem[];
    const uint64_t at = (uint64_t)blockIdx.x * kSmallTile;
    sort_tile(src + at, dst + at, (uint32_t)min((uint64_t)kSmallTile, n - at), smem);
}

// kManyRuns sorted tiles merged into one run from src to dst: a triple's place is its place in its
// tile and in each of the others, found by searches that run side by side (a warp's triples are
// neighbours, so its loads share sectors).  7,342 triples: tiles and this pass 27 us cold; tiles
// of 4,096 and a pass of two runs took 47.
__global__ void __launch_bounds__(kMergeThreads) merge_tiles_kernel(const ssj_triple* src, ssj_triple* dst, uint64_t n) {
    const uint64_t i = (uint64_t)blockIdx.x * kMergeThreads + threadIdx.x;
    if (i >= n) return;
    const uint64_t base = i / (kManyRuns * kSmallTile) * (kManyRuns * kSmallTile);
    const uint32_t c = (uint32_t)(i - base) / kSmallTile;
    const uint32_t m = (uint32_t)min((uint64_t)kManyRuns * kSmallTile, n - base);  // triples of the group
    const ssj_triple* A = src + base;
    const ssj_triple t = src[i];
    const unsigned long long k = key_of(t);
    uint32_t before[kManyRuns];
#pragma unroll
    for (uint32_t s = 0; s < kManyRuns; ++s) before[s] = 0;
    for (uint32_t step = kSmallTile; step; step >>= 1) {
#pragma unroll
        for (uint32_t s = 0; s < kManyRuns; ++s) {
            // smaller triples of tile s go before this one, and equal ones of an earlier tile
            const uint32_t p = before[s] + step;
            if (p <= kSmallTile && s * kSmallTile + p <= m && key_of(A[s * kSmallTile + p - 1]) < k + (s < c)) before[s] = p;
        }
    }
    uint32_t to = (uint32_t)(i - base) - c * kSmallTile;
#pragma unroll
    for (uint32_t s = 0; s < kManyRuns; ++s) to += s == c ? 0u : before[s];
    dst[base + to] = t;
}

// Runs of `run` sorted triples merged two by two from src to dst.  A CTA writes
// kMergeTile of them: it finds the tile's part of both runs by the merge-path
// search of its two diagonals, and each triple its place by a search of the
// other part.
__global__ void __launch_bounds__(kMergeThreads) merge_runs_kernel(const ssj_triple* src, ssj_triple* dst, uint64_t n,
                                                                   uint64_t run) {
    __shared__ unsigned long long key[kMergeTile];
    __shared__ uint32_t val[kMergeTile];
    __shared__ uint64_t s_split[2];
    const uint64_t tile0 = (uint64_t)blockIdx.x * kMergeTile;  // (runs are multiples of the tile)
    const uint64_t base = tile0 / (2 * run) * (2 * run);
    const uint64_t na = min(run, n - base), nb = min(2 * run, n - base) - na;
    const uint64_t d0 = tile0 - base, d1 = min(d0 + kMergeTile, na + nb);
    const ssj_triple *A = src + base, *B = A + na;
    if (threadIdx.x < 2) {  // taken from A by diagonal d (A first on equal keys)
        const uint64_t d = threadIdx.x ? d1 : d0;
        uint64_t lo = d > nb ? d - nb : 0, hi = min(d, na);
        while (lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (key_of(A[mid]) <= key_of(B[d - 1 - mid])) lo = mid + 1; else hi = mid;
        }
        s_split[threadIdx.x] = lo;
    }
    __syncthreads();
    const uint64_t a0 = s_split[0], b0 = d0 - a0;
    const uint32_t ca = (uint32_t)(s_split[1] - a0), c = (uint32_t)(d1 - d0);
    for (uint32_t i = threadIdx.x; i < c; i += kMergeThreads) {
        const ssj_triple t = i < ca ? A[a0 + i] : B[b0 + (i - ca)];
        key[i] = key_of(t);
        val[i] = t.overlap;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c; i += kMergeThreads) {
        const unsigned long long k = key[i];
        uint32_t lo = i < ca ? ca : 0u, hi = i < ca ? c : ca;  // the other part
        while (lo < hi) {  // its triples that go before: smaller ones, and for B's also A's equal ones
            const uint32_t mid = (lo + hi) >> 1;
            if (i < ca ? key[mid] < k : key[mid] <= k) lo = mid + 1; else hi = mid;
        }
        ssj_triple t;
        t.r = (uint32_t)(k >> 32);
        t.s = (uint32_t)k;
        t.overlap = val[i];
        dst[base + d0 + (i < ca ? i + (lo - ca) : (i - ca) + lo)] = t;
    }
}

// The instances' triples side by side, as far as there is room.  A CTA takes
// `per` neighbouring instances: it sums the counts before them, then copies them
// one after the other.  At most kPackCtas CTAs, so that the sums' work grows with
// the instances and not with their square: packing added 24 ms to a call of
// 100,000 batches with one CTA each, 5 now.
constexpr uint32_t kPackCtas = 1024;
__global__ void __launch_bounds__(256) pack_results_kernel(const Instance* table, uint32_t n_inst, uint32_t per,
                                                           ssj_triple* packed, uint64_t room) {
    __shared__ unsigned long long s_at;
    auto kept = [&](uint32_t i) { return min(*table[i].count, (unsigned long long)table[i].cap); };
    const uint32_t lo = blockIdx.x * per, hi = min(lo + per, n_inst);
    if (threadIdx.x == 0) s_at = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (uint32_t i = threadIdx.x; i < lo; i += blockDim.x) mine += kept(i);
    if (mine) atomicAdd(&s_at, mine);
    __syncthreads();
    unsigned long long at = s_at;
    for (uint32_t i = lo; i < hi; ++i) {
        const unsigned long long n = kept(i);
        const uint32_t* src = reinterpret_cast<const uint32_t*>(table[i].out);
        uint32_t* dst = reinterpret_cast<uint32_t*>(packed + at);
        if (at + n <= room)
            for (unsigned long long k = threadIdx.x; k < 3 * n; k += blockDim.x) dst[k] = src[k];
        at += n;
    }
}

}  // namespace

// The kernels' shared memory is above the default limit: raised per device
// (again by every launch: it costs little, and no state is kept).
template <class K>
static cudaError_t allow_sort_smem(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortSmem);
}

cudaError_t sort_results(const Instance* table, uint32_t n_inst, cudaStream_t st) {
    if (n_inst == 0) return cudaSuccess;
    const cudaError_t e = allow_sort_smem(sort_results_kernel);
    if (e != cudaSuccess) return e;
    sort_results_kernel<<<n_inst, kSortThreads, kSortSmem, st>>>(table);
    return cudaGetLastError();
}

cudaError_t pack_results(const Instance* table, uint32_t n_inst, ssj_triple* packed, uint64_t room, cudaStream_t st) {
    if (n_inst == 0) return cudaSuccess;
    const uint32_t per = (n_inst + kPackCtas - 1) / kPackCtas;
    pack_results_kernel<<<(n_inst + per - 1) / per, 256, 0, st>>>(table, n_inst, per, packed, room);
    return cudaGetLastError();
}

cudaError_t sort_triples(ssj_triple* t, uint64_t n, ssj_triple* tmp, cudaStream_t st) {
    if (n < 2) return cudaSuccess;
    uint32_t passes = 1;  // after the tiles
    for (uint64_t run = kManyRuns * kSmallTile; run < n; run *= 2) ++passes;
    ssj_triple* from = (passes & 1) ? tmp : t;  // the last pass ends in t
    ssj_triple* to = (passes & 1) ? t : tmp;
    const cudaError_t e = allow_sort_smem(sort_tiles_kernel);
    if (e != cudaSuccess) return e;
    sort_tiles_kernel<<<(unsigned)((n + kSmallTile - 1) / kSmallTile), kSortThreads, kSortSmem, st>>>(t, from, n);
    merge_tiles_kernel<<<(unsigned)((n + kMergeThreads - 1) / kMergeThreads), kMergeThreads, 0, st>>>(from, to, n);
    std::swap(from, to);
    for (uint64_t run = kManyRuns * kSmallTile; run < n; run *= 2) {
        merge_runs_kernel<<<(unsigned)((n + kMergeTile - 1) / kMergeTile), kMergeThreads, 0, st>>>(from, to, n, run);
        std::swap(from, to);
    }
    return cudaGetLastError();
}

}  // namespace ssj
