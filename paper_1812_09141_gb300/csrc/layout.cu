// Collection layout on the device (Section 3.3.1, Fig. datasetslayout: all
// tokens of a collection in one linear array plus an offsets array that
// delimits the sets, transferred once).
//
// GB300 layout: every set starts on a 16-byte boundary so that verification
// reads sets with aligned 128-bit loads; the gap after a set repeats its
// last token; desc[i] = (first 16-byte chunk of set i, |set i|).
//
// Steps, all on the device after one host-to-device copy of the raw
// offsets and tokens:
//   1. len_kernel   - per set: length, 16-byte chunk count, sortedness check
//   2. scan         - exclusive prefix sum of chunk counts (two or three kernels)
//   3. scatter_kernel - one warp per set copies its tokens and the padding
//   4. record_kernel  - one warp per set: its length, signature and loss
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "ssj_internal.h"

namespace ssj {

namespace {

constexpr int kScanBlock = 1024;             // threads of a scan block
constexpr int kScanTile = 4 * kScanBlock;    // and the values that it sums

__global__ void len_kernel(const uint64_t* __restrict__ offs, const uint32_t* __restrict__ toks, uint32_t n,
                           int validate, uint64_t* __restrict__ chunks, uint32_t* __restrict__ err) {
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t a = offs[i], b = offs[i + 1];
        if (b < a || b - a >= (1ull << 31)) {
            atomicOr(err, 1u);
            chunks[i] = 0;
            continue;
        }
        chunks[i] = (b - a + 3) >> 2;
        if (validate) {
            for (uint64_t t = a + 1; t < b; ++t)
                if (toks[t - 1] >= toks[t]) { atomicOr(err, 2u); break; }
        }
    }
}

// Block-level inclusive scan of 64-bit values (Hillis-Steele over warps).
__device__ uint64_t block_inclusive_scan(uint64_t v, uint64_t* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        uint64_t w = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;
    }
    __syncthreads();
    if (warp > 0) v += sh[warp - 1];
    __syncthreads();
    return v;
}

// in-place exclusive scan per tile; tile totals to sums[blockIdx.x].  blockIdx.y: the array (scanned
// arrays lie `stride` apart).
__global__ void __launch_bounds__(kScanBlock) scan_blocks(uint64_t* data, uint64_t n, uint64_t stride, uint64_t* sums) {
    __shared__ uint64_t sh[32];
    data += blockIdx.y * stride;
    sums += (uint64_t)blockIdx.y * gridDim.x;
    const uint64_t i = (uint64_t)blockIdx.x * kScanTile + 4 * threadIdx.x;
    uint64_t v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = i + k < n ? data[i + k] : 0;
        sum += v[k];
    }
    const uint64_t inc = block_inclusive_scan(sum, sh);
    uint64_t at = inc - sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (i + k < n) data[i + k] = at;
        at += v[k];
    }
    if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = inc;
}

// exclusive scan of the block totals by one block, looping over tiles
__global__ void scan_sums(uint64_t* sums, uint64_t n, uint64_t* total) {
    __shared__ uint64_t sh[32];
    sums += blockIdx.y * n;
    total += blockIdx.y;
    uint64_t carry = 0;
    for (uint64_t base = 0; base < n; base += kScanBlock) {
        const uint64_t i = base + threadIdx.x;
        const uint64_t v = i < n ? sums[i] : 0;
        const uint64_t inc = block_inclusive_scan(v, sh);
        if (i < n) sums[i] = carry + inc - v;
        __shared__ uint64_t tile_total;
        if (threadIdx.x == kScanBlock - 1) tile_total = inc;
        __syncthreads();
        carry += tile_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// Add to a tile what the tiles before it sum to: sums[blockIdx.x] after scan_sums, or (total given)
// the sum of the totals before it, which the block forms itself, the last one the array's total too.
// Up to kScanBlock tiles the second way costs a load and a reduction per block in place of a launch.
__global__ void __launch_bounds__(kScanBlock) scan_add(uint64_t* data, uint64_t n, uint64_t stride,
                                                       const uint64_t* sums, uint64_t* total, uint64_t* copy) {
    __shared__ uint64_t sh[32];
    data += blockIdx.y * stride;
    sums += (uint64_t)blockIdx.y * gridDim.x;
    uint64_t before;
    if (total) {
        __shared__ uint64_t all;
        const uint64_t inc = block_inclusive_scan(threadIdx.x < blockIdx.x ? sums[threadIdx.x] : 0, sh);
        if (threadIdx.x == kScanBlock - 1) {
            all = inc;
            if (blockIdx.x == gridDim.x - 1) total[blockIdx.y] = inc + sums[blockIdx.x];
        }
        __syncthreads();
        before = all;
    } else {
        before = sums[blockIdx.x];
    }
    const uint64_t i = (uint64_t)blockIdx.x * kScanTile + threadIdx.x;
#pragma unroll
    for (int k = 0; k < kScanTile; k += kScanBlock) {
        if (i + k >= n) return;
        const uint64_t v = data[i + k] + before;
        data[i + k] = v;
        if (copy) copy[i + k] = v;
    }
}

// one warp per set: tokens to their 16-byte aligned slot, padding after
__global__ void scatter_kernel(const uint64_t* __restrict__ offs, const uint32_t* __restrict__ toks, uint32_t n,
                               const uint64_t* __restrict__ start_chunk, uint32_t* __restrict__ dst,
                               uint2* __restrict__ desc) {
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const uint64_t a = offs[i], b = offs[i + 1];
        const uint64_t len = b >= a ? b - a : 0;
        const uint64_t sc = start_chunk[i];
        const uint64_t padded = ((len + 3) >> 2) << 2;
        uint32_t* d = dst + (sc << 2);
        // the padding repeats the set's last token (the verify kernel's block
        // compare relies on it: a repeated token neither adds a match on the
        // candidate side nor changes the block's last token)
        for (uint64_t t = lane; t < padded; t += 32) d[t] = toks[a + (t < len ? t : len - 1)];
        if (lane == 0) desc[i] = make_uint2((uint32_t)sc, (uint32_t)len);
    }
}

// One warp per set: the signature (a bit per token, at a multiplicative hash of
// its value scaled to the bitmap) collected in shared memory, then the record
// in whole 16-byte words.
constexpr int kRecWarps = 8;
__global__ void __launch_bounds__(kRecWarps * 32) record_kernel(const uint4* __restrict__ toks4,
                                                                const uint2* __restrict__ desc, uint32_t n,
                                                                uint32_t sectors, uint4* __restrict__ rec) {
    __shared__ uint4 s_rec[kRecWarps][2 * rec_sectors(kRecClasses - 1)];
    const uint32_t warps = gridDim.x * kRecWarps;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* w = reinterpret_cast<uint32_t*>(s_rec[warp]);
    const uint32_t words = 8 * sectors, bits = 32 * (words - 1);
    for (uint32_t i = blockIdx.x * kRecWarps + warp; i < n; i += warps) {
        const uint2 d = desc[i];
        const uint32_t* t = reinterpret_cast<const uint32_t*>(toks4 + d.x);
        for (uint32_t k = lane; k < words; k += 32) w[k] = 0u;
        __syncwarp();
        for (uint32_t k = lane; k < d.y; k += 32) {
            const uint32_t b = __umulhi(t[k] * 0x9E3779B1u, bits);
            atomicOr(w + 1 + (b >> 5), 1u << (b & 31u));
        }
        __syncwarp();
        uint32_t set = 0;
        for (uint32_t k = 1 + lane; k < words; k += 32) set += __popc(w[k]);
        set = __reduce_add_sync(0xFFFFFFFFu, set);
        if (lane == 0) w[0] = d.y >= 0xFFFFu ? 0xFFFF0000u : (d.y << 16) | (d.y - set);
        __syncwarp();
        if (lane < 2 * sectors) rec[(uint64_t)i * 2 * sectors + lane] = s_rec[warp][lane];
        __syncwarp();
    }
}

}  // namespace

cudaError_t build_records(const uint4* toks4, const uint2* desc, uint32_t n, uint32_t c, uint4* rec, cudaStream_t st,
                          int num_sms) {
    if (n == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)std::min<uint64_t>(((uint64_t)n + kRecWarps - 1) / kRecWarps, (uint64_t)num_sms * 8);
    record_kernel<<<blocks, kRecWarps * 32, 0, st>>>(toks4, desc, n, rec_sectors(c), rec);
    return cudaGetLastError();
}

// Build the padded device layout from raw device copies of offsets/tokens.
// Returns the number of 16-byte chunks via *n_chunks (host), after a sync.
// scratch must hold layout_scratch_words(n) uint64 values.
cudaError_t layout_lengths(const uint64_t* d_offs, const uint32_t* d_toks, uint32_t n, int validate,
                           uint64_t* d_scratch, uint32_t* d_err, uint64_t* n_chunks_host, cudaStream_t st,
                           int num_sms) {
    uint64_t* chunks = d_scratch;
    uint64_t* sums = d_scratch + n + 1;
    uint64_t* total = sums + (n + kScanTile - 1) / kScanTile;
    cudaError_t e = cudaMemsetAsync(d_err, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    if (n > 0) {
        unsigned blocks = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)num_sms * 8);
        len_kernel<<<blocks, 256, 0, st>>>(d_offs, d_toks, n, validate, chunks, d_err);
    }
    e = exclusive_scan_u64(chunks, n, sums, total, st);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(n_chunks_host, total, sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(st);
}

cudaError_t layout_scatter(const uint64_t* d_offs, const uint32_t* d_toks, uint32_t n, const uint64_t* d_scratch,
                           uint32_t* d_dst, uint2* d_desc, cudaStream_t st, int num_sms) {
    if (n == 0) return cudaSuccess;
    unsigned blocks = (unsigned)std::min<uint64_t>(((uint64_t)n * 32 + 255) / 256, (uint64_t)num_sms * 16);
    scatter_kernel<<<blocks, 256, 0, st>>>(d_offs, d_toks, n, d_scratch, d_dst, d_desc);
    return cudaGetLastError();
}

size_t layout_scratch_words(uint32_t n) {
    return (size_t)n + 1 + scan_scratch_words(n) + 1;
}

size_t scan_scratch_words(uint64_t n) { return (n + kScanTile - 1) / kScanTile; }

cudaError_t exclusive_scan_u64(uint64_t* data, uint64_t n, uint64_t* scratch, uint64_t* total, cudaStream_t st,
                               uint64_t* copy, uint32_t arrays, uint64_t stride) {
    if (n == 0) return cudaMemsetAsync(total, 0, sizeof(uint64_t) * arrays, st);
    const uint64_t nb = scan_scratch_words(n);
    const dim3 grid((unsigned)nb, arrays);
    const bool sums = nb > kScanBlock;
    scan_blocks<<<grid, kScanBlock, 0, st>>>(data, n, stride, scratch);
    if (sums) scan_sums<<<dim3(1, arrays), kScanBlock, 0, st>>>(scratch, nb, total);
    scan_add<<<grid, kScanBlock, 0, st>>>(data, n, stride, scratch, sums ? nullptr : total, copy);
    return cudaGetLastError();
}

}  // namespace ssj
