// Host side of the C ABI declared in include/ssj.h: contexts, collection
// store, batch validation, synchronous and stream-ordered verification, and
// the continuous-batching serving loop (submit / poll / results).
//
// The co-process scheme of Section 3.2 (Fig. executionoverlap) maps onto
// this file as follows: the caller's filtering thread (H0) submits chunks;
// each admitted chunk gets a slot with its own CUDA stream, so its copies
// and kernels overlap with other chunks on the device (H1); a completion
// thread reads the result count, copies back exactly that many triples and
// releases device memory (H2).  Admission is by a device-memory budget
// (M_c, Section 4.1.2) and a slot count.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <tuple>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "arith.h"
#include "ssj_internal.h"

namespace ssj {
cudaError_t layout_lengths(const uint64_t* d_offs, const uint32_t* d_toks, uint32_t n, int validate,
                           uint64_t* d_scratch, uint32_t* d_err, uint64_t* n_chunks_host, cudaStream_t st,
                           int num_sms);
cudaError_t layout_scatter(const uint64_t* d_offs, const uint32_t* d_toks, uint32_t n, const uint64_t* d_scratch,
                           uint32_t* d_dst, uint2* d_desc, cudaStream_t st, int num_sms);
size_t layout_scratch_words(uint32_t n);
void renumber_by_frequency(const uint64_t* offsets, const uint32_t* tokens, uint32_t n, std::vector<uint32_t>& out);
}  // namespace ssj

using namespace ssj;

namespace {

// An NVTX range over a scope: names the API calls and the serving phases on
// a profiler's timeline (a no-op when no tool is attached).
struct NvtxScope {
    explicit NvtxScope(const char* name) { nvtxRangePushA(name); }
    ~NvtxScope() { nvtxRangePop(); }
    NvtxScope(const NvtxScope&) = delete;
    NvtxScope& operator=(const NvtxScope&) = delete;
};

}  // namespace

namespace {

// Default of the context's index-item threshold (ssj_set_index_items, probe_bin).
constexpr uint32_t kIndexMinCandsDefault = 256;
// ssj_verify_batches plans a call in up to kMaxPieces pieces of whole waves of plan chunks, each as
// soon as its candidate ids are on the device.  The host link moves 211 GB/s, to the copy engine and to
// kernels alike; 8.1e7 candidates of 12 joins take 1.53 ms to copy and 0.8 ms to plan.  In pieces the
// call takes 1.9 ms; in two groups of batches, copied first, 2.1; with the kernels reading all inputs
// over the link 2.2 in pieces and 2.3 in two groups, and the same with only probe ids and offsets read
// so (the search for a chunk's first probe is a chain of reads).
constexpr uint32_t kMaxPieces = 16;
// Candidates of one batch, and of one call or prepared launch: 2^40 ids are 4 TiB, beyond any
// device's memory, and keep every workspace size computed from the count far from 64-bit wrap.
constexpr uint64_t kMaxCands = 1ull << 40;
// Host inputs of one batch up to this size are gathered in pinned memory and go to the device in one
// copy that the call does not wait for: three copies from the caller's arrays and the wait for them
// take about 25 us, gathering 128 KiB 8.
constexpr size_t kSmallInput = 128 << 10;
// Results copied to pinned memory along with their count, before the host knows it, so that calls
// with up to that many wait for the device once (48 KiB take about 2 us; a second wait and copy
// take about 15): of one batch, and of all batches of ssj_verify_batches.
constexpr uint64_t kFirstResults = 4096;
constexpr uint64_t kPackResults = 16384;
// Device memory that the pool of the calls' own memory keeps between them; a call that took more
// gives the rest back before it returns.  (Self-joins of up to a million sets take 70 to 150 MB.)
constexpr uint64_t kKeepCallMemory = 256ull << 20;

struct Collection {
    uint32_t n_sets = 0;
    uint64_t n_tokens = 0;
    uint64_t n_chunks = 0;
    uint32_t* d_toks = nullptr;  // n_chunks * 4 tokens
    uint2* d_desc = nullptr;
    uint4* d_rec[kRecClasses] = {};  // records of class 0 .. rec_classes - 1
    uint32_t rec_classes = 0;        // 0: no records (sets too long for a signature, or no memory)
    double typical_len = 0;          // size-weighted mean set size
    bool renumbered = false;
    uint32_t max_len = 0;        // longest set
    uint32_t vocab = 0;          // largest token on the device + 1
    uint32_t busy = 0;           // submitted batches not yet collected
    size_t l2_window = 0;        // SSJ_PIN_L2: bytes of the token array kept in the persisting L2 set-aside
    float l2_hit_ratio = 0.f;    // share of the window the set-aside holds
};

enum class TicketState { kRunning, kDone, kFailed };

struct Ticket {
    uint64_t id = 0;
    ssj_coll R = 0, S = 0;
    uint32_t flags = 0;
    cudaStream_t stream = nullptr;
    cudaEvent_t kernel_done = nullptr;
    void* d_mem = nullptr;           // one stream-ordered allocation for the whole batch
    uint64_t bytes = 0;              // charged to the budget
    ssj_triple* d_out = nullptr;
    uint64_t out_cap = 0;
    ssj_triple* d_tmp = nullptr;     // the workspace behind the counters, free once the kernels are done
    uint64_t tmp_cap = 0;            // triples it holds
    ssj_triple* h_out = nullptr;     // pinned, grown as needed
    bool sorted = false;             // h_out is sorted
    uint64_t count = 0;
    TicketState state = TicketState::kRunning;
    std::string error;
    uint32_t derr = 0;  // device check bits of a failed batch
    int slot = -1;
};

struct Slot {
    cudaStream_t stream = nullptr;
    cudaEvent_t ev = nullptr;
    cudaEvent_t copied = nullptr;   // host-to-device copies of a submission done
    // pinned staging for host inputs
    uint32_t* h_probe = nullptr;
    uint64_t* h_offs = nullptr;
    uint32_t* h_cand = nullptr;
    uint64_t h_probe_cap = 0, h_offs_cap = 0, h_cand_cap = 0;
    char* h_in = nullptr;           // small inputs, as they lie on the device
    uint64_t h_in_cap = 0;
    ssj_triple* h_out = nullptr;
    uint64_t h_out_cap = 0;
    Counters* h_ctr = nullptr;
    bool busy = false;          // reserved by a ticket until ssj_results collects it
    struct Ticket* pending = nullptr;  // launched, waiting for the completion thread
    // Wakes this slot's completion thread alone: one condition for all slots woke every thread at
    // each submission and completion, and submissions waited about 35 us for the lock they took in
    // turn (16 slots).
    std::unique_ptr<std::condition_variable> wake;
    std::thread completer;
};

}  // namespace

struct ssj_ctx {
    int device = 0;
    int num_sms = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    uint64_t budget = 0;
    uint32_t max_inflight = 0;
    uint32_t thread_max_key = 128;
    uint32_t drain_min_live = 0;  // short-pair policy (0: default)
    uint32_t lane_max_key = 2048;
    uint32_t warp_max_key = 2048;
    uint32_t block_threads = 256;
    uint32_t index_min_cands = kIndexMinCandsDefault;  // probes with this many candidates become index items
    // SSJ_PIN_L2: the context's persisting-L2 set-aside as found (restored when the last pinned
    // collection is unloaded), whether the library raised it, and the pinned collections
    size_t l2_limit_found = 0;
    bool l2_limit_raised = false;
    uint32_t n_pinned = 0;
    std::string err;

    std::map<ssj_coll, Collection> colls;
    ssj_coll next_coll = 1;

    // workspace for synchronous/stream-ordered calls
    void* ws = nullptr;
    size_t ws_bytes = 0;
    // device staging for synchronous host-pointer calls
    void* io = nullptr;
    size_t io_bytes = 0;
    uint64_t* h_count = nullptr;  // pinned, two words
    uint32_t* h_err = nullptr;    // pinned
    Counters* h_ctr = nullptr;    // pinned
    // pinned: results that come back with their count (kFirstResults; ssj_verify_batches:
    // kPackResults), and ssj_verify_batches' counts and instance table
    char* h_in = nullptr;         // pinned: small inputs, as they lie on the device
    uint64_t h_in_cap = 0;
    ssj_triple* h_first = nullptr;
    uint64_t h_first_cap = 0;
    uint64_t* h_counts = nullptr;
    uint64_t h_counts_cap = 0;
    Instance* h_table = nullptr;
    uint64_t h_table_cap = 0;
    // ssj_verify_batches: the stream and events that carry the pieces' copies
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t copy_done[kMaxPieces] = {};
    cudaEvent_t call_start = nullptr;
    Counters* last_ctr = nullptr;
    // kernel timing (SSJ_CTX_PROFILE): events around plan and verify of each launch
    bool profile = false;
    std::vector<cudaEvent_t> prof_ev;  // 3 per recorded launch
    size_t prof_used = 0;             // launches recorded since the last read

    // serving
    std::mutex mu;
    std::condition_variable cv;  // a ticket completed
    cudaMemPool_t pool = nullptr;       // submitted batches
    cudaMemPool_t call_pool = nullptr;  // CallMemory
    std::vector<Slot> slots;
    std::map<uint64_t, std::unique_ptr<Ticket>> tickets;
    uint64_t next_ticket = 1;
    uint64_t used_bytes = 0;
    bool pool_grown = false;   // the pool holds the whole budget (first submission)
    bool stopping = false;
};

namespace {

ssj_status fail(ssj_ctx* ctx, ssj_status st, const char* fmt, ...) {
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        ctx->err = buf;
    }
    return st;
}

ssj_status cuda_fail(ssj_ctx* ctx, cudaError_t e, const char* what) {
    return fail(ctx, SSJ_EDEVICE, "%s: %s", what, cudaGetErrorString(e));
}

#define CUDA_TRY(ctx, expr)                                   \
    do {                                                      \
        cudaError_t e_ = (expr);                              \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #expr); \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        cudaGetDevice(&cur);
        if (prev >= 0 && cur != prev) cudaSetDevice(prev);
    }
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

ssj_status ensure_device_buffer(ssj_ctx* ctx, void** buf, size_t* have, size_t need) {
    if (*have >= need && *buf) return SSJ_OK;
    if (*buf) {
        cudaStreamSynchronize(ctx->stream);
        cudaFree(*buf);
        *buf = nullptr;
        *have = 0;
    }
    size_t sz = std::max<size_t>(need, 1 << 20);
    cudaError_t e = cudaMalloc(buf, sz);
    if (e != cudaSuccess) {
        *buf = nullptr;
        return fail(ctx, SSJ_ENOMEM, "cudaMalloc(%zu): %s", sz, cudaGetErrorString(e));
    }
    *have = sz;
    return SSJ_OK;
}

template <class T>
ssj_status ensure_pinned(ssj_ctx* ctx, T** buf, uint64_t* have, uint64_t need) {
    if (*have >= need && *buf) return SSJ_OK;
    if (*buf) cudaFreeHost(*buf);
    *buf = nullptr;
    uint64_t n = std::max<uint64_t>(need, std::max<uint64_t>(*have * 2, 1024));
    cudaError_t e = cudaMallocHost(reinterpret_cast<void**>(buf), n * sizeof(T));
    if (e != cudaSuccess) {
        *buf = nullptr;
        *have = 0;
        return fail(ctx, SSJ_ENOMEM, "cudaMallocHost: %s", cudaGetErrorString(e));
    }
    *have = n;
    return SSJ_OK;
}

// The kernels load probe ids and candidate ids as 4-byte words and offsets
// and counts as 8-byte words, and store result triples field by field (4
// bytes).  An address the device reads or writes off that alignment would
// fault the context, so such arrays are refused (device memory) or staged
// (pinned host memory).
bool aligned_to(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

ssj_status check_device_alignment(ssj_ctx* ctx, const ssj_batch* b, const void* out, const void* count) {
    if (!aligned_to(b->probe_ids, 4) || !aligned_to(b->cand_offsets, 8) || !aligned_to(b->cand_ids, 4) ||
        !aligned_to(out, 4) || !aligned_to(count, 8))
        return fail(ctx, SSJ_EINVAL,
                    "device arrays must be aligned to their element size (4 bytes for ids and triples, 8 for "
                    "cand_offsets and counts)");
    return SSJ_OK;
}

// Device address of pinned host memory the device can read directly, or
// NULL (pageable memory, no mapping, or an address off the element alignment
// a, which is then staged by a copy).
const void* device_view(const void* p, uintptr_t a) {
    if (!p || !aligned_to(p, a)) return nullptr;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

// Host-side checks of a host batch.  Only what the host needs is read here
// (the first and last offsets); ids and the monotonicity of the offsets are
// checked on the device by the plan and verify kernels, which report
// violations through the error word.
// Status of a launch's device check bits: the caller's input errors (ids,
// offsets) are SSJ_EINVAL even when a capacity guard fired as their
// consequence; a guard or bounds check alone is a library bug, SSJ_EDEVICE.
ssj_status device_check_status(ssj_ctx* ctx, uint32_t derr) {
    if (derr & (ERR_PROBE_ID | ERR_CAND_ID | ERR_OFFSETS))
        return fail(ctx, SSJ_EINVAL, "batch rejected by the device checks (code %u: %s%s%s)", derr,
                    (derr & ERR_PROBE_ID) ? "probe id out of range " : "",
                    (derr & ERR_CAND_ID) ? "candidate id out of range " : "",
                    (derr & ERR_OFFSETS) ? "offsets not nondecreasing from 0 to n_cands" : "");
    if (derr)
        return fail(ctx, SSJ_EDEVICE, "internal device check fired (code %u: %s%s)", derr,
                    (derr & ERR_GUARD) ? "loop bound reached " : "", (derr & ERR_BOUNDS) ? "index out of bounds" : "");
    return SSJ_OK;
}

ssj_status validate_host_batch(ssj_ctx* ctx, const ssj_batch* b, uint64_t* n_cands) {
    if (b->n_probes && (!b->probe_ids || !b->cand_offsets)) return fail(ctx, SSJ_EINVAL, "NULL batch arrays");
    if (!b->cand_offsets) {
        *n_cands = 0;
        return SSJ_OK;
    }
    if (b->cand_offsets[0] != 0) return fail(ctx, SSJ_EINVAL, "cand_offsets[0] must be 0");
    const uint64_t nc = b->cand_offsets[b->n_probes];
    if (nc >= kMaxCands) return fail(ctx, SSJ_EINVAL, "n_cands must be below 2^40");
    if (b->n_cands && b->n_cands != nc) return fail(ctx, SSJ_EINVAL, "n_cands != cand_offsets[n_probes]");
    if (nc && !b->cand_ids) return fail(ctx, SSJ_EINVAL, "NULL cand_ids");
    *n_cands = nc;
    return SSJ_OK;
}

ssj_status resolve(ssj_ctx* ctx, const ssj_batch* b, Collection** R, Collection** S) {
    if (!ctx || !b) return fail(ctx, SSJ_EINVAL, "NULL argument");
    const uint32_t sim = (b->flags & SSJ_SIM_MASK) >> 8;
    if (sim == SIM_OVERLAP) {
        if (b->p == 0 || b->q == 0 || b->p >= (1u << 31) || b->q >= (1u << 31))
            return fail(ctx, SSJ_EINVAL, "overlap threshold must be 0 < p, q < 2^31");
    } else if (b->p == 0 || b->p > b->q || b->q >= (1u << 31)) {
        return fail(ctx, SSJ_EINVAL, "threshold must be 0 < p <= q < 2^31");
    }
    // sizes derived from n_probes (n_probes + 1 offsets, 32-probe tiles) stay within 32 bits
    if (b->n_probes >= (1u << 31)) return fail(ctx, SSJ_EINVAL, "n_probes must be below 2^31");
    if (b->n_cands >= kMaxCands) return fail(ctx, SSJ_EINVAL, "n_cands must be below 2^40");
    auto ir = ctx->colls.find(b->R);
    auto is = ctx->colls.find(b->S);
    if (ir == ctx->colls.end() || is == ctx->colls.end()) return fail(ctx, SSJ_ENOTFOUND, "unknown collection");
    if (b->R != b->S && (ir->second.renumbered || is->second.renumbered))
        return fail(ctx, SSJ_EINVAL, "renumbered collections can only be self-joined");
    const uint32_t known = SSJ_COUNT_ONLY | SSJ_SORTED | SSJ_DEVICE_PTRS | SSJ_EMIT_ALL | SSJ_FORCE_THREAD |
                           SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE | SSJ_FORCE_INDEX | SSJ_SIM_MASK |
                           SSJ_KEEP_INPUTS | SSJ_HOST_DIRECT | SSJ_HOST_STAGED;
    if (b->flags & ~known) return fail(ctx, SSJ_EINVAL, "unknown batch flag");
    const uint32_t forced =
        b->flags & (SSJ_FORCE_THREAD | SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE | SSJ_FORCE_INDEX);
    if (forced & (forced - 1)) return fail(ctx, SSJ_EINVAL, "at most one SSJ_FORCE_* flag");
    *R = &ir->second;
    *S = &is->second;
    return SSJ_OK;
}

uint32_t vflags(uint32_t f) {
    uint32_t v = 0;
    if (f & SSJ_COUNT_ONLY) v |= VF_COUNT_ONLY;
    if (f & SSJ_EMIT_ALL) v |= VF_EMIT_ALL;
    if (f & SSJ_FORCE_THREAD) v |= VF_FORCE_THREAD;
    if (f & SSJ_FORCE_WARP) v |= VF_FORCE_WARP;
    if (f & SSJ_FORCE_BLOCK) v |= VF_FORCE_BLOCK;
    if (f & SSJ_FORCE_LANE) v |= VF_FORCE_LANE;
    if (f & SSJ_FORCE_INDEX) v |= VF_FORCE_INDEX;
    if ((f & SSJ_SORTED) && !(f & SSJ_COUNT_ONLY)) v |= VF_SORTED;
    return v;
}

// Signature bits per token of a set of typical size (the size-weighted mean:
// long sets have the most candidates) wanted of the two levels.
constexpr double kFirstBits = 1.0, kSecondBits = 3.0;

// The smallest record class with that many bits (the largest if none has).
uint32_t record_class(double bits) {
    uint32_t c = 0;
    while (c + 1 < kRecClasses && rec_bits(c) < bits) ++c;
    return c;
}

// The instance of one batch (arrays, output and count are filled by the caller).
Instance make_instance(const ssj_batch* b, const Collection& R, const Collection& S, uint64_t n_cands) {
    Instance I;
    memset(&I, 0, sizeof(I));
    I.r_toks4 = reinterpret_cast<const uint4*>(R.d_toks);
    I.r_desc = R.d_desc;
    I.r_n_sets = R.n_sets;
    I.s_toks4 = reinterpret_cast<const uint4*>(S.d_toks);
    I.s_desc = S.d_desc;
    I.s_n_sets = S.n_sets;
    I.r_n_chunks = R.n_chunks;
    I.s_n_chunks = S.n_chunks;
    // pairs are dropped by their records unless every pair is asked for, or a granularity is forced
    // (which means every pair that the length filter leaves)
    const uint32_t classes = std::min(R.rec_classes, S.rec_classes);
    const uint32_t every = SSJ_EMIT_ALL | SSJ_FORCE_THREAD | SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE |
                           SSJ_FORCE_INDEX;
    if (classes && !(b->flags & every)) {
        const double len = std::min(R.typical_len, S.typical_len);
        const uint32_t c[2] = {std::min(record_class(kFirstBits * len), classes - 1),
                               std::min(record_class(kSecondBits * len), classes - 1)};
        for (int l = 0; l < 2; ++l) {
            if (l == 1 && c[1] <= c[0]) break;  // the first level is as good
            I.r_rec[l] = R.d_rec[c[l]];
            I.s_rec[l] = S.d_rec[c[l]];
            I.rec_sectors[l] = rec_sectors(c[l]);
        }
    }
    I.p = b->p;
    I.sim = (b->flags & SSJ_SIM_MASK) >> 8;
    switch (I.sim) {
        case SIM_DICE: I.den = 2 * b->q; break;
        case SIM_COSINE: I.den = b->q; break;
        case SIM_OVERLAP: I.den = (uint32_t)(((uint64_t)b->p + b->q - 1) / b->q); break;
        default: I.den = b->p + b->q; break;
    }
    I.magic = (I.sim == SIM_JACCARD || I.sim == SIM_DICE) ? div_magic(I.den) : 0;
    I.flags = vflags(b->flags) | (b->R == b->S ? VF_SELF_JOIN : 0u);
    I.n_probes = b->n_probes;
    I.n_cands = n_cands;
    I.tile_base = 0;
    return I;
}

// Chunk partition of a launch's instances (t: sh.n_inst of them), once their total is known.
void set_chunks(Instance* t, LaunchShape& sh, int num_sms) {
    const uint32_t chunk = plan_chunk(sh.total_cands, num_sms);
    sh.n_chunks = 0;
    for (uint32_t i = 0; i < sh.n_inst; ++i) {
        t[i].chunk_base = sh.n_chunks;
        sh.n_chunks += chunks_of(t[i].n_probes, t[i].n_cands, chunk);
    }
}

// The context's granularity policy for a launch whose collections' token
// values are all below vocab_bound; the probe bitmap of index items is sized
// when index items are on or a batch forces them (and the values fit).
// batch_flags: all batches' flags together.
void apply_policy(const ssj_ctx* ctx, VerifyArgs& a, uint64_t vocab_bound, uint32_t batch_flags) {
    a.thread_max_key = ctx->thread_max_key;
    a.drain_min_live = ctx->drain_min_live;
    a.lane_max_key = ctx->lane_max_key;
    a.warp_max_key = ctx->warp_max_key;
    a.index_min_cands = ctx->index_min_cands;
    a.index_words = (ctx->index_min_cands || (batch_flags & SSJ_FORCE_INDEX)) ? index_words_for(vocab_bound) : 0u;
    a.force_thread = (batch_flags & SSJ_FORCE_THREAD) ? 1u : 0u;
}

// The persisting-L2 window of a pinned collection on the launch (none if c is not pinned).
void set_l2_window(VerifyArgs& a, const Collection& c) {
    a.l2_base = c.l2_window ? c.d_toks : nullptr;
    a.l2_bytes = c.l2_window;
    a.l2_hit_ratio = c.l2_hit_ratio;
}

uint64_t vocab_bound(const Collection& R, const Collection& S) {
    return std::max<uint64_t>(std::max<uint64_t>(R.vocab, S.vocab), 1);
}

VerifyArgs make_args(ssj_ctx* ctx, const ssj_batch* b, const Collection& R, const Collection& S, uint64_t n_cands) {
    VerifyArgs a;
    memset(&a, 0, sizeof(a));
    a.single = make_instance(b, R, S, n_cands);
    a.table = nullptr;
    apply_policy(ctx, a, vocab_bound(R, S), b->flags);
    set_l2_window(a, R.l2_window ? R : S);
    return a;
}

// Three timing events for the next launch of a profiling context (else NULL).
cudaEvent_t* profile_events(ssj_ctx* ctx) {
    if (!ctx->profile) return nullptr;
    const size_t need = 3 * (ctx->prof_used + 1);
    while (ctx->prof_ev.size() < need) {
        cudaEvent_t ev;
        if (cudaEventCreate(&ev) != cudaSuccess) return nullptr;
        ctx->prof_ev.push_back(ev);
    }
    cudaEvent_t* evs = &ctx->prof_ev[3 * ctx->prof_used];
    ctx->prof_used++;
    return evs;
}

// Places of a host batch's arrays in one device block.
struct InputLayout {
    size_t offs, cand, end;  // (probe ids at 0)
    InputLayout(uint32_t n_probes, uint64_t n_cands) {
        offs = align256(4ull * std::max<uint32_t>(n_probes, 1));
        cand = offs + align256(8ull * (n_probes + 1));
        end = cand + align256(4ull * std::max<uint64_t>(n_cands, 1));
    }
};

// Gather a small batch's arrays in h (pinned) and queue their copy to base.
cudaError_t copy_small_input(const ssj_batch* b, uint64_t n_cands, const InputLayout& at, char* h, char* base,
                             cudaStream_t s) {
    if (b->n_probes) {
        memcpy(h, b->probe_ids, 4ull * b->n_probes);
        memcpy(h + at.offs, b->cand_offsets, 8ull * (b->n_probes + 1));
    }
    if (n_cands) memcpy(h + at.cand, b->cand_ids, 4 * n_cands);
    return cudaMemcpyAsync(base, h, at.cand + 4 * n_cands, cudaMemcpyHostToDevice, s);
}

void free_collection(Collection& c) {
    cudaFree(c.d_toks);
    cudaFree(c.d_desc);
    for (uint4* r : c.d_rec) cudaFree(r);
}

// Device memory of one call, from a pool of the context's in the order of its
// stream: up to kKeepCallMemory stays in the pool instead of being mapped and
// unmapped by every call (a dozen cudaMalloc and cudaFree took about 1 ms), and
// goes back with the context.
// An allocation from the pool still takes several microseconds: arrays whose
// sizes are known together are carved out of one (block, then get).
class CallMemory {
public:
    explicit CallMemory(ssj_ctx* c) : ctx_(c) {}
    ~CallMemory() {
        for (void* m : mem_) cudaFreeAsync(m, ctx_->stream);
        uint64_t held = 0;
        if (cudaMemPoolGetAttribute(ctx_->call_pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess ||
            held <= kKeepCallMemory)
            return;
        cudaStreamSynchronize(ctx_->stream);
        cudaMemPoolTrimTo(ctx_->call_pool, kKeepCallMemory);
    }
    CallMemory(const CallMemory&) = delete;
    CallMemory& operator=(const CallMemory&) = delete;
    // What get takes of a block for n elements.
    template <class T>
    static size_t room(uint64_t n) {
        return align256(std::max<size_t>(n * sizeof(T), 16));
    }
    // One allocation for the next get calls (the rest of the last one is not used any more).
    void block(size_t bytes) {
        void* m = nullptr;
        at_ = end_ = nullptr;
        if (cudaMallocFromPoolAsync(&m, bytes, ctx_->call_pool, ctx_->stream) != cudaSuccess) {
            cudaGetLastError();
            failed_ = true;
            return;
        }
        mem_.push_back(m);
        at_ = static_cast<char*>(m);
        end_ = at_ + bytes;
    }
    template <class T>
    T* get(uint64_t n) {
        if (failed_) return nullptr;
        if (room<T>(n) > (size_t)(end_ - at_)) block(room<T>(n));
        if (failed_) return nullptr;
        T* m = reinterpret_cast<T*>(at_);
        at_ += room<T>(n);
        return m;
    }
    bool ok() const { return !failed_; }

private:
    ssj_ctx* ctx_;
    std::vector<void*> mem_;
    char* at_ = nullptr;
    char* end_ = nullptr;
    bool failed_ = false;
};

// Queue, after the verify kernel of a one-batch launch on the context's
// stream, the sort of the results and their way back: the counters (with the
// count), and with `host` the first results.
ssj_status queue_results(ssj_ctx* ctx, const VerifyArgs& a, bool host) {
    cudaStream_t s = ctx->stream;
    if (a.single.flags & VF_SORTED) CUDA_TRY(ctx, sort_results(a.table_out, 1, s));
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_ctr, a.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
    if (host && a.single.cap) {
        const ssj_status st = ensure_pinned(ctx, &ctx->h_first, &ctx->h_first_cap, kFirstResults);
        if (st != SSJ_OK) return st;
        CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_first, a.single.out,
                                      sizeof(ssj_triple) * std::min<uint64_t>(a.single.cap, kFirstResults),
                                      cudaMemcpyDeviceToHost, s));
    }
    return SSJ_OK;
}

ssj_status device_check_status(ssj_ctx* ctx, uint32_t derr);

bool triple_less(const ssj_triple& x, const ssj_triple& y) { return x.r != y.r ? x.r < y.r : x.s < y.s; }

// n triples in device memory sorted on the context's stream (on the host if
// there is no memory for the passes).
cudaError_t sort_in_place(ssj_ctx* ctx, ssj_triple* t, uint64_t n) {
    CallMemory mem(ctx);
    ssj_triple* tmp = mem.get<ssj_triple>(n);
    if (mem.ok()) return sort_triples(t, n, tmp, ctx->stream);
    std::vector<ssj_triple> h(n);
    cudaError_t e = cudaMemcpyAsync(h.data(), t, sizeof(ssj_triple) * n, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    std::sort(h.begin(), h.end(), triple_less);
    if (e == cudaSuccess) e = cudaMemcpyAsync(t, h.data(), sizeof(ssj_triple) * n, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    return e;
}

// After a wait for what queue_results queued: the count, and the results to
// `out` (host; NULL: they stay where the launch wrote them), sorted if asked for.
ssj_status collect_results(ssj_ctx* ctx, const VerifyArgs& a, ssj_triple* out, uint64_t cap, uint64_t* n_out) {
    const uint64_t count = ctx->h_ctr->results;
    *n_out = count;
    if (ctx->h_ctr->err) return device_check_status(ctx, ctx->h_ctr->err);
    if (a.single.flags & VF_COUNT_ONLY) return SSJ_OK;
    const uint64_t n = std::min(count, a.single.cap);
    const bool sort = (a.single.flags & VF_SORTED) && n > kSortTile;
    cudaStream_t s = ctx->stream;
    if (sort) {
        CUDA_TRY(ctx, sort_in_place(ctx, a.single.out, n));
        if (!out) CUDA_TRY(ctx, cudaStreamSynchronize(s));
    }
    if (out && n) {
        if (n <= kFirstResults && !sort) {
            memcpy(out, ctx->h_first, sizeof(ssj_triple) * n);
        } else {
            CUDA_TRY(ctx, cudaMemcpyAsync(out, a.single.out, sizeof(ssj_triple) * n, cudaMemcpyDeviceToHost, s));
            CUDA_TRY(ctx, cudaStreamSynchronize(s));
        }
    }
    if (count > cap) return fail(ctx, SSJ_ENOMEM, "%llu result pairs, room for %llu", (unsigned long long)count,
                                 (unsigned long long)cap);
    return SSJ_OK;
}


void completion_loop(ssj_ctx* ctx, int slot);

}  // namespace

// ===========================================================================
// Context
// ===========================================================================

extern "C" ssj_status ssj_create(const ssj_config* config, ssj_ctx** out) {
    if (!config || !out) return SSJ_EINVAL;
    if (config->flags & ~SSJ_CTX_PROFILE) return SSJ_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || config->device < 0 || config->device >= ndev) return SSJ_EINVAL;
    std::unique_ptr<ssj_ctx> ctx(new ssj_ctx());
    ctx->device = config->device;
    ctx->profile = (config->flags & SSJ_CTX_PROFILE) != 0;
    DeviceGuard g(ctx->device);
    if (cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess)
        return SSJ_EDEVICE;
    ctx->budget = config->mem_budget_bytes ? config->mem_budget_bytes : (4ull << 30);
    ctx->max_inflight = config->max_inflight ? config->max_inflight : 4;
    if (config->stream) {
        ctx->stream = static_cast<cudaStream_t>(config->stream);
    } else {
        if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess) return SSJ_EDEVICE;
        ctx->own_stream = true;
    }
    if (cudaMallocHost(reinterpret_cast<void**>(&ctx->h_count), 2 * sizeof(uint64_t)) != cudaSuccess) return SSJ_EDEVICE;
    if (cudaMallocHost(reinterpret_cast<void**>(&ctx->h_err), sizeof(uint32_t)) != cudaSuccess) return SSJ_EDEVICE;
    if (cudaMallocHost(reinterpret_cast<void**>(&ctx->h_ctr), sizeof(Counters)) != cudaSuccess) return SSJ_EDEVICE;
    cudaMemPoolProps props;
    memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = ctx->device;
    if (cudaMemPoolCreate(&ctx->pool, &props) != cudaSuccess) return SSJ_EDEVICE;
    uint64_t threshold = ctx->budget;
    cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &threshold);
    if (cudaMemPoolCreate(&ctx->call_pool, &props) != cudaSuccess) return SSJ_EDEVICE;
    threshold = kKeepCallMemory;
    cudaMemPoolSetAttribute(ctx->call_pool, cudaMemPoolAttrReleaseThreshold, &threshold);
    ctx->slots.resize(ctx->max_inflight);
    for (auto& s : ctx->slots) {
        s.wake.reset(new std::condition_variable());
        if (cudaStreamCreateWithFlags(&s.stream, cudaStreamNonBlocking) != cudaSuccess) return SSJ_EDEVICE;
        // the completion threads sleep on their events instead of spinning, so that many
        // slots do not take the host cores the submitting threads need
        if (cudaEventCreateWithFlags(&s.ev, cudaEventDisableTiming | cudaEventBlockingSync) != cudaSuccess)
            return SSJ_EDEVICE;
        if (cudaEventCreateWithFlags(&s.copied, cudaEventDisableTiming) != cudaSuccess) return SSJ_EDEVICE;
        if (cudaMallocHost(reinterpret_cast<void**>(&s.h_ctr), sizeof(Counters)) != cudaSuccess) return SSJ_EDEVICE;
    }
    ssj_ctx* raw = ctx.release();
    for (size_t i = 0; i < raw->slots.size(); ++i) raw->slots[i].completer = std::thread(completion_loop, raw, (int)i);
    *out = raw;
    return SSJ_OK;
}

// The persisting-L2 set-aside back to what the context had before SSJ_PIN_L2
// raised it, with the persisting lines released.
void release_l2(ssj_ctx* ctx) {
    if (!ctx->l2_limit_raised) return;
    cudaCtxResetPersistingL2Cache();
    cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, ctx->l2_limit_found);
    cudaGetLastError();
    ctx->l2_limit_raised = false;
}

extern "C" void ssj_destroy(ssj_ctx* ctx) {
    if (!ctx) return;
    {
        std::unique_lock<std::mutex> lk(ctx->mu);
        ctx->stopping = true;
    }
    for (auto& s : ctx->slots) s.wake->notify_all();
    for (auto& s : ctx->slots)
        if (s.completer.joinable()) s.completer.join();
    DeviceGuard g(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    for (auto& s : ctx->slots) {
        cudaStreamSynchronize(s.stream);
        cudaStreamDestroy(s.stream);
        cudaEventDestroy(s.ev);
        cudaEventDestroy(s.copied);
        cudaFreeHost(s.h_in);
        cudaFreeHost(s.h_probe);
        cudaFreeHost(s.h_offs);
        cudaFreeHost(s.h_cand);
        cudaFreeHost(s.h_out);
        cudaFreeHost(s.h_ctr);
    }
    for (auto& kv : ctx->tickets)
        if (kv.second->d_mem) {
            cudaFreeAsync(kv.second->d_mem, kv.second->stream);
            cudaStreamSynchronize(kv.second->stream);
        }
    if (ctx->n_pinned) release_l2(ctx);
    for (auto& kv : ctx->colls) free_collection(kv.second);
    cudaFree(ctx->ws);
    cudaFree(ctx->io);
    cudaFreeHost(ctx->h_count);
    cudaFreeHost(ctx->h_err);
    cudaFreeHost(ctx->h_ctr);
    cudaFreeHost(ctx->h_in);
    cudaFreeHost(ctx->h_first);
    cudaFreeHost(ctx->h_counts);
    cudaFreeHost(ctx->h_table);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    for (cudaEvent_t ev : ctx->copy_done)
        if (ev) cudaEventDestroy(ev);
    if (ctx->call_start) cudaEventDestroy(ctx->call_start);

    for (cudaEvent_t ev : ctx->prof_ev) cudaEventDestroy(ev);
    if (ctx->pool) cudaMemPoolDestroy(ctx->pool);
    if (ctx->call_pool) cudaMemPoolDestroy(ctx->call_pool);
    if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
}

extern "C" const char* ssj_last_error(ssj_ctx* ctx) {
    if (!ctx) return "NULL context";
    return ctx->err.c_str();
}

extern "C" ssj_status ssj_set_granularity(ssj_ctx* ctx, uint32_t thread_max_key, uint32_t lane_max_key,
                                          uint32_t warp_max_key, uint32_t block_threads) {
    if (!ctx) return SSJ_EINVAL;
    const uint32_t bt = block_threads & ~(SSJ_WIDE_REGISTERS | SSJ_BULK_STAGING);
    if (block_threads && bt != 128 && bt != 256 && bt != 512)
        return fail(ctx, SSJ_EINVAL,
                    "block_threads must be 128, 256 or 512 (optionally | SSJ_WIDE_REGISTERS | SSJ_BULK_STAGING)");
    if (thread_max_key) ctx->thread_max_key = thread_max_key;
    if (lane_max_key) ctx->lane_max_key = lane_max_key;
    if (warp_max_key) ctx->warp_max_key = warp_max_key;
    if (block_threads) ctx->block_threads = block_threads;
    return SSJ_OK;
}

extern "C" ssj_status ssj_set_index_items(ssj_ctx* ctx, uint32_t min_cands) {
    if (!ctx) return SSJ_EINVAL;
    ctx->index_min_cands = min_cands;
    return SSJ_OK;
}

extern "C" ssj_status ssj_set_short_pairs(ssj_ctx* ctx, uint32_t drain_min_live) {
    if (!ctx) return SSJ_EINVAL;
    if (drain_min_live > 24) return fail(ctx, SSJ_EINVAL, "drain_min_live must be 0 .. 24");
    ctx->drain_min_live = drain_min_live;
    return SSJ_OK;
}

// ===========================================================================
// Collections
// ===========================================================================

extern "C" ssj_status ssj_load_collection(ssj_ctx* ctx, const uint64_t* offsets, const uint32_t* tokens,
                                          uint32_t n_sets, uint32_t flags, ssj_coll* out) {
    NvtxScope nvtx_scope("ssj_load_collection");
    if (!ctx || !offsets || !out) return fail(ctx, SSJ_EINVAL, "NULL argument");
    if (flags & ~(SSJ_RENUMBER_BY_FREQ | SSJ_VALIDATE | SSJ_PIN_L2)) return fail(ctx, SSJ_EINVAL, "unknown load flag");
    // a self-join probes every set, and batches hold fewer than 2^31 probes
    if (n_sets >= (1u << 31)) return fail(ctx, SSJ_EINVAL, "n_sets must be below 2^31");
    if (offsets[0] != 0) return fail(ctx, SSJ_EINVAL, "offsets[0] must be 0");
    for (uint32_t i = 0; i < n_sets; ++i)
        if (offsets[i + 1] < offsets[i]) return fail(ctx, SSJ_EINVAL, "offsets decrease at set %u", i);
    const uint64_t total = offsets[n_sets];
    if (total && !tokens) return fail(ctx, SSJ_EINVAL, "NULL tokens");
    DeviceGuard g(ctx->device);

    std::vector<uint32_t> renum;
    const uint32_t* src = tokens;
    if ((flags & SSJ_RENUMBER_BY_FREQ) && total) {
        if (flags & SSJ_VALIDATE) {  // validate the caller's order before it is rewritten
            for (uint32_t s = 0; s < n_sets; ++s)
                for (uint64_t t = offsets[s] + 1; t < offsets[s + 1]; ++t)
                    if (tokens[t - 1] >= tokens[t]) return fail(ctx, SSJ_EINVAL, "set %u is not strictly increasing", s);
        }
        renumber_by_frequency(offsets, tokens, n_sets, renum);
        src = renum.data();
    }

    // raw copies on the device, then the padded layout built there
    uint64_t* d_offs = nullptr;
    uint32_t* d_raw = nullptr;
    uint64_t* d_scratch = nullptr;
    uint32_t* d_err = nullptr;
    Collection c;
    c.n_sets = n_sets;
    c.n_tokens = total;
    c.renumbered = (flags & SSJ_RENUMBER_BY_FREQ) != 0;
    double sum_sq = 0;
    for (uint32_t i = 0; i < n_sets; ++i) {
        const uint64_t len = offsets[i + 1] - offsets[i];
        c.max_len = std::max<uint32_t>(c.max_len, (uint32_t)std::min<uint64_t>(len, 0xFFFFFFFFu));
        sum_sq += (double)len * (double)len;
    }
    for (uint64_t t = 0; t < total; ++t) c.vocab = std::max<uint32_t>(c.vocab, src[t] == 0xFFFFFFFFu ? src[t] : src[t] + 1);
    auto cleanup = [&]() {
        cudaFree(d_offs);
        cudaFree(d_raw);
        cudaFree(d_scratch);
        cudaFree(d_err);
    };
    cudaError_t e;
    if ((e = cudaMalloc(&d_offs, sizeof(uint64_t) * (n_sets + 1))) != cudaSuccess ||
        (e = cudaMalloc(&d_raw, sizeof(uint32_t) * std::max<uint64_t>(total, 1))) != cudaSuccess ||
        (e = cudaMalloc(&d_scratch, sizeof(uint64_t) * layout_scratch_words(n_sets))) != cudaSuccess ||
        (e = cudaMalloc(&d_err, sizeof(uint32_t))) != cudaSuccess) {
        cleanup();
        return fail(ctx, SSJ_ENOMEM, "collection staging: %s", cudaGetErrorString(e));
    }
    cudaStream_t st = ctx->stream;
    if ((e = cudaMemcpyAsync(d_offs, offsets, sizeof(uint64_t) * (n_sets + 1), cudaMemcpyHostToDevice, st)) !=
            cudaSuccess ||
        (total && (e = cudaMemcpyAsync(d_raw, src, sizeof(uint32_t) * total, cudaMemcpyHostToDevice, st)) !=
                      cudaSuccess)) {
        cleanup();
        return cuda_fail(ctx, e, "collection upload");
    }
    const int validate = (flags & SSJ_VALIDATE) && !(flags & SSJ_RENUMBER_BY_FREQ);
    e = layout_lengths(d_offs, d_raw, n_sets, validate, d_scratch, d_err, ctx->h_count, st, ctx->num_sms);
    if (e != cudaSuccess) {
        cleanup();
        return cuda_fail(ctx, e, "layout_lengths");
    }
    c.n_chunks = *ctx->h_count;
    cudaMemcpy(ctx->h_err, d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost);
    if (*ctx->h_err) {
        cleanup();
        return fail(ctx, SSJ_EINVAL, (*ctx->h_err & 1u) ? "a set holds 2^31 tokens or more" : "a set is not strictly increasing");
    }
    if ((e = cudaMalloc(&c.d_toks, 16 * std::max<uint64_t>(c.n_chunks, 1) + 16)) != cudaSuccess ||
        (e = cudaMalloc(&c.d_desc, sizeof(uint2) * std::max<uint32_t>(n_sets, 1))) != cudaSuccess) {
        cudaFree(c.d_toks);
        cleanup();
        return fail(ctx, SSJ_ENOMEM, "collection: %s", cudaGetErrorString(e));
    }
    e = layout_scatter(d_offs, d_raw, n_sets, d_scratch, c.d_toks, c.d_desc, st, ctx->num_sms);
    // records up to the class that the second level wants; none when even the largest has less than
    // half a bit per token
    c.typical_len = total ? sum_sq / (double)total : 0.0;
    const uint32_t classes = n_sets && rec_bits(kRecClasses - 1) >= 0.5 * c.typical_len
                                 ? record_class(kSecondBits * c.typical_len) + 1 : 0u;
    for (uint32_t k = 0; k < classes && e == cudaSuccess; ++k) {
        if (cudaMalloc(&c.d_rec[k], 32ull * rec_sectors(k) * n_sets) != cudaSuccess) {
            cudaGetLastError();  // no memory: pairs are verified without this class
            c.d_rec[k] = nullptr;
            break;
        }
        e = build_records(reinterpret_cast<const uint4*>(c.d_toks), c.d_desc, n_sets, k, c.d_rec[k], st, ctx->num_sms);
        c.rec_classes = k + 1;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) {
        free_collection(c);
        return cuda_fail(ctx, e, "layout_scatter");
    }
    if (flags & SSJ_PIN_L2) {
        // Persisting-L2 window over the token array, attached to every verify launch that reads
        // this collection.  The context's persisting set-aside (a limit of this context only, gone
        // with it) is raised to the array's size, up to the device's maximum, and restored when
        // the last pinned collection is unloaded.
        int max_persist = 0, max_window = 0;
        cudaDeviceGetAttribute(&max_persist, cudaDevAttrMaxPersistingL2CacheSize, ctx->device);
        cudaDeviceGetAttribute(&max_window, cudaDevAttrMaxAccessPolicyWindowSize, ctx->device);
        size_t setaside = 0;
        cudaDeviceGetLimit(&setaside, cudaLimitPersistingL2CacheSize);
        const size_t bytes = 16 * c.n_chunks;
        const size_t want = std::min(bytes, (size_t)std::max(max_persist, 0));
        if (setaside < want) {
            if (!ctx->l2_limit_raised) ctx->l2_limit_found = setaside;
            if (cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) == cudaSuccess) {
                ctx->l2_limit_raised = true;
                setaside = want;
            }
            cudaGetLastError();  // a refused limit leaves the window smaller, not an error
        }
        c.l2_window = std::min(bytes, (size_t)std::max(max_window, 0));
        if (setaside == 0) c.l2_window = 0;
        c.l2_hit_ratio = c.l2_window ? std::min(1.0f, (float)((double)setaside / (double)c.l2_window)) : 0.f;
        if (c.l2_window) ctx->n_pinned++;
    }
    const ssj_coll h = ctx->next_coll++;
    ctx->colls[h] = c;
    *out = h;
    return SSJ_OK;
}

extern "C" ssj_status ssj_unload_collection(ssj_ctx* ctx, ssj_coll coll) {
    if (!ctx) return SSJ_EINVAL;
    std::unique_lock<std::mutex> lk(ctx->mu);
    auto it = ctx->colls.find(coll);
    if (it == ctx->colls.end()) return fail(ctx, SSJ_ENOTFOUND, "unknown collection %u", coll);
    if (it->second.busy) return fail(ctx, SSJ_EBUSY, "collection %u is used by submitted batches", coll);
    DeviceGuard g(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    free_collection(it->second);
    if (it->second.l2_window && --ctx->n_pinned == 0) release_l2(ctx);
    ctx->colls.erase(it);
    return SSJ_OK;
}

extern "C" ssj_status ssj_collection_info(ssj_ctx* ctx, ssj_coll coll, uint32_t* n_sets, uint64_t* n_tokens) {
    if (!ctx) return SSJ_EINVAL;
    auto it = ctx->colls.find(coll);
    if (it == ctx->colls.end()) return fail(ctx, SSJ_ENOTFOUND, "unknown collection %u", coll);
    if (n_sets) *n_sets = it->second.n_sets;
    if (n_tokens) *n_tokens = it->second.n_tokens;
    return SSJ_OK;
}

// ===========================================================================
// Stream-ordered and synchronous verification
// ===========================================================================

extern "C" ssj_status ssj_reserve(ssj_ctx* ctx, uint32_t n_probes, uint64_t n_cands) {
    if (!ctx) return SSJ_EINVAL;
    if (n_probes >= (1u << 31) || n_cands >= kMaxCands)
        return fail(ctx, SSJ_EINVAL, "n_probes must be below 2^31 and n_cands below 2^40");
    DeviceGuard g(ctx->device);
    return ensure_device_buffer(ctx, &ctx->ws, &ctx->ws_bytes, workspace_bytes(n_probes, n_cands, ctx->num_sms));
}

extern "C" ssj_status ssj_verify_batch_async(ssj_ctx* ctx, const ssj_batch* batch, ssj_triple* d_out, uint64_t cap,
                                             uint64_t* d_count, void* stream) {
    Collection *R, *S;
    ssj_status st = resolve(ctx, batch, &R, &S);
    if (st != SSJ_OK) return st;
    if (!d_count) return fail(ctx, SSJ_EINVAL, "d_count is required");
    if (batch->n_probes && (!batch->probe_ids || !batch->cand_offsets))
        return fail(ctx, SSJ_EINVAL, "NULL batch arrays");
    if (batch->n_cands && !batch->cand_ids) return fail(ctx, SSJ_EINVAL, "NULL cand_ids");
    if (cap && !d_out && !(batch->flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "NULL output");
    st = check_device_alignment(ctx, batch, d_out, d_count);
    if (st != SSJ_OK) return st;
    DeviceGuard g(ctx->device);
    st = ensure_device_buffer(ctx, &ctx->ws, &ctx->ws_bytes, workspace_bytes(batch->n_probes, batch->n_cands, ctx->num_sms));
    if (st != SSJ_OK) return st;
    VerifyArgs a = make_args(ctx, batch, *R, *S, batch->n_cands);
    a.single.probe_ids = batch->probe_ids;
    a.single.cand_offsets = batch->cand_offsets;
    a.single.cand_ids = batch->cand_ids;
    a.single.out = d_out;
    a.single.cap = (batch->flags & SSJ_COUNT_ONLY) ? 0 : cap;
    a.single.count = reinterpret_cast<unsigned long long*>(d_count);
    bind_workspace(a, ctx->ws, batch->n_probes, batch->n_cands, ctx->num_sms);
    ctx->last_ctr = a.ctr;
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : ctx->stream;
    cudaError_t e = launch_verify(a, s, ctx->num_sms, ctx->block_threads, profile_events(ctx));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "launch_verify");
    return SSJ_OK;
}

extern "C" ssj_status ssj_device_error(ssj_ctx* ctx, uint32_t* code) {
    if (!ctx || !code) return SSJ_EINVAL;
    *code = 0;
    if (!ctx->last_ctr) return SSJ_OK;
    DeviceGuard g(ctx->device);
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_err, &ctx->last_ctr->err, sizeof(uint32_t), cudaMemcpyDeviceToHost,
                                  ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    *code = *ctx->h_err;
    CUDA_TRY(ctx, cudaMemsetAsync(&ctx->last_ctr->err, 0, sizeof(uint32_t), ctx->stream));
    return SSJ_OK;
}

namespace {

// Launch one batch (a: everything but the workspace and the count) on the
// context's stream and wait for its results; host_out: where they go, NULL if
// they stay in a.single.out.
ssj_status run_batch(ssj_ctx* ctx, VerifyArgs& a, uint32_t n_probes, uint64_t n_cands, ssj_triple* host_out,
                     uint64_t cap, uint64_t* n_out) {
    ssj_status st = ensure_device_buffer(ctx, &ctx->ws, &ctx->ws_bytes, workspace_bytes(n_probes, n_cands, ctx->num_sms));
    if (st != SSJ_OK) return st;
    bind_workspace(a, ctx->ws, n_probes, n_cands, ctx->num_sms);
    a.single.count = &a.ctr->results;
    ctx->last_ctr = a.ctr;
    const cudaError_t e = launch_verify(a, ctx->stream, ctx->num_sms, ctx->block_threads, profile_events(ctx));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "launch_verify");
    st = queue_results(ctx, a, host_out != nullptr);
    if (st != SSJ_OK) return st;
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return collect_results(ctx, a, host_out, cap, n_out);
}

}  // namespace

extern "C" ssj_status ssj_verify_batch(ssj_ctx* ctx, const ssj_batch* batch, ssj_triple* out, uint64_t cap,
                                       uint64_t* n_out) {
    NvtxScope nvtx_scope("ssj_verify_batch");
    Collection *R, *S;
    ssj_status st = resolve(ctx, batch, &R, &S);
    if (st != SSJ_OK) return st;
    if (!n_out) return fail(ctx, SSJ_EINVAL, "n_out is required");
    if (cap && !out && !(batch->flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "NULL output with cap > 0");
    DeviceGuard g(ctx->device);
    const bool dev = (batch->flags & SSJ_DEVICE_PTRS) != 0;
    const bool count_only = (batch->flags & SSJ_COUNT_ONLY) != 0;
    cudaStream_t s = ctx->stream;
    uint64_t n_cands = 0;
    VerifyArgs a;
    if (!dev) {
        st = validate_host_batch(ctx, batch, &n_cands);
        if (st != SSJ_OK) return st;
        a = make_args(ctx, batch, *R, *S, n_cands);
        // device staging: probe ids, offsets, candidates, count, output
        const uint64_t out_cap = count_only ? 0 : std::min<uint64_t>(cap, n_cands);
        const InputLayout at(batch->n_probes, n_cands);
        st = ensure_device_buffer(ctx, &ctx->io, &ctx->io_bytes,
                                  at.end + align256(sizeof(ssj_triple) * std::max<uint64_t>(out_cap, 1)));
        if (st != SSJ_OK) return st;
        char* base = static_cast<char*>(ctx->io);
        uint32_t* d_probe = reinterpret_cast<uint32_t*>(base);
        uint64_t* d_offs = reinterpret_cast<uint64_t*>(base + at.offs);
        uint32_t* d_cand = reinterpret_cast<uint32_t*>(base + at.cand);
        ssj_triple* d_out = reinterpret_cast<ssj_triple*>(base + at.end);
        const bool small = at.end <= kSmallInput;
        if (small) {
            st = ensure_pinned(ctx, &ctx->h_in, &ctx->h_in_cap, kSmallInput);
            if (st != SSJ_OK) return st;
            CUDA_TRY(ctx, copy_small_input(batch, n_cands, at, ctx->h_in, base, s));
        }
        if (batch->n_probes && !small) {
            CUDA_TRY(ctx, cudaMemcpyAsync(d_probe, batch->probe_ids, 4ull * batch->n_probes, cudaMemcpyHostToDevice, s));
            CUDA_TRY(ctx, cudaMemcpyAsync(d_offs, batch->cand_offsets, 8ull * (batch->n_probes + 1),
                                          cudaMemcpyHostToDevice, s));
        }
        if (n_cands && !small)
            CUDA_TRY(ctx, cudaMemcpyAsync(d_cand, batch->cand_ids, 4ull * n_cands, cudaMemcpyHostToDevice, s));
        a.single.probe_ids = d_probe;
        a.single.cand_offsets = d_offs;
        a.single.cand_ids = d_cand;
        a.single.out = d_out;
        a.single.cap = out_cap;
    } else {
        n_cands = batch->n_cands;
        if (batch->n_probes && (!batch->probe_ids || !batch->cand_offsets))
            return fail(ctx, SSJ_EINVAL, "NULL batch arrays");
        if (n_cands && !batch->cand_ids) return fail(ctx, SSJ_EINVAL, "NULL cand_ids");
        st = check_device_alignment(ctx, batch, out, nullptr);
        if (st != SSJ_OK) return st;
        a = make_args(ctx, batch, *R, *S, n_cands);
        a.single.probe_ids = batch->probe_ids;
        a.single.cand_offsets = batch->cand_offsets;
        a.single.cand_ids = batch->cand_ids;
        a.single.out = out;
        a.single.cap = count_only ? 0 : cap;
    }
    return run_batch(ctx, a, batch->n_probes, n_cands, dev ? nullptr : out, cap, n_out);
}

extern "C" ssj_status ssj_verify_batches(ssj_ctx* ctx, const ssj_batch* batches, uint32_t n_batches,
                                         ssj_triple* const* outs, const uint64_t* caps, uint64_t* n_outs) {
    NvtxScope nvtx_scope("ssj_verify_batches");
    if (!ctx || (n_batches && (!batches || !outs || !caps || !n_outs))) return fail(ctx, SSJ_EINVAL, "NULL argument");
    if (n_batches == 0) return SSJ_OK;
    std::vector<Instance> table(n_batches);
    std::vector<uint64_t> n_cands(n_batches), io_off(n_batches);
    LaunchShape sh;
    sh.n_inst = n_batches;
    sh.n_tiles = 0;
    sh.total_probes = 0;
    sh.total_cands = 0;
    sh.n_chunks = 0;
    const size_t packed_bytes = sizeof(ssj_triple) * kPackResults;  // results for one copy
    size_t off = align256(sizeof(uint64_t) * n_batches) + align256(packed_bytes);  // counts and these first
    uint64_t launch_vocab = 1;
    uint32_t launch_flags = 0;
    const Collection* pinned = nullptr;  // the first pinned collection: its L2 window
    for (uint32_t i = 0; i < n_batches; ++i) {
        const ssj_batch* b = &batches[i];
        if (b->flags & SSJ_DEVICE_PTRS) return fail(ctx, SSJ_EINVAL, "batch %u: host pointers expected", i);
        Collection *R, *S;
        ssj_status st = resolve(ctx, b, &R, &S);
        if (st != SSJ_OK) return st;
        st = validate_host_batch(ctx, b, &n_cands[i]);
        if (st != SSJ_OK) return st;
        if (caps[i] && !outs[i] && !(b->flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "batch %u: NULL output", i);
        table[i] = make_instance(b, *R, *S, n_cands[i]);
        if (!pinned) pinned = R->l2_window ? R : (S->l2_window ? S : nullptr);
        launch_vocab = std::max(launch_vocab, vocab_bound(*R, *S));
        launch_flags |= b->flags;
        table[i].tile_base = sh.n_tiles;
        const uint64_t tiles = ((uint64_t)b->n_probes + 31) / 32;
        if ((uint64_t)sh.n_tiles + tiles > 0x7FFFFFFull) return fail(ctx, SSJ_EINVAL, "too many probes in one call");
        sh.n_tiles += (uint32_t)tiles;
        sh.total_probes += b->n_probes;
        sh.total_cands += n_cands[i];
        if (sh.total_cands >= kMaxCands) return fail(ctx, SSJ_EINVAL, "2^40 or more candidates in one call");
        // device staging of this batch: probe ids, offsets, candidate ids, output
        io_off[i] = off;
        off += align256(4ull * std::max<uint32_t>(b->n_probes, 1)) + align256(8ull * (b->n_probes + 1)) +
               align256(4ull * std::max<uint64_t>(n_cands[i], 1));
        const uint64_t cap = (b->flags & SSJ_COUNT_ONLY) ? 0 : std::min(caps[i], n_cands[i]);
        off += align256(sizeof(ssj_triple) * std::max<uint64_t>(cap, 1));
    }
    set_chunks(table.data(), sh, ctx->num_sms);
    DeviceGuard g(ctx->device);
    ssj_status st = ensure_device_buffer(ctx, &ctx->io, &ctx->io_bytes, off);
    if (st != SSJ_OK) return st;
    st = ensure_device_buffer(ctx, &ctx->ws, &ctx->ws_bytes, workspace_bytes(sh, ctx->num_sms));
    if (st != SSJ_OK) return st;
    if ((st = ensure_pinned(ctx, &ctx->h_counts, &ctx->h_counts_cap, n_batches)) != SSJ_OK ||
        (st = ensure_pinned(ctx, &ctx->h_table, &ctx->h_table_cap, n_batches)) != SSJ_OK ||
        (st = ensure_pinned(ctx, &ctx->h_first, &ctx->h_first_cap, kPackResults)) != SSJ_OK)
        return st;
    cudaStream_t s = ctx->stream;
    char* base = static_cast<char*>(ctx->io);
    uint64_t* d_counts = reinterpret_cast<uint64_t*>(base);
    ssj_triple* d_packed = reinterpret_cast<ssj_triple*>(base + align256(sizeof(uint64_t) * n_batches));
    bool any_sorted = false, any_results = false;
    std::vector<uint32_t*> staged(n_batches, nullptr);  // device place of the candidate ids that are copied
    for (uint32_t i = 0; i < n_batches; ++i) {
        const ssj_batch* b = &batches[i];
        char* p = base + io_off[i];
        uint32_t* d_probe = reinterpret_cast<uint32_t*>(p); p += align256(4ull * std::max<uint32_t>(b->n_probes, 1));
        uint64_t* d_offs = reinterpret_cast<uint64_t*>(p);  p += align256(8ull * (b->n_probes + 1));
        uint32_t* d_cand = reinterpret_cast<uint32_t*>(p);  p += align256(4ull * std::max<uint64_t>(n_cands[i], 1));
        // SSJ_HOST_DIRECT: pinned arrays the device can address are read by the kernels
        // themselves (over the host link), with no staging copy
        const bool direct = (b->flags & SSJ_HOST_DIRECT) != 0;
        const void* dv_probe = direct ? device_view(b->probe_ids, 4) : nullptr;
        const void* dv_offs = direct ? device_view(b->cand_offsets, 8) : nullptr;
        const void* dv_cand = direct ? device_view(b->cand_ids, 4) : nullptr;
        if (b->n_probes && !dv_probe)
            CUDA_TRY(ctx, cudaMemcpyAsync(d_probe, b->probe_ids, 4ull * b->n_probes, cudaMemcpyHostToDevice, s));
        if (b->n_probes && !dv_offs)
            CUDA_TRY(ctx, cudaMemcpyAsync(d_offs, b->cand_offsets, 8ull * (b->n_probes + 1), cudaMemcpyHostToDevice, s));
        if (n_cands[i] && !dv_cand) staged[i] = d_cand;
        Instance& I = table[i];
        I.probe_ids = dv_probe ? static_cast<const uint32_t*>(dv_probe) : d_probe;
        I.cand_offsets = dv_offs ? static_cast<const uint64_t*>(dv_offs) : d_offs;
        I.cand_ids = dv_cand ? static_cast<const uint32_t*>(dv_cand) : d_cand;
        I.out = reinterpret_cast<ssj_triple*>(p);
        I.cap = (b->flags & SSJ_COUNT_ONLY) ? 0 : std::min(caps[i], n_cands[i]);
        I.count = reinterpret_cast<unsigned long long*>(d_counts + i);
        any_sorted = any_sorted || (I.flags & VF_SORTED);
        any_results = any_results || I.cap;
    }
    VerifyArgs a;
    memset(&a, 0, sizeof(a));
    apply_policy(ctx, a, launch_vocab, launch_flags);
    if (pinned) set_l2_window(a, *pinned);
    bind_workspace(a, ctx->ws, sh, ctx->num_sms);
    a.table = a.table_out;
    memcpy(ctx->h_table, table.data(), sizeof(Instance) * n_batches);
    CUDA_TRY(ctx, cudaMemcpyAsync(a.table_out, ctx->h_table, sizeof(Instance) * n_batches, cudaMemcpyHostToDevice, s));
    ctx->last_ctr = a.ctr;
    // pieces of whole waves (plan_wave chunks), each planned when its ids have come over the copy stream
    const uint64_t wave = plan_wave(ctx->num_sms), waves = std::max<uint64_t>((sh.n_chunks + wave - 1) / wave, 1);
    const uint64_t per_piece = wave * ((waves + kMaxPieces - 1) / kMaxPieces);
    const uint32_t pieces = (uint32_t)std::max<uint64_t>((sh.n_chunks + per_piece - 1) / per_piece, 1);
    cudaStream_t cs = s;
    if (pieces > 1) {
        if (!ctx->copy_stream) CUDA_TRY(ctx, cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
        for (uint32_t k = 0; k < pieces; ++k)
            if (!ctx->copy_done[k]) CUDA_TRY(ctx, cudaEventCreateWithFlags(&ctx->copy_done[k], cudaEventDisableTiming));
        if (!ctx->call_start) CUDA_TRY(ctx, cudaEventCreateWithFlags(&ctx->call_start, cudaEventDisableTiming));
        cs = ctx->copy_stream;
        // the copy stream starts after everything already queued on the context's stream
        CUDA_TRY(ctx, cudaEventRecord(ctx->call_start, s));
        CUDA_TRY(ctx, cudaStreamWaitEvent(cs, ctx->call_start, 0));
    }
    cudaEvent_t* ev = profile_events(ctx);
    CUDA_TRY(ctx, cudaMemsetAsync(a.ctr, 0, sizeof(Counters), s));
    if (ev) CUDA_TRY(ctx, cudaEventRecord(ev[0], s));
    for (uint32_t k = 0, i0 = 0; k < pieces; ++k) {
        const uint64_t c0 = k * per_piece, c1 = std::min(c0 + per_piece, sh.n_chunks);
        for (uint32_t i = i0; i < n_batches && table[i].chunk_base < c1; ++i) {
            const uint64_t begin = table[i].chunk_base, end = i + 1 < n_batches ? table[i + 1].chunk_base : sh.n_chunks;
            if (end <= c0) {
                i0 = i + 1;
                continue;
            }
            if (!staged[i]) continue;
            const uint64_t f0 = (std::max(c0, begin) - begin) * a.chunk;
            const uint64_t f1 = std::min((std::min(c1, end) - begin) * a.chunk, n_cands[i]);
            if (f1 > f0)
                CUDA_TRY(ctx, cudaMemcpyAsync(staged[i] + f0, batches[i].cand_ids + f0, 4 * (f1 - f0),
                                              cudaMemcpyHostToDevice, cs));
        }
        if (pieces > 1) {
            CUDA_TRY(ctx, cudaEventRecord(ctx->copy_done[k], cs));
            CUDA_TRY(ctx, cudaStreamWaitEvent(s, ctx->copy_done[k], 0));
        }
        VerifyArgs piece = a;
        piece.chunk_begin = c0;
        piece.n_chunks = c1;
        const cudaError_t e = launch_plan(piece, s, ctx->num_sms);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "launch_plan");
    }
    if (ev) CUDA_TRY(ctx, cudaEventRecord(ev[1], s));
    const cudaError_t e = launch_merge(a, s, ctx->num_sms, ctx->block_threads);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "launch_merge");
    if (ev) CUDA_TRY(ctx, cudaEventRecord(ev[2], s));
    // sorted where asked for, and packed, so that all batches' results come back in one copy
    if (any_sorted) CUDA_TRY(ctx, sort_results(a.table_out, n_batches, s));
    if (any_results) {
        CUDA_TRY(ctx, pack_results(a.table_out, n_batches, d_packed, kPackResults, s));
        CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_first, d_packed, packed_bytes, cudaMemcpyDeviceToHost, s));
    }
    const uint64_t* counts = ctx->h_counts;
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_err, &a.ctr->err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_counts, d_counts, sizeof(uint64_t) * n_batches, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (*ctx->h_err) return device_check_status(ctx, *ctx->h_err);
    bool short_cap = false, waiting = false;
    uint64_t total = 0;
    for (uint32_t i = 0; i < n_batches; ++i) {
        n_outs[i] = counts[i];
        if (batches[i].flags & SSJ_COUNT_ONLY) continue;
        total += std::min(counts[i], table[i].cap);
        short_cap = short_cap || counts[i] > caps[i];
    }
    const ssj_triple* from = ctx->h_first;
    for (uint32_t i = 0; i < n_batches; ++i) {
        if (batches[i].flags & SSJ_COUNT_ONLY) continue;
        const uint64_t n = std::min(counts[i], table[i].cap);
        const bool sort = (table[i].flags & VF_SORTED) && n > kSortTile;
        if (total <= kPackResults && !sort) {
            if (n) memcpy(outs[i], from, sizeof(ssj_triple) * n);
        } else if (n) {
            if (sort) CUDA_TRY(ctx, sort_in_place(ctx, table[i].out, n));
            CUDA_TRY(ctx, cudaMemcpyAsync(outs[i], table[i].out, sizeof(ssj_triple) * n, cudaMemcpyDeviceToHost, s));
            waiting = true;
        }
        from += n;
    }
    if (waiting) CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (short_cap) return fail(ctx, SSJ_ENOMEM, "a batch has more result pairs than its capacity (see n_outs)");
    return SSJ_OK;
}

// ===========================================================================
// Self-join with candidates generated on the device
// ===========================================================================

extern "C" ssj_status ssj_self_join(ssj_ctx* ctx, ssj_coll coll, uint32_t p, uint32_t q, uint32_t flags,
                                    ssj_triple* out, uint64_t cap, uint64_t* n_out, uint64_t* n_candidates) {
    NvtxScope nvtx_scope("ssj_self_join");
    if (!ctx || !n_out) return fail(ctx, SSJ_EINVAL, "NULL argument");
    const uint32_t known = SSJ_COUNT_ONLY | SSJ_SORTED | SSJ_DEVICE_PTRS | SSJ_SIM_MASK | SSJ_JOIN_POSITIONAL |
                           SSJ_FORCE_THREAD | SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE | SSJ_FORCE_INDEX;
    if (flags & ~known) return fail(ctx, SSJ_EINVAL, "unknown flag");
    if (cap && !out && !(flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "NULL output with cap > 0");
    if ((flags & SSJ_DEVICE_PTRS) && !aligned_to(out, 4))
        return fail(ctx, SSJ_EINVAL, "device output must be aligned to 4 bytes");
    // threshold and collection checks through the batch path's resolve()
    ssj_batch probe_b;
    memset(&probe_b, 0, sizeof(probe_b));
    probe_b.R = probe_b.S = coll;
    probe_b.p = p;
    probe_b.q = q;
    probe_b.flags = flags & (SSJ_SIM_MASK | SSJ_FORCE_THREAD | SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE |
                             SSJ_FORCE_INDEX);
    Collection *R, *S;
    ssj_status st = resolve(ctx, &probe_b, &R, &S);
    if (st != SSJ_OK) return st;
    const Collection& C = *R;
    if (C.vocab > (1u << 30)) return fail(ctx, SSJ_EINVAL, "token values above 2^30: load with SSJ_RENUMBER_BY_FREQ");
    DeviceGuard g(ctx->device);
    cudaStream_t s = ctx->stream;
    const uint32_t n = C.n_sets;
    CallMemory mem(ctx);
    CandgenIndex ix;
    const uint64_t cells = candgen_cells(C.vocab);
    const uint64_t scan_n = std::max<uint64_t>((uint64_t)C.max_len + 2, cells + 1);
    const uint64_t toff_at = candgen_toff_at(C.max_len);
    mem.block(CallMemory::room<uint64_t>(toff_at + cells + 1) + 2 * CallMemory::room<uint32_t>(n) +
              CallMemory::room<uint64_t>(cells + 1) + CallMemory::room<uint64_t>(scan_scratch_words(scan_n)) +
              CallMemory::room<uint64_t>(1));
    ix.size_hist = mem.get<uint64_t>(toff_at + cells + 1);
    ix.toff = ix.size_hist + toff_at;
    ix.probes = mem.get<uint32_t>(n);
    ix.rank = mem.get<uint32_t>(n);
    ix.tcnt = mem.get<uint64_t>(cells + 1);
    ix.scan_scratch = mem.get<uint64_t>(scan_scratch_words(scan_n));
    ix.total = mem.get<uint64_t>(1);
    if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "candidate generation index");
    CandgenInput in;
    memset(&in, 0, sizeof(in));
    in.toks4 = reinterpret_cast<const uint4*>(C.d_toks);
    in.desc = C.d_desc;
    in.n = n;
    in.max_len = C.max_len;
    in.vocab = C.vocab;
    in.sim = (flags & SSJ_SIM_MASK) >> 8;
    in.p = p;
    in.q = q;
    in.positional = (flags & SSJ_JOIN_POSITIONAL) ? 1u : 0u;
    in.stage = 0;
    cudaError_t e = candgen_run(in, s, ctx->num_sms, &ix, ctx->h_count);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "candidate generation (index)");
    const uint64_t entries = ix.entries = *ctx->h_count;
    ix.post = mem.get<char>(candgen_entry_bytes(in.positional != 0) * entries);
    if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "prefix index of %llu entries", (unsigned long long)entries);
    in.stage = 1;
    e = candgen_run(in, s, ctx->num_sms, &ix, ctx->h_count);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "candidate generation (lists)");
    // probe, test and verify; the queue is sized for the pairs that joins usually leave, and once
    // more from the counted pairs if they were more
    const bool count_only = (flags & SSJ_COUNT_ONLY) != 0;
    const bool dev_out = (flags & SSJ_DEVICE_PTRS) != 0;
    ssj_batch b;
    memset(&b, 0, sizeof(b));
    b.R = b.S = coll;
    b.p = p;
    b.q = q;
    b.n_probes = n;
    b.flags = flags & ~(SSJ_JOIN_POSITIONAL | SSJ_DEVICE_PTRS);
    VerifyArgs a;
    uint64_t room = std::min<uint64_t>(std::max<uint64_t>(8ull * n, 1u << 18), 1u << 22);
    ssj_triple* d_out = nullptr;
    for (;;) {
        a = make_args(ctx, &b, *R, *S, 0);
        a.single.probe_ids = ix.probes;
        if (!count_only) {
            // no more results than queued pairs
            const uint64_t d_cap = dev_out ? cap : std::min<uint64_t>(cap, room);
            d_out = dev_out ? out : mem.get<ssj_triple>(std::max<uint64_t>(d_cap, 1));
            if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "join output");
            a.single.out = d_out;
            a.single.cap = d_cap;
        }
        st = ensure_device_buffer(ctx, &ctx->ws, &ctx->ws_bytes, join_workspace_bytes(n, room, ctx->num_sms));
        if (st != SSJ_OK) return st;
        const JoinQueue queue = bind_join_workspace(a, ctx->ws, n, room, ctx->num_sms);
        a.single.count = &a.ctr->results;
        ctx->last_ctr = a.ctr;
        cudaEvent_t* ev = profile_events(ctx);
        if (ev) cudaEventRecord(ev[0], s);
        e = join_probe(in, ix, a, queue, s, ctx->num_sms);
        if (ev) cudaEventRecord(ev[1], s);
        if (e == cudaSuccess) e = launch_merge(a, s, ctx->num_sms, ctx->block_threads);
        if (ev) cudaEventRecord(ev[2], s);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "candidate generation (probe)");
        st = queue_results(ctx, a, !dev_out);
        if (st != SSJ_OK) return st;
        CUDA_TRY(ctx, cudaStreamSynchronize(s));
        if (ctx->h_ctr->join_pairs <= room) break;
        room = ctx->h_ctr->join_pairs;
    }
    if (n_candidates) *n_candidates = ctx->h_ctr->candidates;
    return collect_results(ctx, a, dev_out ? nullptr : out, cap, n_out);
}

// ===========================================================================
// GroupJoin: group candidates expanded on the device
// ===========================================================================

extern "C" ssj_status ssj_verify_groups(ssj_ctx* ctx, const ssj_group_batch* gb, ssj_triple* out, uint64_t cap,
                                        uint64_t* n_out, uint64_t* n_pairs) {
    NvtxScope nvtx_scope("ssj_verify_groups");
    if (!ctx || !gb || !n_out) return fail(ctx, SSJ_EINVAL, "NULL argument");
    const uint32_t known = SSJ_COUNT_ONLY | SSJ_SORTED | SSJ_DEVICE_PTRS | SSJ_SIM_MASK | SSJ_FORCE_THREAD |
                           SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE | SSJ_FORCE_INDEX;
    if (gb->flags & ~known) return fail(ctx, SSJ_EINVAL, "unknown flag");
    if (cap && !out && !(gb->flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "NULL output with cap > 0");
    if ((gb->flags & SSJ_DEVICE_PTRS) && !aligned_to(out, 4))
        return fail(ctx, SSJ_EINVAL, "device output must be aligned to 4 bytes");
    if (!gb->group_offsets || (gb->n_groups && !gb->members) || (gb->n_probe_groups && (!gb->probe_groups ||
        !gb->cand_offsets)))
        return fail(ctx, SSJ_EINVAL, "NULL group arrays");
    ssj_batch probe_b;
    memset(&probe_b, 0, sizeof(probe_b));
    probe_b.R = probe_b.S = gb->coll;
    probe_b.p = gb->p;
    probe_b.q = gb->q;
    probe_b.flags = gb->flags & (SSJ_SIM_MASK | SSJ_FORCE_THREAD | SSJ_FORCE_WARP | SSJ_FORCE_BLOCK | SSJ_FORCE_LANE |
                                SSJ_FORCE_INDEX);
    Collection *R, *S;
    ssj_status st = resolve(ctx, &probe_b, &R, &S);
    if (st != SSJ_OK) return st;
    const Collection& C = *R;
    // host-side checks of the group layout (ids are the collection's)
    const uint64_t n_members = gb->group_offsets[gb->n_groups];
    if (gb->group_offsets[0] != 0) return fail(ctx, SSJ_EINVAL, "group_offsets[0] must be 0");
    for (uint32_t g = 0; g < gb->n_groups; ++g)
        if (gb->group_offsets[g + 1] <= gb->group_offsets[g]) return fail(ctx, SSJ_EINVAL, "group %u is empty", g);
    for (uint64_t i = 0; i < n_members; ++i)
        if (gb->members[i] >= C.n_sets) return fail(ctx, SSJ_EINVAL, "member id out of range");
    const uint64_t n_cg = gb->n_probe_groups ? gb->cand_offsets[gb->n_probe_groups] : 0;
    if (gb->n_probe_groups && gb->cand_offsets[0] != 0) return fail(ctx, SSJ_EINVAL, "cand_offsets[0] must be 0");
    for (uint32_t k = 0; k < gb->n_probe_groups; ++k) {
        if (gb->probe_groups[k] >= gb->n_groups || gb->cand_offsets[k + 1] < gb->cand_offsets[k])
            return fail(ctx, SSJ_EINVAL, "probe group entry %u invalid", k);
    }
    for (uint64_t c = 0; c < n_cg; ++c)
        if (gb->cand_groups[c] >= gb->n_groups) return fail(ctx, SSJ_EINVAL, "candidate group id out of range");
    DeviceGuard g(ctx->device);
    cudaStream_t s = ctx->stream;
    CallMemory mem(ctx);
    const uint64_t n_entries = (uint64_t)gb->n_groups + gb->n_probe_groups;
    GroupExpand x;
    memset(&x, 0, sizeof(x));
    x.toks4 = reinterpret_cast<const uint4*>(C.d_toks);
    x.desc = C.d_desc;
    x.sim = (gb->flags & SSJ_SIM_MASK) >> 8;
    x.p = gb->p;
    x.q = gb->q;
    x.n_groups = gb->n_groups;
    x.n_probe_groups = gb->n_probe_groups;
    const uint64_t scan_words = 2 * scan_scratch_words(n_entries + 1);
    mem.block(CallMemory::room<uint64_t>((uint64_t)gb->n_groups + 1) + CallMemory::room<uint32_t>(n_members) +
              CallMemory::room<uint32_t>(gb->n_probe_groups) +
              CallMemory::room<uint64_t>((uint64_t)gb->n_probe_groups + 1) + CallMemory::room<uint32_t>(n_cg) +
              CallMemory::room<uint64_t>(2 * (n_entries + 1)) + CallMemory::room<uint64_t>(n_entries) +
              CallMemory::room<uint64_t>(scan_words) + CallMemory::room<uint64_t>(2));
    uint64_t* d_goff = mem.get<uint64_t>((uint64_t)gb->n_groups + 1);
    uint32_t* d_mem = mem.get<uint32_t>(n_members);
    uint32_t* d_pg = mem.get<uint32_t>(gb->n_probe_groups);
    uint64_t* d_coff = mem.get<uint64_t>((uint64_t)gb->n_probe_groups + 1);
    uint32_t* d_cg = mem.get<uint32_t>(n_cg);
    x.probe_off = mem.get<uint64_t>(2 * (n_entries + 1));
    x.pair_off = x.probe_off + n_entries + 1;
    x.per_probe = mem.get<uint64_t>(n_entries);
    x.scan_scratch = mem.get<uint64_t>(scan_words);
    x.total = mem.get<uint64_t>(2);
    if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "group expansion");
    cudaError_t e = cudaMemcpyAsync(d_goff, gb->group_offsets, 8ull * (gb->n_groups + 1), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && n_members) e = cudaMemcpyAsync(d_mem, gb->members, 4ull * n_members, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && gb->n_probe_groups) {
        e = cudaMemcpyAsync(d_pg, gb->probe_groups, 4ull * gb->n_probe_groups, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(d_coff, gb->cand_offsets, 8ull * (gb->n_probe_groups + 1), cudaMemcpyHostToDevice, s);
    }
    if (e == cudaSuccess && n_cg) e = cudaMemcpyAsync(d_cg, gb->cand_groups, 4ull * n_cg, cudaMemcpyHostToDevice, s);
    x.group_offsets = d_goff;
    x.members = d_mem;
    x.probe_groups = d_pg;
    x.cand_offsets = d_coff;
    x.cand_groups = d_cg;
    x.stage = 0;
    if (e == cudaSuccess) e = expand_groups(x, s, ctx->num_sms, ctx->h_count);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "group expansion (count)");
    const uint64_t probes = ctx->h_count[0], pairs = ctx->h_count[1];
    if (n_pairs) *n_pairs = pairs;
    if (probes > 0xFFFFFFFFull) return fail(ctx, SSJ_EINVAL, "too many expanded probes");
    const bool count_only = (gb->flags & SSJ_COUNT_ONLY) != 0;
    const bool dev_out = (gb->flags & SSJ_DEVICE_PTRS) != 0;
    const uint64_t out_room = count_only || dev_out ? 0 : std::max<uint64_t>(std::min<uint64_t>(cap, pairs), 1);
    mem.block(CallMemory::room<uint32_t>(probes) + CallMemory::room<uint64_t>(probes + 1) +
              CallMemory::room<uint32_t>(pairs) + (out_room ? CallMemory::room<ssj_triple>(out_room) : 0));
    x.probe_ids = mem.get<uint32_t>(probes);
    x.cand_offsets_out = mem.get<uint64_t>(probes + 1);
    x.cand_ids = mem.get<uint32_t>(pairs);
    if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "expanded candidates (%llu pairs)", (unsigned long long)pairs);
    x.stage = 1;
    e = expand_groups(x, s, ctx->num_sms, nullptr);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "group expansion (write)");
    ssj_batch b;
    memset(&b, 0, sizeof(b));
    b.R = b.S = gb->coll;
    b.p = gb->p;
    b.q = gb->q;
    b.n_probes = (uint32_t)probes;
    b.flags = gb->flags & ~SSJ_DEVICE_PTRS;
    if (probes >= (1u << 31) || pairs >= kMaxCands) return fail(ctx, SSJ_EINVAL, "too many expanded pairs");
    VerifyArgs a = make_args(ctx, &b, *R, *S, pairs);
    a.single.probe_ids = x.probe_ids;
    a.single.cand_offsets = x.cand_offsets_out;
    a.single.cand_ids = x.cand_ids;
    if (!count_only) {
        a.single.cap = dev_out ? cap : std::min<uint64_t>(cap, pairs);
        a.single.out = dev_out ? out : mem.get<ssj_triple>(out_room);
        if (!mem.ok()) return fail(ctx, SSJ_ENOMEM, "group join output");
    }
    return run_batch(ctx, a, (uint32_t)probes, pairs, dev_out || count_only ? nullptr : out, cap, n_out);
}

// ===========================================================================
// Serving: continuous batching
// ===========================================================================

namespace {

uint64_t batch_device_bytes(uint32_t n_probes, uint64_t n_cands, bool count_only, bool dev_ptrs, int num_sms) {
    uint64_t b = 0;
    if (!dev_ptrs) {
        b += align256(4ull * std::max<uint32_t>(n_probes, 1));
        b += align256(8ull * (n_probes + 1));
        b += align256(4ull * std::max<uint64_t>(n_cands, 1));
    }
    b += align256(workspace_bytes(n_probes, n_cands, num_sms));
    if (!count_only) b += align256(sizeof(ssj_triple) * std::max<uint64_t>(n_cands, 1));
    return b;
}

// True if p lies in page-locked host memory (cudaMallocHost, cudaHostAlloc,
// cudaHostRegister), which the copy engines read directly.
bool is_pinned(const void* p) {
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeHost;
}

// memcpy of pageable input into pinned staging; a large copy is split over a
// few threads, since one core's copy rate is well below the host-to-device
// link's.
void staged_copy(void* dst, const void* src, size_t bytes) {
    constexpr size_t kPart = size_t(8) << 20;
    const size_t hw = std::max(2u, std::thread::hardware_concurrency());
    const size_t parts = std::min<size_t>(std::min<size_t>(bytes / kPart, 8), hw / 2);
    if (parts <= 1) {
        memcpy(dst, src, bytes);
        return;
    }
    const size_t step = ((bytes + parts - 1) / parts + 63) & ~size_t(63);
    std::vector<std::thread> th;
    for (size_t i = 1; i < parts; ++i) {
        const size_t b0 = std::min(bytes, i * step), b1 = std::min(bytes, b0 + step);
        if (b1 > b0)
            th.emplace_back([=] { memcpy(static_cast<char*>(dst) + b0, static_cast<const char*>(src) + b0, b1 - b0); });
    }
    memcpy(dst, src, std::min(bytes, step));
    for (auto& t : th) t.join();
}

void completion_loop(ssj_ctx* ctx, int slot) {
    cudaSetDevice(ctx->device);
    Slot& sl = ctx->slots[slot];
    for (;;) {
        Ticket* t = nullptr;
        {
            std::unique_lock<std::mutex> lk(ctx->mu);
            sl.wake->wait(lk, [&] { return ctx->stopping || sl.pending != nullptr; });
            if (!sl.pending) return;  // stopping with nothing in flight
            t = sl.pending;
        }
        std::string err;
        NvtxScope nvtx_scope("ssj serving: wait for the batch's kernels, copy its results");
        cudaError_t e = cudaEventSynchronize(t->kernel_done);
        uint64_t count = 0;
        if (e == cudaSuccess) {
            count = sl.h_ctr->results;
            if (sl.h_ctr->err) {
                err = "device-side batch check failed";
                t->derr = sl.h_ctr->err;
            }
        } else {
            err = std::string("batch failed: ") + cudaGetErrorString(e);
        }
        if (err.empty() && !(t->flags & SSJ_COUNT_ONLY)) {
            // the first results came with the counters; more are sorted if asked for and copied now
            const uint64_t n_copy = std::min(count, t->out_cap);
            const bool sort = (t->flags & SSJ_SORTED) && n_copy > kSortTile;
            t->sorted = !sort || n_copy <= t->tmp_cap;
            if (sort && t->sorted) {
                e = sort_triples(t->d_out, n_copy, t->d_tmp, sl.stream);
                if (e != cudaSuccess) err = std::string("result sort: ") + cudaGetErrorString(e);
            }
            if (err.empty() && (n_copy > kFirstResults || sort)) {
                if (ensure_pinned(nullptr, &sl.h_out, &sl.h_out_cap, n_copy) != SSJ_OK) err = "pinned output";
                if (err.empty()) {
                    e = cudaMemcpyAsync(sl.h_out, t->d_out, sizeof(ssj_triple) * n_copy, cudaMemcpyDeviceToHost,
                                        sl.stream);
                    if (e == cudaSuccess) e = cudaStreamSynchronize(sl.stream);
                    if (e != cudaSuccess) err = std::string("result copy: ") + cudaGetErrorString(e);
                }
            }
        }
        if (t->d_mem) {
            cudaFreeAsync(t->d_mem, sl.stream);
            t->d_mem = nullptr;
        }
        {
            std::unique_lock<std::mutex> lk(ctx->mu);
            t->count = count;
            t->h_out = sl.h_out;
            t->error = err;
            t->state = err.empty() ? TicketState::kDone : TicketState::kFailed;
            ctx->used_bytes -= t->bytes;
            t->bytes = 0;
            sl.pending = nullptr;
        }
        ctx->cv.notify_all();
    }
}

}  // namespace

extern "C" ssj_status ssj_submit(ssj_ctx* ctx, const ssj_batch* batch, uint64_t* ticket) {
    NvtxScope nvtx_scope("ssj_submit");
    if (!ctx || !batch || !ticket) return fail(ctx, SSJ_EINVAL, "NULL argument");
    std::unique_lock<std::mutex> lk(ctx->mu);
    Collection *R, *S;
    ssj_status st = resolve(ctx, batch, &R, &S);
    if (st != SSJ_OK) return st;
    const bool dev = (batch->flags & SSJ_DEVICE_PTRS) != 0;
    const bool count_only = (batch->flags & SSJ_COUNT_ONLY) != 0;
    uint64_t n_cands = batch->n_cands;
    if (dev) {
        st = check_device_alignment(ctx, batch, nullptr, nullptr);
        if (st != SSJ_OK) return st;
    } else {
        lk.unlock();  // validation reads only the caller's arrays and immutable collection sizes
        st = validate_host_batch(ctx, batch, &n_cands);
        lk.lock();
        if (st != SSJ_OK) return st;
    }
    const uint64_t bytes = batch_device_bytes(batch->n_probes, n_cands, count_only, dev, ctx->num_sms);
    if (bytes > ctx->budget) return fail(ctx, SSJ_EINVAL, "batch needs %llu bytes, budget is %llu",
                                         (unsigned long long)bytes, (unsigned long long)ctx->budget);
    if (!ctx->pool_grown) {
        // reserve the budget in the pool once, so that later submissions never wait on the
        // driver for memory (the release threshold keeps it there)
        DeviceGuard g0(ctx->device);
        void* tmp = nullptr;
        cudaStream_t s0 = ctx->slots.empty() ? ctx->stream : ctx->slots[0].stream;
        if (cudaMallocFromPoolAsync(&tmp, ctx->budget, ctx->pool, s0) == cudaSuccess) {
            cudaFreeAsync(tmp, s0);
            cudaStreamSynchronize(s0);
        } else {
            cudaGetLastError();  // not reserved up front; allocations grow the pool as they come
        }
        ctx->pool_grown = true;
    }
    int slot = -1;
    for (size_t i = 0; i < ctx->slots.size(); ++i)
        if (!ctx->slots[i].busy) { slot = (int)i; break; }
    if (slot < 0 || ctx->used_bytes + bytes > ctx->budget) return SSJ_EAGAIN;
    // reserve the slot, the budget and the collections, then work without the lock
    Slot& sl = ctx->slots[slot];
    sl.busy = true;
    ctx->used_bytes += bytes;
    R->busy++;
    S->busy++;
    std::unique_ptr<Ticket> t(new Ticket());
    t->id = ctx->next_ticket++;
    VerifyArgs a = make_args(ctx, batch, *R, *S, n_cands);
    lk.unlock();

    auto unreserve = [&](ssj_status code) {
        std::unique_lock<std::mutex> l2(ctx->mu);
        sl.busy = false;
        ctx->used_bytes -= bytes;
        R->busy--;
        S->busy--;
        return code;
    };
    DeviceGuard g(ctx->device);
    cudaStream_t s = sl.stream;
    t->R = batch->R;
    t->S = batch->S;
    t->flags = batch->flags;
    t->stream = s;
    t->kernel_done = sl.ev;
    t->slot = slot;
    t->bytes = bytes;
    cudaError_t e = cudaMallocFromPoolAsync(&t->d_mem, bytes, ctx->pool, s);
    if (e != cudaSuccess) return unreserve(fail(ctx, SSJ_ENOMEM, "pool allocation: %s", cudaGetErrorString(e)));
    bool direct_copy = false;
    char* base = static_cast<char*>(t->d_mem);
    size_t off = 0;
    if (!dev) {
        // Small inputs are gathered in this slot's pinned memory.  Larger ones in pinned memory are
        // copied straight from the caller's arrays, and the call waits for those copies before it
        // returns; pageable ones go through the slot's pinned staging.  Either way the caller may
        // reuse its arrays once ssj_submit returns.
        const InputLayout at(batch->n_probes, n_cands);
        uint32_t* d_probe = reinterpret_cast<uint32_t*>(base);
        uint64_t* d_offs = reinterpret_cast<uint64_t*>(base + at.offs);
        uint32_t* d_cand = reinterpret_cast<uint32_t*>(base + at.cand);
        off = at.end;
        if (at.end <= kSmallInput) {
            if ((st = ensure_pinned(ctx, &sl.h_in, &sl.h_in_cap, kSmallInput)) != SSJ_OK) {
                cudaFreeAsync(t->d_mem, s);
                return unreserve(st);
            }
            e = copy_small_input(batch, n_cands, at, sl.h_in, base, s);
        } else {
            const uint64_t offs_n = batch->n_probes ? batch->n_probes + 1ull : 0;
            const bool pin_probe = batch->n_probes && is_pinned(batch->probe_ids);
            const bool pin_offs = offs_n && is_pinned(batch->cand_offsets);
            const bool pin_cand = n_cands && is_pinned(batch->cand_ids);
            direct_copy = pin_probe || pin_offs || pin_cand;
            if ((!pin_probe && (st = ensure_pinned(ctx, &sl.h_probe, &sl.h_probe_cap, std::max<uint64_t>(batch->n_probes, 1))) != SSJ_OK) ||
                (!pin_offs && (st = ensure_pinned(ctx, &sl.h_offs, &sl.h_offs_cap, batch->n_probes + 1ull)) != SSJ_OK) ||
                (!pin_cand && (st = ensure_pinned(ctx, &sl.h_cand, &sl.h_cand_cap, std::max<uint64_t>(n_cands, 1))) != SSJ_OK)) {
                cudaFreeAsync(t->d_mem, s);
                return unreserve(st);
            }
            const void* src_probe = batch->probe_ids;
            const void* src_offs = batch->cand_offsets;
            const void* src_cand = batch->cand_ids;
            if (batch->n_probes && !pin_probe) {
                staged_copy(sl.h_probe, batch->probe_ids, 4ull * batch->n_probes);
                src_probe = sl.h_probe;
            }
            if (offs_n && !pin_offs) {
                staged_copy(sl.h_offs, batch->cand_offsets, 8ull * offs_n);
                src_offs = sl.h_offs;
            }
            if (n_cands && !pin_cand) {
                staged_copy(sl.h_cand, batch->cand_ids, 4ull * n_cands);
                src_cand = sl.h_cand;
            }
            if (batch->n_probes) e = cudaMemcpyAsync(d_probe, src_probe, 4ull * batch->n_probes, cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess && offs_n) e = cudaMemcpyAsync(d_offs, src_offs, 8ull * offs_n, cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess && n_cands) e = cudaMemcpyAsync(d_cand, src_cand, 4ull * n_cands, cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess && direct_copy) e = cudaEventRecord(sl.copied, s);
        }
        if (e != cudaSuccess) {
            cudaStreamSynchronize(s);  // no copy may still read the caller's arrays
            cudaFreeAsync(t->d_mem, s);
            return unreserve(cuda_fail(ctx, e, "submit copy"));
        }
        a.single.probe_ids = d_probe;
        a.single.cand_offsets = d_offs;
        a.single.cand_ids = d_cand;
    } else {
        a.single.probe_ids = batch->probe_ids;
        a.single.cand_offsets = batch->cand_offsets;
        a.single.cand_ids = batch->cand_ids;
    }
    void* ws = base + off;
    const size_t ws_bytes = align256(workspace_bytes(batch->n_probes, n_cands, ctx->num_sms));
    off += ws_bytes;
    ssj_triple* d_out = count_only ? nullptr : reinterpret_cast<ssj_triple*>(base + off);
    a.single.out = d_out;
    a.single.cap = count_only ? 0 : n_cands;
    bind_workspace(a, ws, batch->n_probes, n_cands, ctx->num_sms);
    a.single.count = &a.ctr->results;
    t->d_tmp = reinterpret_cast<ssj_triple*>(static_cast<char*>(ws) + align256(sizeof(Counters)));
    t->tmp_cap = (ws_bytes - align256(sizeof(Counters))) / sizeof(ssj_triple);
    e = launch_verify(a, s, ctx->num_sms, ctx->block_threads, nullptr);
    if (e == cudaSuccess && (a.single.flags & VF_SORTED)) e = sort_results(a.table_out, 1, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sl.h_ctr, a.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && a.single.cap) {
        if (ensure_pinned(ctx, &sl.h_out, &sl.h_out_cap, kFirstResults) != SSJ_OK) e = cudaErrorMemoryAllocation;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(sl.h_out, d_out, sizeof(ssj_triple) * std::min<uint64_t>(a.single.cap, kFirstResults),
                                cudaMemcpyDeviceToHost, s);
    }
    if (e == cudaSuccess) e = cudaEventRecord(sl.ev, s);
    // pinned inputs: wait for their copies unless the caller keeps them until the ticket is done
    if (e == cudaSuccess && direct_copy && !(batch->flags & SSJ_KEEP_INPUTS)) e = cudaEventSynchronize(sl.copied);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(s);
        cudaFreeAsync(t->d_mem, s);
        return unreserve(cuda_fail(ctx, e, "submit"));
    }
    t->d_out = d_out;
    t->out_cap = a.single.cap;
    lk.lock();
    Ticket* raw = t.get();
    ctx->tickets[raw->id] = std::move(t);
    sl.pending = raw;
    *ticket = raw->id;
    lk.unlock();
    sl.wake->notify_one();
    return SSJ_OK;
}

extern "C" ssj_status ssj_poll(ssj_ctx* ctx, uint64_t ticket, int timeout_ms, int* done) {
    if (!ctx || !done) return SSJ_EINVAL;
    std::unique_lock<std::mutex> lk(ctx->mu);
    auto it = ctx->tickets.find(ticket);
    if (it == ctx->tickets.end()) return fail(ctx, SSJ_ENOTFOUND, "unknown ticket %llu", (unsigned long long)ticket);
    Ticket* t = it->second.get();
    auto ready = [&] { return t->state != TicketState::kRunning; };
    if (timeout_ms < 0) {
        ctx->cv.wait(lk, ready);
    } else if (timeout_ms > 0) {
        ctx->cv.wait_for(lk, std::chrono::milliseconds(timeout_ms), ready);
    }
    *done = ready() ? 1 : 0;
    if (!*done) return SSJ_ETIMEDOUT;
    if (t->state == TicketState::kFailed)
        return t->derr ? device_check_status(ctx, t->derr) : fail(ctx, SSJ_EDEVICE, "%s", t->error.c_str());
    return SSJ_OK;
}

extern "C" ssj_status ssj_results(ssj_ctx* ctx, uint64_t ticket, ssj_triple* out, uint64_t cap, uint64_t* n_out) {
    NvtxScope nvtx_scope("ssj_results");
    if (!ctx || !n_out) return SSJ_EINVAL;
    std::unique_lock<std::mutex> lk(ctx->mu);
    auto it = ctx->tickets.find(ticket);
    if (it == ctx->tickets.end()) return fail(ctx, SSJ_ENOTFOUND, "unknown ticket %llu", (unsigned long long)ticket);
    Ticket* t = it->second.get();
    if (t->state == TicketState::kRunning) return SSJ_EAGAIN;
    *n_out = t->count;
    if (!out && t->state == TicketState::kDone) return SSJ_OK;
    ssj_status st = SSJ_OK;
    if (t->state == TicketState::kFailed) {
        st = t->derr ? device_check_status(ctx, t->derr) : fail(ctx, SSJ_EDEVICE, "%s", t->error.c_str());
    } else if (!(t->flags & SSJ_COUNT_ONLY)) {
        if (cap < t->count) return fail(ctx, SSJ_ENOMEM, "%llu result pairs, room for %llu",
                                        (unsigned long long)t->count, (unsigned long long)cap);
        if (t->count) memcpy(out, t->h_out, sizeof(ssj_triple) * t->count);
        if ((t->flags & SSJ_SORTED) && !t->sorted) std::sort(out, out + t->count, triple_less);
    }
    ctx->slots[t->slot].busy = false;
    auto ir = ctx->colls.find(t->R);
    if (ir != ctx->colls.end() && ir->second.busy) ir->second.busy--;
    auto is = ctx->colls.find(t->S);
    if (is != ctx->colls.end() && is->second.busy) is->second.busy--;
    ctx->tickets.erase(it);
    return st;
}

extern "C" ssj_status ssj_profile_read(ssj_ctx* ctx, uint32_t* launches, double* plan_ms, double* verify_ms) {
    if (!ctx || !launches || !plan_ms || !verify_ms) return SSJ_EINVAL;
    *launches = 0;
    *plan_ms = 0;
    *verify_ms = 0;
    if (!ctx->profile) return fail(ctx, SSJ_EINVAL, "context was created without SSJ_CTX_PROFILE");
    DeviceGuard g(ctx->device);
    for (size_t i = 0; i < ctx->prof_used; ++i) {
        cudaEvent_t* ev = &ctx->prof_ev[3 * i];
        CUDA_TRY(ctx, cudaEventSynchronize(ev[2]));
        float a = 0, b = 0;
        CUDA_TRY(ctx, cudaEventElapsedTime(&a, ev[0], ev[1]));
        CUDA_TRY(ctx, cudaEventElapsedTime(&b, ev[1], ev[2]));
        *plan_ms += a;
        *verify_ms += b;
    }
    *launches = (uint32_t)ctx->prof_used;
    ctx->prof_used = 0;
    return SSJ_OK;
}

// ===========================================================================
// Helpers for the scratch-free entry point (noalloc.cu): they read the
// context and never allocate.
// ===========================================================================

namespace ssj {

ssj_status resolve_device_batch(ssj_ctx* ctx, const ssj_batch* batch, const void* out, const void* count,
                                VerifyArgs* a, int* device, int* num_sms, uint32_t* block_threads,
                                cudaStream_t* ctx_stream) {
    Collection *R, *S;
    ssj_status st = resolve(ctx, batch, &R, &S);
    if (st != SSJ_OK) return st;
    if (batch->n_probes && (!batch->probe_ids || !batch->cand_offsets))
        return fail(ctx, SSJ_EINVAL, "NULL batch arrays");
    if (batch->n_cands && !batch->cand_ids) return fail(ctx, SSJ_EINVAL, "NULL cand_ids");
    st = check_device_alignment(ctx, batch, out, count);
    if (st != SSJ_OK) return st;
    *a = make_args(ctx, batch, *R, *S, batch->n_cands);
    a->single.probe_ids = batch->probe_ids;
    a->single.cand_offsets = batch->cand_offsets;
    a->single.cand_ids = batch->cand_ids;
    *device = ctx->device;
    *num_sms = ctx->num_sms;
    *block_threads = ctx->block_threads;
    *ctx_stream = ctx->stream;
    return SSJ_OK;
}

ssj_status report(ssj_ctx* ctx, ssj_status st, const char* msg) { return fail(ctx, st, "%s", msg); }

void remember_counters(ssj_ctx* ctx, Counters* c) { ctx->last_ctr = c; }

}  // namespace ssj

// ===========================================================================
// Batched instances
// ===========================================================================

struct ssj_multi {
    VerifyArgs a;
    LaunchShape shape;
    uint32_t block_threads = 256;
    uint32_t index_words_fit = 0;  // probe bitmap words the instances' token values need (0: too many)
    uint32_t batch_flags = 0;      // of all instances together
    void* ws = nullptr;
    std::vector<ssj_coll> colls;  // collections marked busy
    cudaStream_t capture_stream = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

extern "C" ssj_status ssj_multi_create(ssj_ctx* ctx, const ssj_batch* batches, uint32_t n_batches,
                                       ssj_triple* const* d_outs, const uint64_t* caps, uint64_t* d_counts,
                                       ssj_multi** out) {
    if (!ctx || !out || (n_batches && (!batches || !d_outs || !caps || !d_counts)))
        return fail(ctx, SSJ_EINVAL, "NULL argument");
    std::vector<Instance> table(n_batches);
    LaunchShape sh;
    sh.n_inst = n_batches;
    sh.n_tiles = 0;
    sh.total_probes = 0;
    sh.total_cands = 0;
    sh.n_chunks = 0;
    std::unique_ptr<ssj_multi> m(new ssj_multi());
    uint64_t vocab = 1;
    const Collection* pinned = nullptr;  // the first pinned collection: its L2 window
    for (uint32_t i = 0; i < n_batches; ++i) {
        const ssj_batch* b = &batches[i];
        Collection *R, *S;
        ssj_status st = resolve(ctx, b, &R, &S);
        if (st != SSJ_OK) return st;
        if (b->n_probes && (!b->probe_ids || !b->cand_offsets)) return fail(ctx, SSJ_EINVAL, "batch %u: NULL arrays", i);
        if (b->n_cands && !b->cand_ids) return fail(ctx, SSJ_EINVAL, "batch %u: NULL cand_ids", i);
        if (caps[i] && !d_outs[i] && !(b->flags & SSJ_COUNT_ONLY)) return fail(ctx, SSJ_EINVAL, "batch %u: NULL output", i);
        st = check_device_alignment(ctx, b, d_outs[i], d_counts + i);
        if (st != SSJ_OK) return st;
        Instance I = make_instance(b, *R, *S, b->n_cands);
        I.probe_ids = b->probe_ids;
        I.cand_offsets = b->cand_offsets;
        I.cand_ids = b->cand_ids;
        I.out = d_outs[i];
        I.cap = (b->flags & SSJ_COUNT_ONLY) ? 0 : caps[i];
        I.count = reinterpret_cast<unsigned long long*>(d_counts + i);
        I.tile_base = sh.n_tiles;
        const uint64_t tiles = ((uint64_t)b->n_probes + 31) / 32;
        if ((uint64_t)sh.n_tiles + tiles > 0x7FFFFFFull) return fail(ctx, SSJ_EINVAL, "too many probes in one launch");
        sh.n_tiles += (uint32_t)tiles;
        sh.total_probes += b->n_probes;
        sh.total_cands += b->n_cands;
        if (sh.total_cands >= kMaxCands) return fail(ctx, SSJ_EINVAL, "2^40 or more candidates in one launch");
        table[i] = I;
        m->colls.push_back(b->R);
        m->colls.push_back(b->S);
        vocab = std::max(vocab, vocab_bound(*R, *S));
        m->batch_flags |= b->flags;
        if (!pinned) pinned = R->l2_window ? R : (S->l2_window ? S : nullptr);
    }
    set_chunks(table.data(), sh, ctx->num_sms);
    DeviceGuard g(ctx->device);
    const size_t bytes = workspace_bytes(sh, ctx->num_sms);
    cudaError_t e = cudaMalloc(&m->ws, bytes);
    if (e != cudaSuccess) return fail(ctx, SSJ_ENOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
    memset(&m->a, 0, sizeof(m->a));
    apply_policy(ctx, m->a, vocab, m->batch_flags);
    if (pinned) set_l2_window(m->a, *pinned);
    m->index_words_fit = index_words_for(vocab);
    m->block_threads = ctx->block_threads;
    bind_workspace(m->a, m->ws, sh, ctx->num_sms);
    m->a.table = m->a.table_out;
    m->shape = sh;
    if (n_batches) {
        e = cudaMemcpy(m->a.table_out, table.data(), sizeof(Instance) * n_batches, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            cudaFree(m->ws);
            return cuda_fail(ctx, e, "instance table upload");
        }
    }
    e = prepare_verify(ctx->block_threads, m->a.index_words);
    if (e != cudaSuccess) {
        cudaFree(m->ws);
        return cuda_fail(ctx, e, "prepare_verify");
    }
    {
        std::unique_lock<std::mutex> lk(ctx->mu);
        for (ssj_coll c : m->colls) ctx->colls[c].busy++;
    }
    *out = m.release();
    return SSJ_OK;
}

extern "C" ssj_status ssj_multi_launch(ssj_ctx* ctx, ssj_multi* m, void* stream) {
    NvtxScope nvtx_scope("ssj_multi_launch");
    if (!ctx || !m) return SSJ_EINVAL;
    DeviceGuard g(ctx->device);
    ctx->last_ctr = m->a.ctr;
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : ctx->stream;
    cudaError_t e = launch_verify(m->a, s, ctx->num_sms, m->block_threads, profile_events(ctx));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "launch_verify");
    return SSJ_OK;
}

extern "C" ssj_status ssj_multi_graph_launch(ssj_ctx* ctx, ssj_multi* m, void* stream) {
    if (!ctx || !m) return SSJ_EINVAL;
    DeviceGuard g(ctx->device);
    if (!m->exec) {
        CUDA_TRY(ctx, cudaStreamCreateWithFlags(&m->capture_stream, cudaStreamNonBlocking));
        CUDA_TRY(ctx, cudaStreamBeginCapture(m->capture_stream, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = launch_verify(m->a, m->capture_stream, ctx->num_sms, m->block_threads, nullptr);
        cudaGraph_t graph = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(m->capture_stream, &graph);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "capture launch_verify");
        if (e2 != cudaSuccess) return cuda_fail(ctx, e2, "cudaStreamEndCapture");
        m->graph = graph;
        CUDA_TRY(ctx, cudaGraphInstantiate(&m->exec, m->graph, 0));
    }
    ctx->last_ctr = m->a.ctr;
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : ctx->stream;
    CUDA_TRY(ctx, cudaGraphLaunch(m->exec, s));
    return SSJ_OK;
}

extern "C" void ssj_multi_destroy(ssj_ctx* ctx, ssj_multi* m) {
    if (!m) return;
    if (ctx) {
        DeviceGuard g(ctx->device);
        cudaDeviceSynchronize();
        std::unique_lock<std::mutex> lk(ctx->mu);
        for (ssj_coll c : m->colls) {
            auto it = ctx->colls.find(c);
            if (it != ctx->colls.end() && it->second.busy) it->second.busy--;
        }
        if (ctx->last_ctr == m->a.ctr) ctx->last_ctr = nullptr;
    }
    if (m->exec) cudaGraphExecDestroy(m->exec);
    if (m->graph) cudaGraphDestroy(m->graph);
    if (m->capture_stream) cudaStreamDestroy(m->capture_stream);
    cudaFree(m->ws);
    delete m;
}

// ===========================================================================
// Autotuning of a batched launch
// ===========================================================================

namespace {

// Median device time (ms) of reps launches of m with the given granularity,
// after one untimed launch; negative on a CUDA error (*err receives it).
float time_setting(ssj_ctx* ctx, const ssj_multi* m, uint32_t tmax, uint32_t lmax, uint32_t wmax, uint32_t bt,
                   uint32_t dml, uint32_t imin, uint32_t reps, cudaStream_t s, cudaEvent_t* ev, cudaError_t* err) {
    VerifyArgs a = m->a;
    a.thread_max_key = tmax;
    a.lane_max_key = lmax;
    a.warp_max_key = wmax;
    a.drain_min_live = dml;
    a.index_min_cands = imin;
    a.index_words = (imin || (m->batch_flags & SSJ_FORCE_INDEX)) ? m->index_words_fit : 0u;
    cudaError_t e = prepare_verify(bt, a.index_words);
    if (e == cudaSuccess) e = launch_verify(a, s, ctx->num_sms, bt, nullptr);
    std::vector<float> ms;
    for (uint32_t i = 0; e == cudaSuccess && i < reps; ++i) {
        e = cudaEventRecord(ev[0], s);
        if (e == cudaSuccess) e = launch_verify(a, s, ctx->num_sms, bt, nullptr);
        if (e == cudaSuccess) e = cudaEventRecord(ev[1], s);
        if (e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
        float t = 0;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t, ev[0], ev[1]);
        ms.push_back(t);
    }
    if (e != cudaSuccess) {
        *err = e;
        return -1.0f;
    }
    std::sort(ms.begin(), ms.end());
    return ms[ms.size() / 2];
}

}  // namespace

extern "C" ssj_status ssj_multi_autotune(ssj_ctx* ctx, ssj_multi* m, void* stream, uint32_t reps,
                                         ssj_tune_result* out) {
    NvtxScope nvtx_scope("ssj_multi_autotune");
    if (!ctx || !m || !out) return fail(ctx, SSJ_EINVAL, "NULL argument");
    reps = std::max<uint32_t>(reps, 3);
    DeviceGuard g(ctx->device);
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : ctx->stream;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    CUDA_TRY(ctx, cudaEventCreate(&ev[0]));
    if (cudaEventCreate(&ev[1]) != cudaSuccess) {
        cudaEventDestroy(ev[0]);
        return fail(ctx, SSJ_EDEVICE, "cudaEventCreate");
    }
    // Candidate values per coordinate: the thread bin's upper key, the lane
    // bin's upper key (1: no lane bin), the warp bin's upper key (the largest
    // value sends no probe to the block bin) and the block size, which also
    // sets the block path's window (8 merge steps per thread).
    static const uint32_t kThread[] = {32, 64, 128, 256, 512, 1024, 2048, 4096};
    static const uint32_t kLane[] = {1, 256, 512, 1024, 2048};
    static const uint32_t kWarp[] = {256, 512, 1024, 2048, 4096, 0xFFFFFFFFu};
    static const uint32_t kBlock[] = {128, 256, 512, 128 | SSJ_WIDE_REGISTERS, 256 | SSJ_WIDE_REGISTERS,
                                      512 | SSJ_WIDE_REGISTERS, 256 | SSJ_BULK_STAGING, 512 | SSJ_BULK_STAGING,
                                      256 | SSJ_WIDE_REGISTERS | SSJ_BULK_STAGING,
                                      512 | SSJ_WIDE_REGISTERS | SSJ_BULK_STAGING};
    static const uint32_t kMinLive[] = {8, 12, 16, 20, 24};
    // index-item threshold: 0 sends no probe to index items (values above 480 count as 480)
    static const uint32_t kIndexMin[] = {0, 32, 64, 128, 256, 512};
    std::map<std::tuple<uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t>, float> seen;
    cudaError_t err = cudaSuccess;
    uint32_t bd = m->a.drain_min_live ? m->a.drain_min_live : 16;
    uint32_t bi = m->index_words_fit ? m->a.index_min_cands : 0u;
    auto cost = [&](uint32_t t, uint32_t l, uint32_t w, uint32_t b) -> float {
        auto key = std::make_tuple(t, l, w, b, bd, bi);
        auto it = seen.find(key);
        if (it != seen.end()) return it->second;
        const float v = time_setting(ctx, m, t, l, w, b, bd, bi, reps, s, ev, &err);
        seen[key] = v;
        return v;
    };
    uint32_t bt = m->a.thread_max_key, bl = m->a.lane_max_key, bw = m->a.warp_max_key, bb = m->block_threads;
    const float first = cost(bt, bl, bw, bb);
    float best = first;
    // coordinate descent: thread bin, lane bin, warp bin, block size; repeated while it improves
    for (int sweep = 0; sweep < 3 && err == cudaSuccess; ++sweep) {
        const float before = best;
        for (uint32_t t : kThread) {
            if (err != cudaSuccess) break;
            const uint32_t w = std::max(bw, t);  // a thread bin above the warp bin empties the latter
            const float v = cost(t, bl, w, bb);
            if (v < best) best = v, bt = t, bw = w;
        }
        for (uint32_t l : kLane) {
            if (err != cudaSuccess) break;
            if (l != 1 && l <= bt) continue;  // empty lane bin, same as 1
            const float v = cost(bt, l, bw, bb);
            if (v < best) best = v, bl = l;
        }
        for (uint32_t w : kWarp) {
            if (w < bt || err != cudaSuccess) continue;
            const float v = cost(bt, bl, w, bb);
            if (v < best) best = v, bw = w;
        }
        for (uint32_t b : kBlock) {
            if (err != cudaSuccess) break;
            const float v = cost(bt, bl, bw, b);
            if (v < best) best = v, bb = b;
        }
        for (uint32_t d : kMinLive) {
            if (err != cudaSuccess) break;
            const uint32_t keep = bd;
            bd = d;
            const float v = cost(bt, bl, bw, bb);
            if (v < best) best = v; else bd = keep;
        }
        for (uint32_t x : kIndexMin) {
            if (err != cudaSuccess || (x && !m->index_words_fit)) break;
            const uint32_t keep = bi;
            bi = x;
            const float v = cost(bt, bl, bw, bb);
            if (v < best) best = v; else bi = keep;
        }
        if (!(best < 0.98f * before)) break;  // no gain worth another sweep
    }
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    if (err != cudaSuccess) return cuda_fail(ctx, err, "autotune launch");
    uint32_t derr = 0;
    CUDA_TRY(ctx, cudaMemcpy(&derr, &m->a.ctr->err, sizeof(derr), cudaMemcpyDeviceToHost));
    if (derr) return fail(ctx, SSJ_EDEVICE, "device checks fired during tuning (code %u)", derr);
    // The multi keeps the best setting; a captured graph holds the old one.
    m->a.thread_max_key = bt;
    m->a.lane_max_key = bl;
    m->a.warp_max_key = bw;
    m->a.drain_min_live = bd;
    m->a.index_min_cands = bi;
    m->a.index_words = (bi || (m->batch_flags & SSJ_FORCE_INDEX)) ? m->index_words_fit : 0u;
    m->block_threads = bb;
    CUDA_TRY(ctx, prepare_verify(bb, m->a.index_words));
    if (m->exec) {
        cudaGraphExecDestroy(m->exec);
        m->exec = nullptr;
    }
    if (m->graph) {
        cudaGraphDestroy(m->graph);
        m->graph = nullptr;
    }
    out->thread_max_key = bt;
    out->lane_max_key = bl;
    out->warp_max_key = bw;
    out->block_threads = bb;
    out->drain_min_live = bd;
    out->index_min_cands = bi;
    out->best_ms = best;
    out->initial_ms = first;
    out->settings_tried = (uint32_t)seen.size();
    return SSJ_OK;
}

// ===========================================================================
// Read-bandwidth probe
// ===========================================================================

extern "C" ssj_status ssj_read_bandwidth(ssj_ctx* ctx, uint64_t bytes, uint32_t passes, double* gbs) {
    if (!ctx || !gbs) return fail(ctx, SSJ_EINVAL, "NULL argument");
    bytes &= ~uint64_t(15);
    if (bytes == 0 || passes == 0) return fail(ctx, SSJ_EINVAL, "bytes must be >= 16 and passes > 0");
    DeviceGuard g(ctx->device);
    void* buf = nullptr;
    cudaError_t e = cudaMalloc(&buf, bytes + 256);
    if (e != cudaSuccess) return fail(ctx, SSJ_ENOMEM, "cudaMalloc(%llu): %s", (unsigned long long)bytes,
                                      cudaGetErrorString(e));
    uint32_t* sink = reinterpret_cast<uint32_t*>(static_cast<char*>(buf) + bytes);
    cudaStream_t s = ctx->stream;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    e = cudaMemsetAsync(buf, 0, bytes + 256, s);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = read_probe(buf, bytes, 1, sink, ctx->num_sms, s);  // warm-up pass
    if (e == cudaSuccess) e = cudaEventRecord(e0, s);
    if (e == cudaSuccess) e = read_probe(buf, bytes, passes, sink, ctx->num_sms, s);
    if (e == cudaSuccess) e = cudaEventRecord(e1, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    float ms = 0;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaStreamSynchronize(s);
    cudaFree(buf);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "read probe");
    *gbs = ms > 0 ? (double)bytes * passes / (ms * 1e-3) / 1e9 : 0.0;
    return SSJ_OK;
}
