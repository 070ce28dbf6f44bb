// Internal declarations shared by the host API (api.cu, noalloc.cu) and the
// kernels (verify.cu).  Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/ssj.h"

namespace ssj {

enum : uint32_t {
    VF_COUNT_ONLY = 1u,
    VF_EMIT_ALL = 2u,
    VF_FORCE_THREAD = 4u,
    VF_FORCE_WARP = 8u,
    VF_FORCE_BLOCK = 16u,
    VF_SELF_JOIN = 32u,
    VF_FORCE_LANE = 64u,
    VF_FORCE_INDEX = 128u,
    VF_SORTED = 256u,
};

// One join instance of a launch: its collections, grouped candidate list,
// threshold and output.  A launch verifies any number of instances; the
// table of them lives in device memory (the workspace).
struct Instance {
    const uint4* r_rec[2];      // records of R and S for the two levels of the signature test
    const uint4* s_rec[2];
    const uint4* r_toks4;
    const uint2* r_desc;
    const uint4* s_toks4;
    const uint2* s_desc;
    const uint32_t* probe_ids;
    const uint64_t* cand_offsets;
    const uint32_t* cand_ids;
    ssj_triple* out;
    unsigned long long* count;  // result pairs of this instance (may exceed cap)
    uint64_t magic;             // div_magic(den) for Jaccard and Dice
    uint64_t n_cands;
    uint64_t cap;
    uint64_t chunk_base;        // first candidate chunk of this instance in the launch (VerifyArgs::chunk)
    uint64_t r_n_chunks, s_n_chunks;  // 16-byte blocks of the token arrays (bounds of the checked build)
    uint32_t r_n_sets, s_n_sets;
    uint32_t p, den;            // t = p / q; den: see SIM_*
    uint32_t n_probes;
    uint32_t tile_base;         // first plan tile (32 probes) of this instance
    uint32_t flags;             // VF_*
    uint32_t sim;               // SIM_*
    uint32_t rec_sectors[2];    // their sizes in 32-byte sectors; 0: no such level (no first: the length filter alone)
};

// A set's record: a header word (length in the upper 16 bits, loss in the
// lower: tokens that share a signature bit with another token of the set,
// |x| - popcount), and a bitmap of hash values of its tokens in the remaining
// bits.  A set of 65,535 tokens or more has length 65,535 and loss 0 there.
// Records of class c take 1 << c sectors of 32 bytes; a collection has the
// classes from 0 up to what its set sizes want, so that any two collections
// share some.
constexpr uint32_t kRecClasses = 4;
constexpr uint32_t rec_sectors(uint32_t c) { return 1u << c; }
constexpr uint32_t rec_bits(uint32_t c) { return rec_sectors(c) * 256u - 32u; }

// Similarity function of an instance, and what den / magic hold for it.
enum : uint32_t {
    SIM_JACCARD = 0,  // den = p + q, magic = div_magic(den)
    SIM_DICE = 1,     // den = 2q, magic = div_magic(den)
    SIM_COSINE = 2,   // den = q
    SIM_OVERLAP = 3,  // den = ceil(p / q), the required overlap itself
};

// Work item for lane- or block-per-pair verification: n queued pairs of
// probe set r starting at pair list index c0, in instance inst.  The warp
// list holds lane items (one lane per pair, r in shared memory).  In the
// block list, mode 0 is one thread block per pair, mode 1 an index item: the
// whole block holds r as a bitmap over the token values and every thread
// verifies one candidate at a time against it.
struct WorkItem {
    uint32_t r;
    uint32_t n;
    uint64_t c0;
    uint32_t inst;
    uint32_t pad;  // mode
};

// One queued pair: probe slot k (32 * its instance's tile_base + the probe's
// index) and candidate set id s.  Short pairs grow from the front of the pair
// list, the others from its back.
struct PairRef {
    uint32_t k;
    uint32_t s;
};
constexpr uint32_t kInItem = 0x80000000u;  // in s (set ids are below 2^31): a work item covers the pair

// Per-call counters, cleared by one memset before the plan kernel.
struct Counters {
    unsigned long long thread_pairs;  // short pairs queued at the front of the pair list
    unsigned long long long_pairs;    // other pairs, queued at its back
    unsigned long long warp_pairs;    // those of them that no work item covers
    unsigned long long warp_items;    // lane work items written by the plan kernel
    unsigned long long block_items;   // block work items written by the plan kernel
    uint32_t block_cursor;            // dynamic cursors of the verify kernel
    uint32_t warp_cursor;
    uint32_t long_cursor;
    uint32_t chunk_cursor;
    uint32_t probe_cursor;            // join kernel: probes taken
    unsigned long long candidates;    // join kernel: candidates found
    unsigned long long join_pairs, join_runs;  // and pairs and runs handed over
    unsigned long long results;       // result count of a synchronous call, read back with the rest
    uint32_t err;                     // device-side check bits (see ssj_device_error)
};

enum : uint32_t {
    ERR_PROBE_ID = 1u,
    ERR_CAND_ID = 2u,
    ERR_OFFSETS = 4u,
    ERR_GUARD = 8u,   // an internal loop bound was reached (a bug, reported instead of hanging)
    ERR_BOUNDS = 16u, // checked build (SSJ_CHECKED): an index was out of bounds; the access was skipped
};

// The checked build (-DSSJ_CHECKED, libssj_checked.so) tests the indexes with
// which the plan, verify, join and queue kernels read the batch, the
// collections, their records, the index and the pair lists, and write their
// buffers and lists, against each array's extent before the access; an index
// out of bounds sets ERR_BOUNDS and the access is skipped (a load reads zeros),
// so a bug shows as an error status, never as a fault.  (Not the kernels that
// lay a collection out, build its index, expand groups, scan and sort.)
#ifdef SSJ_CHECKED
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif

constexpr uint32_t kWarpItemCands = 8;   // candidates per entry that the warp list's capacity allows for
constexpr uint32_t kBlockItemCands = 16; // most candidates per block work item
constexpr uint32_t kLaneItemCands = 128; // most candidates per lane work item
constexpr uint32_t kLaneMinCands = 16;   // fewest candidates of a probe sent to the lane bin
constexpr uint32_t kWarpRCap = 1024;     // r kept whole in a warp's shared memory up to this
constexpr uint32_t kPlanFlush = 480;     // pairs left that a plan warp queues at once
constexpr uint32_t kIndexMaxWords = 24576;  // largest probe bitmap (32-bit words, 96 KiB): token values below 786,432

// Kernel arguments of one launch (passed by value).
struct VerifyArgs {
    Instance single;              // the instance of a one-batch launch (table == nullptr)
    const Instance* table;        // device table of n_inst instances, or nullptr
    Instance* table_out;          // where the plan kernel stores `single` for the verify kernel
    uint32_t n_inst;
    uint32_t n_tiles;             // plan tiles over all instances
    uint32_t total_probes;        // probe slots over all instances (instance-major)
    uint32_t chunk;               // candidates per plan chunk (a warp's unit of work)
    uint64_t n_chunks;            // over all instances
    uint64_t chunk_begin;         // a plan launch of one piece: its first chunk (n_chunks: after its last)
    uint64_t total_cands;
    Counters* ctr;
    PairRef* pairs;               // pairs left to verify: short ones from the front, others from the back
    WorkItem* warp_items;
    WorkItem* block_items;
    uint64_t pair_cap;
    uint32_t warp_item_cap, block_item_cap;
    uint32_t block_item_cands;    // candidates per work item
    uint32_t lane_item_cands;
    uint32_t thread_max_key;      // 2|r| <= this: one thread per pair
    uint32_t lane_max_key;        // 2|r| <= this (and r fits, >= kLaneMinCands candidates): one lane per pair
    uint32_t warp_max_key;        // 2|r| <= this: one warp per pair; above: one block
    uint32_t drain_min_live;      // short-pair pass 2 re-parks below this many live lanes (0: default 16)
    uint32_t index_words;         // probe bitmap words (every token value of the launch's collections below
                                  // 32 * index_words); 0: no index items
    uint32_t index_min_cands;     // runs of at least this many pairs become index items (0: none; see probe_bin)
    uint32_t bulk_stage;          // block and warp items stage sets by bulk copies (cp.async.bulk)
    uint32_t force_thread;        // an instance asks for one thread per pair (VF_FORCE_THREAD)
    // host side only: an L2 access-policy window (persisting) for the verify kernel's launch, or none
    const void* l2_base;
    uint64_t l2_bytes;
    float l2_hit_ratio;
};

// Bitmap words for index items over collections whose token values are all
// below vocab_bound (0 when that exceeds kIndexMaxWords); a multiple of 4.
inline uint32_t index_words_for(uint64_t vocab_bound) {
    const uint64_t w = ((vocab_bound + 31) / 32 + 3) & ~3ull;
    return (w == 0 || w > kIndexMaxWords) ? 0u : (uint32_t)w;
}

// Sizes of one launch, from which the workspace is carved.
struct LaunchShape {
    uint32_t n_inst;
    uint32_t n_tiles;
    uint32_t total_probes;
    uint64_t total_cands;
    uint64_t n_chunks;  // plan chunks over all instances (plan_chunk, chunks_of)
};

// Candidates per plan chunk of a launch, and the chunks of one instance.
uint32_t plan_chunk(uint64_t total_cands, int num_sms);
// Chunks that one wave of the plan kernel works on.
inline uint64_t plan_wave(int num_sms) { return 32ull * (uint64_t)num_sms; }
inline uint64_t chunks_of(uint64_t n_probes, uint64_t n_cands, uint32_t chunk) {
    return n_probes ? (n_cands + chunk - 1) / chunk : 0;
}

// Scratch a launch of this shape needs, in bytes, on a device with num_sms SMs.
size_t workspace_bytes(const LaunchShape& sh, int num_sms);
// Shape of a one-batch launch.
LaunchShape single_shape(uint32_t n_probes, uint64_t n_cands, int num_sms);
size_t workspace_bytes(uint32_t n_probes, uint64_t n_cands, int num_sms);

// Carve the workspace and fill the scratch pointers of a.
void bind_workspace(VerifyArgs& a, void* ws, const LaunchShape& sh, int num_sms);
void bind_workspace(VerifyArgs& a, void* ws, uint32_t n_probes, uint64_t n_cands, int num_sms);

// block_threads flag selecting the verify kernel variant compiled for three
// quarters of the CTAs per SM (more registers per thread, fewer spills).
constexpr uint32_t kWideRegisters = SSJ_WIDE_REGISTERS;
// block_threads flag: block and warp items stage the sets by bulk copies.
constexpr uint32_t kBulkStaging = SSJ_BULK_STAGING;

// Set the verify kernel's launch attributes for this device (done by the
// first launch anyway; call before capturing a launch into a graph).
cudaError_t prepare_verify(uint32_t block_threads, uint32_t index_words = 0);

// Enqueue the whole verification (counter clear, plan, verify) on st.
// ev (optional, 3 events): recorded before the plan kernel, between plan and
// verify, and after the verify kernel, on st.
cudaError_t launch_verify(const VerifyArgs& a, cudaStream_t st, int num_sms, uint32_t block_threads,
                          cudaEvent_t* ev = nullptr);
cudaError_t launch_plan(const VerifyArgs& a, cudaStream_t st, int num_sms);
cudaError_t launch_merge(const VerifyArgs& a, cudaStream_t st, int num_sms, uint32_t block_threads);

// Sort the triples of the instances that ask for it (VF_SORTED) and have at
// most kSortTile of them, on st.
constexpr uint32_t kSortTile = 4096;
cudaError_t sort_results(const Instance* table, uint32_t n_inst, cudaStream_t st);
// The instances' triples side by side in packed, complete if they all fit.
cudaError_t pack_results(const Instance* table, uint32_t n_inst, ssj_triple* packed, uint64_t room, cudaStream_t st);
// Sort n triples by (r, s) with room for n more at tmp.
cudaError_t sort_triples(ssj_triple* t, uint64_t n, ssj_triple* tmp, cudaStream_t st);

// Records of class c (rec_bits) of a laid-out collection, on st.
cudaError_t build_records(const uint4* toks4, const uint2* desc, uint32_t n, uint32_t c, uint4* rec, cudaStream_t st,
                          int num_sms);

// Exclusive prefix sums of n 64-bit values each of `arrays` arrays, the k-th at
// data + k * stride, in place on st; total[k] (device) receives the sum.
// scratch holds arrays * scan_scratch_words(n) values.  copy (optional, one
// array) receives the sums too.
size_t scan_scratch_words(uint64_t n);
cudaError_t exclusive_scan_u64(uint64_t* data, uint64_t n, uint64_t* scratch, uint64_t* total, cudaStream_t st,
                               uint64_t* copy = nullptr, uint32_t arrays = 1, uint64_t stride = 0);

// Self-join on the device (candgen.cu).  Scratch of the prefix index, sized by
// the caller: size_hist max_len + 2 words and toff candgen_cells + 1 words, one
// after the other (toff_at), probes and rank n each, tcnt as toff, scan_scratch
// scan_scratch_words(max(max_len + 2, candgen_cells + 1)), total 1 word, post
// candgen_entry_bytes per index entry (known after stage 0).
inline uint64_t candgen_toff_at(uint32_t max_len) { return ((uint64_t)max_len + 2 + 15) / 16 * 16; }
struct CandgenIndex {
    uint64_t* size_hist;          // after stage 0: per size, the position after its last set
    uint32_t* probes;             // the sets from the largest down
    uint32_t* rank;
    uint64_t* tcnt;
    uint64_t* toff;
    uint64_t* scan_scratch;
    uint64_t* total;
    void* post;
    uint64_t entries;             // index entries (after stage 0)
};

// A token's index entries are kept in cells by position: as many (a power of
// two, at most 64) as make at most two million for the vocabulary.  More cells
// skip more entries but their bounds take longer to clear and sum: a join of
// long sets (100,000 tokens) takes 844 us with one cell per token, 543 at one
// million cells, 516 at two, 533 at four, 589 at eight; of short sets (530,000
// tokens) 415, 408, 394, 405, 423.
inline uint32_t candgen_cells_log2(uint32_t vocab) {
    uint32_t b = 0;
    while (b < 6 && ((uint64_t)vocab << (b + 1)) <= (1ull << 21)) ++b;
    return b;
}
inline uint64_t candgen_cells(uint32_t vocab) { return (uint64_t)vocab << candgen_cells_log2(vocab); }
inline uint32_t candgen_cell_shift(uint32_t n, uint32_t cells_log2) {
    uint32_t bits = 0;
    while (bits < 32 && ((uint64_t)n > (1ull << bits))) ++bits;
    return bits > cells_log2 ? bits - cells_log2 : 0u;
}

// Bytes of an index entry.
inline size_t candgen_entry_bytes(bool positional) { return positional ? 16 : 8; }

struct CandgenInput {
    const uint4* toks4;
    const uint2* desc;
    uint32_t n, max_len, vocab;   // vocab: largest token + 1
    uint32_t sim, p, q;           // SIM_*, t = p/q
    uint32_t positional;          // positional bound at the matching prefix token
    int stage;                    // 0: order + token counts; 1: token lists
};

// Run one stage on st.  Stage 0 waits for it and leaves the number of index
// entries in *host_word (pinned).
cudaError_t candgen_run(const CandgenInput& in, cudaStream_t st, int num_sms, CandgenIndex* ix,
                        uint64_t* host_word);

// Pairs that the join kernel hands over to the queue kernel, in runs of up to
// kJoinRun in probe order: (first pair, pairs).
constexpr uint32_t kJoinRun = 288;
struct JoinQueue {
    uint2* pairs;  // (index of the probe, candidate set)
    ulonglong2* runs;
    uint64_t pair_cap, run_cap;
};

// Clear the counters and probe the index (after stage 1): candidates left by
// the signature test are queued in a's lists for launch_merge, a.single being
// the self-join with ix.probes as its probes.  If Counters::join_pairs
// exceeds out.pair_cap, nothing is queued.
cudaError_t join_probe(const CandgenInput& in, const CandgenIndex& ix, const VerifyArgs& a, const JoinQueue& out,
                       cudaStream_t st, int num_sms);

// Room for a self-join's queues of up to `pairs` pairs over n probes, and its
// carving.
size_t join_workspace_bytes(uint32_t n_probes, uint64_t pairs, int num_sms);
JoinQueue bind_join_workspace(VerifyArgs& a, void* ws, uint32_t n_probes, uint64_t pairs, int num_sms);

// GroupJoin expansion on the device (candgen.cu).  Entries: the probe
// groups, then every group (pairs inside it).  probe_off and pair_off hold
// n_entries + 1 words each, one after the other; per_probe n_entries;
// scan_scratch 2 * scan_scratch_words(n_entries + 1); total two words.
struct GroupExpand {
    const uint4* toks4;
    const uint2* desc;
    uint32_t sim, p, q;
    const uint64_t* group_offsets;
    const uint32_t* members;
    const uint32_t* probe_groups;
    const uint64_t* cand_offsets;
    const uint32_t* cand_groups;
    uint32_t n_groups, n_probe_groups;
    uint64_t* probe_off;
    uint64_t* pair_off;
    uint64_t* per_probe;
    uint64_t* scan_scratch;
    uint64_t* total;
    int stage;                 // 0: count and scan; 1: write
    uint32_t* probe_ids;       // stage 1 outputs: the expanded grouped batch
    uint64_t* cand_offsets_out;
    uint32_t* cand_ids;
};

// Stage 0 waits and leaves (expanded probes, expanded pairs) in
// host_words[0..1] (pinned); stage 1 enqueues the writes.
cudaError_t expand_groups(const GroupExpand& x, cudaStream_t st, int num_sms, uint64_t* host_words);

// One launch of the read-bandwidth probe: `passes` sweeps over bytes (a
// multiple of 16) at buf, on st; sink is a device word the kernel may write.
cudaError_t read_probe(const void* buf, uint64_t bytes, uint32_t passes, uint32_t* sink, int num_sms,
                       cudaStream_t st);

}  // namespace ssj
