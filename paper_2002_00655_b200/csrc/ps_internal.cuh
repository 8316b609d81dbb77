// Internal declarations shared by the translation units of the library.
// Nothing here is part of the public interface (see include/ps.h).
#pragma once

#include <atomic>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ps.h"

namespace psb {

constexpr uint32_t kSentinelPad = 0xFFFFFFFFu;   // never a key: num_keys < 2^32 - 1
constexpr int kSortTile = 2048;                  // the sort's counters have room for a block per half of this
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kMaxSortPasses = 4;                // 32-bit keys
constexpr int kSortCtlWords = kMaxSortPasses * kRadix + kMaxSortPasses;   // digit histograms of every pass, then tickets
constexpr int kReduceTile = 32;                  // sorted occurrences per warp in the segmented reduction of long rows
constexpr uint32_t kTiledRow = 512;              // ... rows up to this many values: 8 to 128 (reduce_tile)
constexpr uint32_t kMidTiles = 4096;             // shorter tiles than 32 positions that a call has at most
constexpr int kMaxLossBlocks = 4096;
constexpr uint32_t kSmallOcc = 8192;             // calls of at most this many key occurrences are reduced without a sort (small.cu; steps on wide rows: small_step, small_sgns)
constexpr uint32_t kMaxHot = 8;                  // keys of such a call that all blocks share, at most
constexpr uint32_t kHotStretches = 128;          // ... on rows of at most this many stretches of columns
constexpr int kHostStages = 3;                   // staging areas for batches that arrive from host memory
constexpr int kSortSets = 4;                     // calls whose key sort may be in flight at once (see SortSet)
constexpr int kSideStreams = 3;                  // internal streams that calls with a long sort take in turn

// Device-resident status words.  An error is latched per call with the call's
// epoch, so no kernel has to clear anything before a call starts.
struct DevStatus {
    unsigned int sticky;            // first error code since the last ps_sync
    unsigned int call_err_epoch[4]; // number of the last sorting call with that number mod 4 that failed on the device
                                    // (up to kSortSets such calls of one handle are in flight: later ones' sorts
                                    // beside the current one's kernels; only calls that take a buffer set are numbered)
    unsigned int moved_total;       // localize: number of keys that move in the current call
    unsigned int deferred_now;      // ... of which wait for the call that runs beside the relocation (ps_localize_beside)
    unsigned long long rows_moved;  // rows relocated by all successful localize calls so far
    unsigned long long loc_requested;       // keys handed to localize calls, repeats included
    unsigned long long loc_already_local;   // distinct keys per call that the requester owned already
    unsigned long long loc_moved_again;     // moved keys that had left their initial partition before (taken from a
                                            // worker that had localized them: localization conflicts, Section 3.2)
    unsigned long long loc_deferred;        // moved keys that had to wait for the call running beside the relocation
};

// clusters of a kernel that are resident at once, for the launch shape last asked about
struct ClusterFit {
    const void* fn;
    size_t smem;
    uint32_t threads, blocks, clusters;
};

static_assert(kSortSets <= 4, "one error-epoch word per call in flight");

struct Profile;

// One of the kSortSets sets of buffers the key sort and the segment bookkeeping work in.  Calls rotate
// through the sets so that the sorts of the next steps can run while earlier steps are still reducing.
struct SortSet {
    uint32_t *keysA, *keysB, *valsA, *valsB;
    uint32_t* tile_state;
    uint32_t* sort_ctl;
    unsigned int* group_done;
    uint4* rec;
    uint32_t* cellpos;
    uint4* starters;
    unsigned int* starter_count;
    uint4* mf_dup;
    unsigned int* mf_tickets;
    cudaEvent_t ev_free;            // recorded after the last kernel that used the set
    bool used;
    bool loc_reader;                // a relocation on another stream reads this set's sorted keys (ps_localize_beside)
    int sorted_which;               // which key buffer holds the call's sorted keys (-1: the call sorted none)
    uint32_t sorted_n;
    uint32_t run_base, run_len;     // sorted keys from run_base on stand for run_len consecutive keys (RESCAL: a matrix's rows)
};

}  // namespace psb

struct ps_store {
    ps_config_t cfg;
    uint64_t max_keys;
    int key_bits;                   // bits needed for keys 0..K inclusive (K is the "no key" mark)
    uint32_t sort_blocks_cap;       // blocks the sort's digit counters (tile_state) have room for
    int owner_bits;
    // caller-owned device buffers
    float* store;
    uint2* table;                   // (owner, slot) per key
    unsigned long long* tops;       // N stack heights
    uint32_t* stacks;               // N x S
    char* ws;
    size_t ws_bytes;
    // carved out of the workspace
    psb::DevStatus* status;
    uint32_t *keysA, *keysB, *valsA, *valsB;
    uint32_t* tile_state;           // kMaxSortPasses x sort blocks x kRadix digit counters
    uint32_t* sort_ctl;             // the sort's grid barrier (two words) in kSortCtlWords, followed by group_done
    uint4* rec;                     // MF: {cell, cell value, row of the key, row of the other factor} per sorted position
    uint32_t* cellpos;              // MF: sorted position of each cell's row-factor occurrence
    uint4* mf_dup;                  // MF by column: per column position {first position, count, rank} of its cell's row key
    unsigned int* mf_tickets;       // MF by column: a ticket counter per row-side position, then one per block, then one
    unsigned int* group_done;       // per group of 64 reduction tiles: reduction blocks that have finished
    double* group_sum;              // per group: pre-added parked parts of the segment entering it (row_len)
    uint32_t* scan_sums;            // block sums of the device-wide scan
    uint32_t* loc_counts;           // localize: moving keys per block (512 words), then per block and old owner
    uint32_t* loc_scratch;          // localize: five words per key of the call (old and new places of the moving keys)
    float* upd;                     // max_keys x row_len update rows (also localize scratch)
    double* carry;                  // nReduceTiles x 2 x row_len partial sums of segments that span tiles
    uint4* starters;                // {tile, key, row} of the tiles that start a border-crossing segment
    unsigned int* starter_count;
    unsigned int* hot_tickets;      // calls without a sort: per stretch of columns and hot key, zero between calls
    uint32_t tile_cap;              // tiles that carry and starters have room for
    double* loss_partial;           // max(kMaxLossBlocks, one per 256 key occurrences)
    uint64_t* apply_rows;           // per sorted position: address of the row staged there, or all ones
    char* staging;                  // host-batch staging, max_keys x 8 bytes (the first of `stagings`)
    char* stagings[psb::kHostStages];
    // host state
    uint32_t epoch;
    uint64_t launches;
    int sm_count;
    psb::Profile* prof;             // per-kernel event timing, off unless ps_profile_start was called
    cudaStream_t side;              // key extraction and sort of the current call run here, beside the gradient kernel:
    cudaStream_t sides[psb::kSideStreams];  // one of these; calls whose sort is longer than the rest of the step take them
    int side_idx, side_alt;         // in turn, so that the sorts of several later steps run beside each other
    unsigned long long side_capture_id[psb::kSideStreams];  // graph capture each of them was last forked into (0 = none)
    cudaEvent_t ev_fork, ev_join;
    psb::SortSet sets[psb::kSortSets];           // keysA .. starter_count above always point into sets[cur_set]
    int cur_set;
    cudaStream_t copy;              // host batches are copied here in overlapped mode (ps_set_host_overlap)
    cudaEvent_t ev_copied[psb::kHostStages], ev_consumed[psb::kHostStages];
    bool consumed_valid[psb::kHostStages];
    int host_slot;
    bool host_overlap;
    cudaEvent_t batch_ready;        // set while a call's batch is still on its way: the side stream waits for it
    bool pipelined;                 // see ps_set_pipelining
    CUtensorMap row_map;            // the store as a 2-D tensor (row_len x rows, one row per box) for row gathers by the TMA unit
    bool row_map_ok;
    int mf_path;                    // see ps_set_mf_path
    psb::SortSet* last_set;         // the most recent call's buffer set if that call sorted its keys (else null)
    cudaStream_t last_stream;       // the stream of the most recent call
    cudaEvent_t ev_before, ev_sorted;       // most recent sorting call: the caller's stream before its first kernel; after its sort
    cudaEvent_t ev_loc;             // end of the most recent ps_localize_beside
    bool loc_pending;               // ... which later calls still have to be ordered after
    int push_mode;                  // see ps_set_push_mode
    bool table_dirty[psb::kSideStreams];   // per side stream: the location table was rewritten since that stream last waited
                                    // for the caller's (a sort that reads the table must not start before the rewrite)
    unsigned long long capture_id;  // graph capture the caller's stream was in at the last step call (0 = none)
    psb::ClusterFit kge_fit;
};

namespace psb {

struct WsLayout {
    size_t status, keysA[kSortSets], keysB[kSortSets], valsA[kSortSets], valsB[kSortSets], tile_state[kSortSets],
        sort_ctl[kSortSets], rec[kSortSets], cellpos[kSortSets], mf_dup[kSortSets], mf_tickets[kSortSets], scan_sums, loc_counts, loc_scratch, upd, carry, group_sum, starters[kSortSets], starter_count[kSortSets],
        loss_partial, apply_rows, hot_tickets, staging[kHostStages], total, reduce_tiles;
};
WsLayout ws_layout(const ps_config_t& cfg, uint64_t max_keys);

inline uint32_t div_up_u32(uint64_t a, uint64_t b) { return (uint32_t)((a + b - 1) / b); }

// The opt-in to more than 48 KB of dynamic shared memory is a per-DEVICE attribute of a kernel: `done` keeps one
// bit per device ordinal (a static of the launch site), so every GPU the process uses gets the attribute once.
inline void opt_in_smem(const void* fn, size_t bytes, std::atomic<unsigned long long>* done) {
    int d = -1;
    const bool known = cudaGetDevice(&d) == cudaSuccess && d >= 0 && d < 64;
    if (known && ((done->load(std::memory_order_relaxed) >> d) & 1ull)) return;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (known) done->fetch_or(1ull << d, std::memory_order_relaxed);
}
template <class T> __host__ __device__ inline T tmin(T a, T b) { return a < b ? a : b; }
template <class T> __host__ __device__ inline T tmax(T a, T b) { return a > b ? a : b; }

// ---- ps_api.cu: optional per-kernel timing ----
void prof_before(ps_store* ps, const char* name, cudaStream_t s);
void prof_after(ps_store* ps, cudaStream_t s);

#define PS_LAUNCH(ps, kernel, grid, block, stream, ...)                       \
    do {                                                                     \
        if ((ps)->prof) psb::prof_before((ps), #kernel, (stream));           \
        kernel<<<(grid), (block), 0, (stream)>>>(__VA_ARGS__);               \
        if ((ps)->prof) psb::prof_after((ps), (stream));                     \
        (ps)->launches++;                                                    \
    } while (0)

#define PS_LAUNCH_SMEM(ps, kernel, grid, block, smem, stream, ...)            \
    do {                                                                     \
        if ((ps)->prof) psb::prof_before((ps), #kernel, (stream));           \
        kernel<<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);          \
        if ((ps)->prof) psb::prof_after((ps), (stream));                     \
        (ps)->launches++;                                                    \
    } while (0)

// Programmatic dependent launch, for the kernels of small calls: the kernel may be set up while the one before it on the
// stream still runs, as soon as all blocks of that one have passed pdl_trigger(); it touches no memory before pdl_wait(),
// which returns when everything before has completed.  Takes a launch's latency (a microsecond or two) off each of a
// chain of kernels that run a few microseconds.  Without a trigger in the kernel before it is an ordinary launch.
// What such a kernel reads may be written while it is already on the chip: none of it is passed as `const __restrict__`, which
// would let the compiler read it through the read-only path and before the wait.
template <class... P, class... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#define PS_LAUNCH_PDL(ps, name, kernel, grid, block, smem, stream, ...)        \
    do {                                                                     \
        if ((ps)->prof) psb::prof_before((ps), name, (stream));              \
        psb::launch_pdl(kernel, (grid), (block), (smem), (stream), __VA_ARGS__); \
        if ((ps)->prof) psb::prof_after((ps), (stream));                     \
        (ps)->launches++;                                                    \
    } while (0)

// ---- sort.cu ----
// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the key, one cooperative launch.
// Values are the positions 0..n-1 of the input.  Input in the A buffers (start = 0) or the B buffers
// (start = 1).  If n_dev is not null the element count is read from device memory (n is then an upper
// bound used for the launch shape).  Returns 0 if the result is in the A buffers, 1 if in the B buffers.
// Before its first grid barrier the kernel clears *zero_me (if not null) and the first `zero_groups`
// words of group_done.
int radix_sort_pairs(ps_store* ps, uint32_t n, const unsigned int* n_dev, int bits, cudaStream_t stream, int start,
                     unsigned int* zero_me, uint32_t zero_groups);
// the same on range-checked 64-bit caller keys (no separate key kernel); key_bits bits
int radix_sort_keys64(ps_store* ps, const uint64_t* d_keys, uint32_t n, cudaStream_t stream, unsigned int* zero_me,
                      uint32_t zero_groups);
// the 2 n_cells occurrences of a batch of matrix cells (2t: row factor, 2t + 1: column factor), keys taken
// from the batch arrays inside the sort; with `records` the last pass writes ps->rec beside the sorted keys
int radix_sort_mf(ps_store* ps, const uint32_t* d_i, const uint32_t* d_j, const float* d_v, uint32_t n_cells,
                  uint64_t col_key_base, bool records, cudaStream_t stream, unsigned int* zero_me,
                  uint32_t zero_groups);

// ---- pull_push.cu ----
uint32_t reduce_tile(const ps_store* ps, uint32_t n, bool scaled);      // positions per tile of a push of n occurrences
uint32_t reduce_groups(const ps_store* ps, uint32_t n);                 // groups of 64 tiles, at most
void launch_init_range_partition(ps_store* ps, cudaStream_t s);
void launch_set_rows(ps_store* ps, const uint64_t* d_keys, uint64_t n, const float* d_vals, cudaStream_t s);
void launch_pull(ps_store* ps, const uint64_t* d_keys, uint64_t n, float* d_out, cudaStream_t s);
void launch_get_location(ps_store* ps, const uint64_t* d_keys, uint64_t n, uint32_t* d_owner, uint32_t* d_slot,
                         cudaStream_t s);
void launch_gather_rows_by_key(ps_store* ps, uint64_t first_key, uint64_t n, float* d_out, cudaStream_t s);
// sort keysA (values = occurrence index; returns which buffer holds the result), then reduce `upd` rows per key, apply them
// to the store, and add the first `loss_blocks` loss partials to *d_loss_accum (if not null).  With d_scales, occurrence
// o contributes d_scales[o] times a shared source row of d_upd: row 2e for slot 0 of example e = o / slots, row 2e + 1
// for its other slots.
int run_push_sort(ps_store* ps, uint32_t n, cudaStream_t s);
int run_segment_sort(ps_store* ps, uint32_t n, cudaStream_t s);     // the same; also clears the counters of seg_lists
void run_push_reduce(ps_store* ps, uint32_t n, int which, const float* d_upd, double* d_loss_accum,
                     uint32_t loss_blocks, cudaStream_t s, const float* d_scales = nullptr, uint32_t slots = 0,
                     bool skip_singles = false);        // keys that occur once have been updated already

// push by atomic adds, no sort (ps_set_push_mode)
void run_push_atomic(ps_store* ps, const uint64_t* d_keys, uint64_t n, const float* d_upd, cudaStream_t s);

// MF step working on the sorted occurrences directly (rows of at most 512 values): gradient, reduction,
// then the fix-up launch that also moves the staged rows into the store
void run_mf_fused(ps_store* ps, uint32_t n_cells, int which, uint64_t col_key_base, float lr, float lambda,
                  double* d_loss_accum, cudaStream_t s, bool gather4);
// ---- mf_col.cu ----
// MF step as one launch over the column side of the sorted occurrences (rows of at most 128 values).  launch_mf_plan
// goes on the stream the sort ran on, right after it; run_mf_col on the caller's stream after the join.
void launch_mf_plan(ps_store* ps, uint32_t n_cells, int which, cudaStream_t side);
void run_mf_col(ps_store* ps, uint32_t n_cells, int which, float lr, float lambda, double* d_loss_accum, cudaStream_t s);

// ---- small.cu ----
// Calls of at most kSmallOcc key occurrences, all on the caller's stream, no sort.  The step's gradient kernel leaves the
// slots' keys in small_keys (num_keys: no key; kSentinelPad: index out of range) and its rows in ps->upd, as for the
// sorted reductions.
inline bool small_call(uint64_t n_occ) { return n_occ <= kSmallOcc; }
// ComplEx and skip-gram on wide rows sort even fewer occurrences than that: a sort costs 12 to 25 us however wide the rows are; without
// one every gradient is written out and read again, with one most rows are updated in place and the reduction is tiled.  One limit for
// ordered and pipelined handles, whose results are the same bits, and it lies where a pipelined handle, whose sorts run beside
// other calls, breaks even (between 1.5 and 2.0M; an ordered one would at about 3M).
// ComplEx (dim complex dimensions): no sort up to kSmallValues dimensions of all occurrences.  us per step, ordered without and with a sort,
// pipelined without and with, 10 negatives: 476 data points of 250 dimensions (1.55M) 39.0 56.3, 39.1 39.0, 615 of 250 (2.0M) 52.3 66.4,
// 52.0 49.8; 238 of 500 37.1 57.4, 37.2 43.9, 307 of 500 48.9 61.4, 48.7 46.3, 461 of 500 (3.0M) 66.2 71.1, 66.1 55.9; 119 of 1,000
// 34.7 50.1, 34.8 37.6, 153 of 1,000 48.3 59.3, 48.4 45.8.  Odd dimensions, whose gradients are written out as finished steps: 297 of
// 401 (1.55M) 55.2 60.6, 55.0 45.7, 383 of 401 (2.0M) 82.0 64.8, 81.8 49.2.
// Pushes and matrix factorization gain nothing from a sort (8,000 rows of 1,024 values: 64 / 87).
constexpr uint64_t kSmallValues = 1600000;
inline bool small_step(uint64_t n_occ, uint64_t dim) { return small_call(n_occ) && n_occ * dim <= kSmallValues; }
// Skip-gram (rows of row_len values, slots per center): a sort from 5,001 occurrences and kSmallValues values on, if a center has 26 to
// 48 slots.  With fewer the gradient kernel is too short to cover a sort, with more it is most of the step either way.  us per step as
// above: rows of 512 values, 13 slots (window 2, 2 negatives): 7,000 occurrences 34 41, 34 37; 25 slots 39 36, 39 37; 31 slots 47 40, 47
// 42; 41 slots (window 5, 3 negatives) 4,900 occurrences 45 42, 44 44, 7,000 53 44, 53 46; 61 slots 54 53, 53 57; 113 slots 71 72,
// 71 78.  Rows of 300: 41 slots 4,000 occurrences 31 34, 31 37, 6,600 41 36, 41 38.
constexpr uint64_t kSgnsSortOcc = 5000, kSgnsSortFrom = 26, kSgnsSortTo = 48;
inline bool small_sgns(uint64_t n_occ, uint64_t row_len, uint64_t slots) {
    return small_step(n_occ, row_len) || (small_call(n_occ) && (n_occ <= kSgnsSortOcc || slots < kSgnsSortFrom || slots > kSgnsSortTo));
}
uint32_t* small_keys(ps_store* ps);
void run_small_push_keys(ps_store* ps, const uint64_t* d_keys, uint32_t n, const float* d_upd, cudaStream_t s);
void run_small_reduce(ps_store* ps, uint32_t n, double* d_loss_accum, uint32_t loss_blocks, cudaStream_t s,
                      const float* d_scales = nullptr, uint32_t slots = 0);
void run_small_adagrad(ps_store* ps, uint32_t n, float lr, float eps, double* d_loss_accum, uint32_t loss_blocks,
                       cudaStream_t s, const double* loss_terms = nullptr);     // null: ps->loss_partial

// ---- segments.cu ----
constexpr uint32_t kRelPiece = 8;                // data points of one relation that a block of rescal_points_kernel takes, at most
constexpr uint32_t kRelChunk = 64;               // ... that a block of rescal_matrix_kernel sums before parking
constexpr uint32_t kRelTickets = 16;             // ticket words per chunk of a relation of several chunks
constexpr uint32_t kRelGroup = 8;                // ... chunks whose sums are added before they meet the others
struct SegLists {
    unsigned int* counts;           // entries of shorts, longs, pieces, chunks; partial sums parked; what warps have drawn
    uint8_t* single;                // per occurrence
    uint2 *shorts, *pieces;         // {first position, length}
    uint32_t short_room;            // entries `shorts` has room for
    uint4 *longs, *chunks;          // {first position, length, the segment's first parked sum, piece | pieces << 16}
    unsigned int *tickets, *long_tickets;
    uint32_t strips;                // long_tickets per parked sum
};
constexpr uint32_t kSegMediums = 8 + 64, kSegCounters = kSegMediums + 1;        // lengths and single keys drawn (rows whose single keys are reduced have at most two stretches of columns); short segments drawn, by stretch; medium ones
SegLists seg_lists(ps_store* ps);   // of the current buffer set
const uint8_t* launch_singles(ps_store* ps, uint32_t n, int which, cudaStream_t s);     // per occurrence: its key occurs once
// after the sort, on its stream; keys from rel_key_base on are RESCAL's relations (num_keys: none), of n_points data points
void launch_segments(ps_store* ps, uint32_t n, int which, uint32_t half_row, uint64_t rel_key_base, uint32_t n_points, cudaStream_t s);
uint32_t rel_piece_len(uint32_t d);     // data points per piece of a relation's run: 8, or 4 for small matrices
// gradient rows (half_row values per occurrence, in ps->upd) -> AdaGrad, of the keys that occur several times and, with
// singles, of those that occur once; loss terms.  parked: room for the long segments' partial sums.  beside: the kernel before
// it on the stream has triggered it, is still running, and touches none of what this one does
void run_segment_adagrad(ps_store* ps, uint32_t n, int which, uint32_t half_row, bool singles, float lr, float eps,
                         double* parked, const double* loss_terms, uint32_t n_loss, double* d_loss_accum, cudaStream_t s, bool beside = false);

// ---- complex.cu ----
struct KgeBatch {
    const uint32_t *s, *r, *o, *neg_ent;
    const uint8_t* neg_side;
    uint64_t n;
    uint32_t n_neg;
    uint64_t rel_key_base;
    uint32_t dim;
    float lr, eps;
};
void launch_keys_kge(ps_store* ps, const KgeBatch& B, cudaStream_t s);
// single: per slot, does its key occur once in the batch (such rows are updated in place).  Gradient rows of 2 dim values
// per slot in ps->upd (finished: rows of 4 dim values, step and squared gradient).  Returns the number of loss partials.
uint32_t launch_points_kge(ps_store* ps, const KgeBatch& B, const uint8_t* single, bool finished, uint32_t* keys_out, cudaStream_t s);

// ---- rescal.cu ----
struct RescalBatch {
    const uint32_t *s, *r, *o, *neg_ent;
    const uint8_t* neg_side;
    uint64_t n;
    uint32_t n_neg;
    uint64_t rel_key_base;
    uint32_t dim;
    float lr, eps;
};
void launch_keys_rescal(ps_store* ps, const RescalBatch& B, cudaStream_t s);    // 3 + n_neg slots per data point
// Return where the data points' loss terms are.  small: gradient rows and keys of all 2 + n_neg + dim slots; sorted:
// matrices and keys that occur once are updated, gradient rows of the other entity slots written.
const double* run_rescal_small(ps_store* ps, const RescalBatch& B, uint32_t* keys_out, cudaStream_t s);
void run_rescal_sorted(ps_store* ps, const RescalBatch& B, int which, uint32_t n_loss, double* d_loss_accum, cudaStream_t s);

// ---- localize.cu ----
// busy_keys: sorted keys of a call that may run beside this relocation (null: none); moving keys among them keep
// table entry and row until run_localize_deferred, which the caller enqueues once that call is through.
struct BusyKeys {
    const uint32_t* keys;
    uint32_t n, run_base, run_len;      // as in SortSet
};
void run_localize(ps_store* ps, uint32_t worker, uint32_t n, int which, cudaStream_t s, BusyKeys busy = {nullptr, 0u, 0u, 1u});
// Few keys: the whole call, without a sort, in one launch on the caller's stream.
bool localize_is_small(const ps_store* ps, uint64_t n);
void run_localize_small(ps_store* ps, uint32_t worker, const uint64_t* d_keys, uint32_t n, cudaStream_t s);
void run_localize_deferred(ps_store* ps, uint32_t worker, uint32_t n, cudaStream_t s);

// ---- steps.cu ----
// launch_keys_* write the keys of a batch's occurrence slots to keysA (they depend on the batch
// only, so they and the sort can run beside the gradient kernel); launch_step_* write the slots'
// update rows to `upd` (launch_step_sgns: two source rows per center and one factor per slot, to be
// reduced with run_push_reduce's d_scales) and return the number of per-block loss partials they wrote.  With keys_out
// (calls without a sort, small.cu) they write the slots' keys there themselves and latch errors for no call number.
void launch_keys_sgns(ps_store* ps, const uint32_t* d_tokens, uint64_t tok_first, uint64_t first_pos,
                      uint64_t n_centers, uint64_t corpus_len, uint32_t window, const uint32_t* d_negs, uint32_t n_neg,
                      uint64_t out_key_base, uint8_t* single, cudaStream_t s);
uint32_t launch_step_mf(ps_store* ps, const uint32_t* d_i, const uint32_t* d_j, const float* d_v, uint64_t n,
                        uint64_t col_key_base, float lr, float lambda, uint32_t* keys_out, cudaStream_t s);
float* sgns_scales(ps_store* ps, uint64_t n_centers);     // where launch_step_sgns puts the per-slot factors
uint32_t launch_step_sgns(ps_store* ps, const uint32_t* d_tokens, uint64_t tok_first, uint64_t first_pos,
                          uint64_t n_centers, uint64_t corpus_len, uint32_t window, const uint32_t* d_negs,
                          uint32_t n_neg, uint64_t out_key_base, float lr, uint32_t* keys_out, cudaStream_t s,
                          const uint8_t* single = nullptr);     // per slot: such rows are updated in place

// ---- device helpers ----
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// epoch 0: a call without later kernels to cancel (pull, set rows, get location); only the sticky code is latched
__device__ __forceinline__ void latch_error(DevStatus* st, unsigned int epoch, unsigned int code) {
    atomicCAS(&st->sticky, 0u, code);
    if (epoch != 0u) atomicExch(&st->call_err_epoch[epoch & 3u], epoch);
}
__device__ __forceinline__ bool call_failed(const DevStatus* st, unsigned int epoch) {
    return *((const volatile unsigned int*)&st->call_err_epoch[epoch & 3u]) == epoch;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ uint64_t phys_row(uint2 e, uint64_t S) { return (uint64_t)e.x * S + e.y; }
// AdaGrad's step -lr g / (sqrt(x) + eps), x = accumulator + g^2, with the hardware reciprocal square root and
// reciprocal (each within 2 ulp, far inside the fp32 tolerance of the result); x = 0 is kept away from 0 * inf
__device__ __forceinline__ float adagrad_step(float g, float x, float lr, float eps) {
    const float root = x > 0.f ? x * rsqrtf(x) : 0.f;
    return __fdividef(-lr * g, root + eps);
}
// The same for N values at a time.  Once sqrt(x) is thousands of times eps, which is all but the very first steps of a
// parameter, 1 / (sqrt(x) + eps) = r (1 - eps r) with r = 1 / sqrt(x), to within (eps r)^2 < 4e-8: one operation of the
// special-function unit instead of two, and that unit (16 lanes per clock and SM, conversions to and from fp64 included)
// is what bounds the reductions with AdaGrad.  Which form a value takes depends on that value alone (so results do not
// depend on how values are grouped), but one test serves all N, so that their chains interleave.  True if that form was taken
// by all and all steps are finite: x < 3e38 bounds g by 2e19, and lr is bounded too.
template <int N>
__device__ __forceinline__ bool adagrad_steps(const float (&g)[N], const float (&x)[N], float lr, float eps, float (&step)[N]) {
    float er[N];
    bool fine = fabsf(lr) < 1e18f;                                      // (false for a NaN, here and below)
#pragma unroll
    for (int i = 0; i < N; ++i) {
        float r;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x[i]));      // (zero or denormal: infinite, the other form)
        er[i] = __fmul_rn(eps, r);
        step[i] = __fmul_rn(__fmul_rn(-lr, g[i]), fmaf(-er[i], r, r));
        fine = fine && fabsf(er[i]) < 2e-4f && x[i] < 3e38f;
    }
    if (fine) return true;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (!(fabsf(er[i]) < 2e-4f && x[i] < 3e38f)) step[i] = adagrad_step(g[i], x[i], lr, eps);
    return false;
}
__device__ __forceinline__ void adagrad_steps4(const float4& g, const float4& x, float lr, float eps, float4& step) {
    const float gv[4] = {g.x, g.y, g.z, g.w}, xv[4] = {x.x, x.y, x.z, x.w};
    float sv[4];
    adagrad_steps<4>(gv, xv, lr, eps, sv);
    step = make_float4(sv[0], sv[1], sv[2], sv[3]);
}
// A finite fp32 value times 2^-896 as fp64, exactly, by integer operations: fp32's exponent and mantissa put into fp64's
// fields without a change of bias (denormals included).  Sums of such terms are the sums of the terms times 2^-896, with
// the same roundings; kUnscale takes the factor out again.  For sums whose conversions would queue for the
// special-function unit; the integer pipe has room there.
constexpr double kUnscale = 0x1p896, kScale = 0x1p-896;
__device__ __forceinline__ double widen_scaled(float v) {
    const int b = __float_as_int(v);
    return __hiloint2double((b >> 3) & 0x8fffffff, b << 29);
}

constexpr unsigned kBarrierSpins = 1u << 21;     // x ~100 ns: gives up after about a fifth of a second

// Barrier over all blocks of a cooperative launch.  bar[0] counts arrivals and only grows while the kernel
// runs: the k-th barrier is passed once it reaches k times the number of blocks.  bar[1] counts the blocks that
// have left the kernel; the last one to leave puts both words back to zero, so a launch always starts from
// zero without a clearing step in between.
__device__ __forceinline__ bool grid_barrier(unsigned int* bar, unsigned int target, int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(bar) : "memory");
        unsigned int seen = 0, spins = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(bar) : "memory");
            if (seen >= target || spins >= kBarrierSpins) break;
            __nanosleep(spins < 256 ? 20 : 100);
            ++spins;
        }
        *s_ok = seen >= target;
    }
    __syncthreads();
    return *s_ok != 0;
}
// The same barrier in two halves, for a block that has work to do between arriving and needing the others' results:
// everything the block wrote before grid_arrive is visible to a block that has passed grid_wait.
__device__ __forceinline__ void grid_arrive(unsigned int* bar) {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(bar) : "memory");
}
__device__ __forceinline__ bool grid_wait(unsigned int* bar, unsigned int target, int* s_ok) {
    if (threadIdx.x == 0) {
        unsigned int seen = 0, spins = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(bar) : "memory");
            if (seen >= target || spins >= kBarrierSpins) break;
            __nanosleep(spins < 256 ? 20 : 100);
            ++spins;
        }
        *s_ok = seen >= target;
    }
    __syncthreads();
    return *s_ok != 0;
}
__device__ __forceinline__ void grid_leave(unsigned int* bar, unsigned int n_blocks) {
    if (threadIdx.x == 0 && atomicAdd(bar + 1, 1u) == n_blocks - 1) {
        // every other block has left, so nobody is waiting on the arrival count any more
        atomicExch(bar, 0u);
        atomicExch(bar + 1, 0u);
    }
}

// Asks for a row to be in L2 (lane by lane, so that a warp's rows are on their way from memory together).
__device__ __forceinline__ void prefetch_row(const void* row, uint32_t bytes) {
    const char* p = (const char*)row;
    for (uint32_t o = 0; o < bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + bytes - 16));         // (rows need not start on a line)
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// ---- thread-block clusters: the hardware barrier (all threads of all blocks), addresses in another block's shared memory ----
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ uint32_t peer_smem(const void* p, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ int peer_i32(const int* p, uint32_t rank) {
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];\n" : "=r"(v) : "r"(peer_smem(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ double peer_f64(const double* p, uint32_t rank) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(v) : "r"(peer_smem(p, rank)) : "memory");
    return v;
}

// ---- bulk asynchronous copies global -> shared, reporting to a barrier word in shared memory ----
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
// one arrival that also announces `bytes` of copies
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// 16-byte aligned source and destination, size a multiple of 16 bytes
__device__ __forceinline__ void bulk_g2s(void* smem, const void* gmem, unsigned bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_addr(smem)),
                 "l"(gmem), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
// Waits for the phase of the given parity to complete; gives up (false) after a bounded number of polls.  Each poll
// may stay suspended in hardware for up to kBarSuspendNs (it returns as soon as the phase completes), so that a
// waiting warp does not spend issue slots on polling: about a quarter of a second per call at most.
constexpr unsigned kBarPollLimit = 1u << 17;
constexpr unsigned kBarSuspendNs = 2000;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
    const unsigned a = smem_addr(bar);
    for (unsigned i = 0; i < kBarPollLimit; ++i) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity), "r"(kBarSuspendNs)
            : "memory");
        if (done) return true;
    }
    return false;
}

// shared -> global, tracked in the issuing thread's bulk groups
__device__ __forceinline__ void bulk_s2g(void* gmem, const void* smem, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(gmem), "r"(smem_addr(smem)), "r"(bytes)
                 : "memory");
}
// Four rows of a 2-D tensor (one row per box) into consecutive rows of shared memory with ONE instruction of the TMA
// unit: column x (x times the element size a multiple of 16 bytes), rows y0..y3.  The destination is 128-byte aligned.
__device__ __forceinline__ void tma_gather4(void* smem, const CUtensorMap* map, int x, int y0, int y1, int y2, int y3,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];\n" ::"r"(smem_addr(smem)),
        "l"(map), "r"(x), "r"(y0), "r"(y1), "r"(y2), "r"(y3), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// until at most kPending of this thread's bulk groups still have to READ their source
template <int kPending>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(kPending) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// Exclusive scan of one value per thread over a block of 256 threads.
// `smem` must hold 8 uint32.  Returns the exclusive prefix; *total = block sum.
__device__ __forceinline__ uint32_t block_exclusive_scan_256(uint32_t v, uint32_t* smem, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) smem[w] = incl;
    __syncthreads();
    uint32_t wbase = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        uint32_t t = smem[i];
        if (i < w) wbase += t;
        tot += t;
    }
    __syncthreads();
    *total = tot;
    return wbase + incl - v;
}
#endif

}  // namespace psb
