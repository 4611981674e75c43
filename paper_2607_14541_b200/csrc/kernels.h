// Kernel parameter blocks and host-side launchers (internal to the library).
#pragma once
#include "atrex_dev.cuh"
#include "host_wait.h"

namespace atrex {

// Build-time variant of the scatter pass (the default is the fastest measured; the other is kept so
// that the comparison can be repeated):
//   ATREX_SCATTER_RING   stages of a shared-memory ring that a producer warp fills with bulk
//                        asynchronous copies of record tiles (0: records are loaded straight into
//                        registers, two 32-byte loads alternating per thread)
#ifndef ATREX_SCATTER_RING
#define ATREX_SCATTER_RING 0
#endif

// Shared memory of the scatter pass (dynamic, one CTA per SM) and what fits in it.  Per partition a
// cursor word, 16 KB of card-hour weights, the record ring if there
// is one, then the hot directory, in one of two forms (scatter.cu says which and why):
//   words  a 32-bit word that identifies the key inside its bucket and 12 bytes of accumulators per slot, 2-way buckets
//   tags   a tag byte, an 8-byte key and 12 bytes of accumulators per slot, 4-way buckets
constexpr uint32_t APPW_SMEM_MAX = 4096;
constexpr uint32_t SCATTER_SMEM_BYTES = 232448 - 1024;
constexpr uint32_t SCATTER_RING_STAGES = ATREX_SCATTER_RING;
constexpr uint32_t SCATTER_CONSUMER_WARPS = SCATTER_RING_STAGES ? 31 : 32;
constexpr uint32_t SCATTER_RING_TILE = SCATTER_CONSUMER_WARPS * 32 * 16;   // one record per consumer thread
constexpr uint32_t scatter_fixed_bytes(uint32_t lp) {
    return (4u << lp) + 4u * APPW_SMEM_MAX + SCATTER_RING_STAGES * SCATTER_RING_TILE + 128u;
}
constexpr uint32_t WORD_WAYS = 2, TAG_WAYS = 4;
constexpr uint32_t scatter_slots(uint32_t lp, bool words) { return ((SCATTER_SMEM_BYTES - scatter_fixed_bytes(lp)) / (words ? 16u : 21u)) & ~31u; }
constexpr uint32_t scatter_hot_slots(uint32_t lp) { return scatter_slots(lp, true); }   // of the directory image, either form

// Where one key dominates the trace, the last part of the accumulators holds the warps' queues instead (64 records
// each), and the directory is that much smaller.
constexpr uint32_t SCATTER_QUEUE = 64, SCATTER_QUEUE_BYTES = 32 * SCATTER_QUEUE * 16;
constexpr uint32_t scatter_dominated_slots(uint32_t lp, bool words) { return ((scatter_slots(lp, words) * 12u - SCATTER_QUEUE_BYTES - 16u) / 12u) & ~31u; }

struct IngestParams {
    const void* recs;          // all records of this launch (16-byte aligned) ...
    ull n_recs;
    const void* body;          // ... and the same split up: first record of the 32-byte aligned run of record pairs
    ull n_pairs;               // pairs in the body
    const void* single[2];     // records outside the body (unaligned head, odd tail)
    uint32_t n_single;
    uint32_t n_apps, n_phases;
    uint32_t phase_lim;        // n_phases << 16: bound of (phase << 16 | op_id)
    uint32_t appw_in_smem;
    const uint32_t* app_w;     // device copy of the card-hour weights
    ShortFormat fmt;           // short spill entries and directory words
    const ull* hot_keys;       // directory image, hot_slots entries of ~key (0 = empty)
    uint32_t hot_slots;        // multiple of 4
    const uint4* hot_words;    // the slots' words (words form)
    uint32_t img_rows;         // rows of hot_img that hold sums since the last fold; a CTA beyond them starts its row afresh
    ulonglong2* hot_img;       // [n_groups][hot_slots] each CTA's directory sums since the last fold, {lo, count | hi << 40}
    TableRef t;
    // spill buffers: entry i of scatter CTA g for partition p at spill + ((g * P + p) * cap + i) * 12 bytes: an 8-byte
    // word {product, operator} and a 4-byte word {phase, low hash bits}, the 8-byte word at the 8-byte aligned end;
    // short entries (ShortFormat) at spill + ((g * P + p) * short_cap + i) * 8 bytes
    unsigned char* spill;
    uint32_t* spill_cnt;       // [n_groups][P]
    uint32_t n_groups;         // G, row pitch of the buffers (= CTAs of the widest scatter launch)
    uint32_t cap;              // entries per (partition, CTA) buffer, a multiple of 32 (whole 128-byte lines)
    uint32_t drain_above;      // ask for a drain when a buffer holds more entries than this
    uint32_t short_cap, short_drain_above;   // the same in short entries ...
    uint32_t long_drain_above;               // ... of which many records take two
    ull seq;                   // sequence number of this launch
};

// Small calls (direct.cu): records straight into the table.
constexpr uint32_t DIRECT_RECORDS_MAX = 8192;   // up to here a thread per record, beyond it a shared-memory table per CTA
struct DirectParams {
    const uint4* recs;
    uint32_t n;
    uint32_t n_apps;
    uint32_t phase_lim;        // n_phases << 16
    const uint32_t* app_w;
    TableRef t;
    uint32_t share;            // records per CTA
    uint32_t slots;            // slots of a CTA's table
};

struct PartitionParams {
    TableRef t;
    const unsigned char* spill;
    uint32_t* spill_cnt;
    uint32_t n_groups;         // scatter CTAs whose buffers are read
    uint32_t cap, short_cap;
    ShortFormat fmt;           // as in IngestParams
    uint32_t misfit_max;       // more records than this that do not fit: drain, and long entries from here on
    uint32_t n_apps;
    const uint32_t* app_w;     // card-hour weights (short entries)
    uint32_t force;            // 1: drain unconditionally; 0: only if the scatter launch `seq` asked for it
    ull seq;
    ulonglong2* queue;         // [gridDim][queue_cap] entries whose first look failed, settled after the partition's stream
    uint32_t queue_cap;
    ull* told_long;            // pinned: `trace`, once its entries had to become long
    ull trace;
};

// Scratch of the directory build's last steps (cleared by every build up to `key`).
constexpr uint32_t HOT_SELECT_MAX = 27648;   // candidates kept (see hot_level_kernel)
constexpr uint32_t HOT_BUCKETS_MAX = 6912;   // directory buckets
static_assert(scatter_slots(8, true) / WORD_WAYS <= HOT_BUCKETS_MAX && scatter_slots(8, false) / TAG_WAYS <= HOT_BUCKETS_MAX &&
              scatter_slots(8, true) * 2 <= HOT_SELECT_MAX, "directory build scratch");
struct HotBuildScratch {
    uint32_t n, most, threshold, done;
    uint32_t weight, max_op, n_long, pad;        // sampled weight in the directory, largest operator, durations of two short entries
    uint32_t lost[4];                            // sampled weight each multiplier would lose
    uint32_t hist[1024];                         // candidates by count
    uint32_t occupancy[4][HOT_BUCKETS_MAX];
    uint32_t listed[HOT_BUCKETS_MAX];
    ull key[HOT_SELECT_MAX];                     // ~key
    uint32_t count[HOT_SELECT_MAX];
    uint32_t list[HOT_BUCKETS_MAX][16];          // candidates of each bucket
};

struct HotBuildParams {
    const uint4* recs;
    ull stride;                // records per sampled one (below 2^32)
    uint32_t n_sample;         // n_sample * stride <= records of the call
    uint32_t n_apps, n_phases;
    uint32_t max_ops, dur_mask;   // as in ShortFormat (max_ops 0: no short entries)
    ull* hot_keys;
    uint32_t hot_slots;        // of the image
    uint32_t* hot_words;       // [hot_slots] (words form)
    uint32_t phase_bits;       // as in ShortFormat
    uint32_t slots[2][2];      // slots in use by [words][one key dominates]
    ull* sample;               // [n_sample] the sampled keys, all ones = invalid record
    uint32_t* sketch;          // [2^20] sample counters by hash
    ull* cand_keys;            // [1 << cand_bits] candidate table: ~key, 0 = empty
    uint32_t* cand_cnt;        // [1 << cand_bits] exact sample counts of the candidates
    uint32_t cand_bits;
    HotBuildScratch* scratch;
    Control* ctl;
};

struct WorkRef {
    ull* keys;           // [P * Cw], nullptr when no work table was provisioned
    double2* rows;       // [P * Cw] {flops, bytes}, rounded once
    uint32_t lp;         // log2(P), same partitioning as the key table
    uint32_t Cw;         // slots per partition, whole buckets
    ull strides;         // eight probe strides in buckets, one byte each: odd primes that do not divide their number (double hashing)
};

struct FinalizeParams {
    TableRef t;
    ull n_slots;
    Control* ctl;
    ulonglong2* told;    // pinned: the control block's first CONTROL_WORDS words for the host, each with the stamp
    uint32_t stamp;
    WorkRef work;
    atrex_hw_peaks_t peaks;
    atrex_entry_t* out;
    ull out_cap;
};

struct GivenTotals {     // totals to normalise by instead of the table's own
    ull lo[ATREX_MAX_PHASES], hi[ATREX_MAX_PHASES];
    uint32_t use;
};

// Top-k of every phase at once (the usual way): see topk_first_digit in finalize.cu.
struct PickParams {
    FinalizeParams fin;
    uint32_t n_phases, k;
    uint32_t* hist;            // [n_phases][TOPK_BINS] first-digit counts
    ull* sel;                  // [n_phases][TOPK_PICK_MAX][4]
    atrex_entry_t* host_top;   // pinned: [n_phases][TOPK_PICK_K] (k > TOPK_TOLD_K)
    ulonglong2* host_told;     // pinned: [n_phases][TOPK_TOLD_K][6] rows with stamps (smaller k)
    ull* host_n;               // pinned: [n_phases] fin.stamp << 32 | entries written (PICK_NONE: not answered this way)
};

// Top-k, the long way: phases in one pass over the table, each with its own place in the ranking (see finalize.cu).
constexpr uint32_t TOPK_DIGITS = 12;                   // 12-bit digits behind the first one, at most
struct TopkAllParams {
    TableRef t;
    ull n_slots;
    uint32_t active_mask;                              // phases taking part in this pass
    uint32_t collect_all_mask;                         // ... of which every entry is collected
    uint32_t row[ATREX_MAX_PHASES];                    // counting: each active phase's row in shared memory
    uint32_t first[ATREX_MAX_PHASES];                  // first digit of the k-th key
    uint32_t n_digits[ATREX_MAX_PHASES];               // further digits already known
    uint16_t digit[ATREX_MAX_PHASES][TOPK_DIGITS];
    uint32_t* hist;                                    // [n_phases][TOPK_BINS] counts of the next digit
    ull* sel;                                          // [n_phases][sel_cap][4]: composite words 2, 1, 0 and the slot index
    ull* sel_count;                                    // [ATREX_MAX_PHASES]
    uint32_t sel_cap;
};
struct TopkDigit {                                     // in pinned memory: where a phase's k-th key lies
    ull seq, bin, above, in_bin;                       // ... its digit, keys in higher bins, keys in its own
};
struct TopkDigitParams {
    const uint32_t* hist;                              // [n_phases][TOPK_BINS]
    uint32_t active_mask;
    uint32_t need[ATREX_MAX_PHASES];                   // the wanted key's place among the counted ones
    TopkDigit* answers;                                // [n_phases], `seq` last
    ull seq;
};
struct TopkSortParams {
    ull* sel;                                          // [n_phases][sel_cap][4]
    uint32_t sel_cap;
    uint32_t n_pow2[ATREX_MAX_PHASES];                 // items of each phase with padding, 0 = nothing to do
};

// Launches a kernel whose set-up may overlap its predecessor on the stream (the kernel starts with
// grid_dependency_wait): between kernels of a few microseconds the gap is a third of their time.  Only grids of
// up to two CTAs per SM: the CTAs of a wide grid that fill up the SMs while the predecessor drains end up
// unevenly spread (emit kernel over a 566 MB table: 1 120 us chained, 614 us not).
constexpr uint32_t CHAIN_MAX_CTAS = 296;
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), uint32_t grid, uint32_t block, size_t smem, cudaStream_t stream, const A&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = attr;
    c.numAttrs = grid <= CHAIN_MAX_CTAS ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// Pinned host memory, visible to the device, that kernels write results to (pinned.cu).  Blocks of up to 512 KB come from
// a pool of the process, so that creating a handle does not pay for pinning; at most eight wait there.
cudaError_t pinned_alloc(void** out, size_t bytes);
void pinned_free(void* block, size_t bytes);

// CTAs of a grid-stride kernel: as many as the SMs hold at once (a second, partly filled wave would cost as
// much as a full one), fewer when there is less work.  `per_sm` comes from resident_ctas, asked once.
template <typename K>
inline uint32_t resident_ctas(K* kernel, int threads, size_t smem) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) n = 1;
    return (uint32_t)n;
}
inline uint32_t grid_for_work(ull items, ull items_per_cta, int n_sms, uint32_t per_sm) {
    const ull want = (items + items_per_cta - 1) / items_per_cta, most = (ull)n_sms * per_sm;
    return (uint32_t)(want < 1 ? 1 : (want < most ? want : most));
}

cudaError_t ingest_prepare();
cudaError_t direct_prepare();
cudaError_t launch_direct(DirectParams p, int n_sms, cudaStream_t stream);
cudaError_t scatter_prepare();
cudaError_t launch_scatter(const IngestParams& p, bool hot, int grid, cudaStream_t stream);
cudaError_t launch_partition(const PartitionParams& p, int n_sms, cudaStream_t stream);
inline size_t partition_smem_bytes(uint32_t C, uint32_t n_apps, bool short_entries) { return (size_t)C * 20 + (short_entries ? (size_t)n_apps * 4 : 0); }
cudaError_t launch_hot_build(const HotBuildParams& p, int n_sms, cudaStream_t stream);
cudaError_t launch_hot_fold(const ull* hot_keys, const ulonglong2* hot_img, uint32_t n_groups, uint32_t hot_slots,
                            const TableRef& t, cudaStream_t stream);
cudaError_t launch_merge(const atrex_entry_t* in, ull n, const TableRef& t, cudaStream_t stream);

cudaError_t finalize_prepare();
cudaError_t launch_totals(const TableRef& t, ull n_slots, uint32_t n_phases, const GivenTotals& given, uint32_t* hist, uint32_t* next_hist, int n_sms,
                          cudaStream_t stream);
cudaError_t launch_emit(const FinalizeParams& p, int n_sms, cudaStream_t stream);
bool finalize_in_one_cluster(ull n_slots);       // totals and entries in one launch, the best k in another (asked after finalize_prepare)
cudaError_t launch_finalize_small(const FinalizeParams& p, uint32_t n_phases, const GivenTotals& given, uint32_t* hist, uint32_t* next_hist,
                                  cudaStream_t stream);
cudaError_t launch_work_insert(const atrex_work_t* rows, ull n, const WorkRef& w, Control* ctl, int grid,
                               cudaStream_t stream);
cudaError_t launch_topk_pick(const PickParams& p, bool one_cluster, int n_sms, cudaStream_t stream);
cudaError_t launch_topk_collect_all(const TopkAllParams& p, int grid, cudaStream_t stream);
cudaError_t launch_topk_hist(const TopkAllParams& p, int n_sms, cudaStream_t stream);
cudaError_t launch_topk_digit(const TopkDigitParams& p, uint32_t n_phases, cudaStream_t stream);
cudaError_t launch_topk_sort(const TopkSortParams& p, uint32_t n_phases, cudaStream_t stream);
cudaError_t launch_topk_emit(const FinalizeParams& p, const ull* sel, uint32_t n, cudaStream_t stream);

}  // namespace atrex
