// C ABI of the trace-aggregation library: argument checks, workspace carving, launches.
// The declarations and their contracts are in include/atrex_agg.h.
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <new>

#include <nvtx3/nvToolsExt.h>

#include "kernels.h"

using namespace atrex;

namespace {

constexpr size_t ALIGN = 256;
constexpr size_t STAGING_BYTES = 64ull << 20;          // per staging buffer (two of them)
constexpr uint32_t LP_MIN = 8, LP_MAX = 12;             // 256 .. 4096 partitions
constexpr ull MAX_KEYS = 1ull << 25;
constexpr ull MAX_RECORDS_TOTAL = 1ull << 40;
constexpr size_t L2_TABLE_BYTES = 48ull << 20;           // a table up to this size stays in the 126 MB L2
constexpr uint32_t HOT_SAMPLE = 1u << 20;
constexpr uint32_t CAND_BITS = 17;                     // candidate table of the directory build
constexpr size_t SKETCH_BYTES = (size_t)4 << 20;        // 2^20 counters (ingest.cu SKETCH_BITS)
// sketch, candidate table and the first part of HotBuildScratch are cleared by every build; the sampled keys lie behind
constexpr size_t HOT_SELECT_OFF = SKETCH_BYTES + ((size_t)12 << CAND_BITS);
constexpr size_t HOT_COUNT_BYTES = HOT_SELECT_OFF + offsetof(HotBuildScratch, key);
constexpr size_t HOT_SAMPLE_OFF = HOT_SELECT_OFF + (sizeof(HotBuildScratch) + 255) / 256 * 256;
constexpr size_t HOT_SCRATCH_BYTES = HOT_SAMPLE_OFF + (size_t)HOT_SAMPLE * 8;
constexpr uint32_t SEL_CAP = ATREX_MAX_TOPK;           // items of a phase that the long way to the top-k sorts
static_assert((SEL_CAP & (SEL_CAP - 1)) == 0 && SEL_CAP >= TOPK_PICK_MAX, "a power of two");

size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// A named range around each entry point's host work, for timelines taken with a tracing tool (the
// header-only NVTX: a no-op costing one pointer check when no tool is attached).
struct TraceRange {
    explicit TraceRange(const char* name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange&) = delete;
    TraceRange& operator=(const TraceRange&) = delete;
};

ull pow2_at_least(ull x) {
    ull p = 1;
    while (p < x) p <<= 1;
    return p;
}

struct Layout {
    size_t off_ctl, off_keys, off_vals, off_work, off_appw, off_hot, off_hot_words, off_staging[2], off_sel, off_pick, off_topk_out, off_hist_all, off_hist_next,
        off_spill_cnt, off_spill, off_hot_scratch, off_queue, off_hot_img, total;
    ull n_slots, work_slots;
    uint32_t lp, C;              // partitions = 1 << lp, slots per partition
    uint32_t Cw;                 // work-table slots per partition
    uint32_t n_groups, cap;      // spill buffers: [P][n_groups][cap] entries
    ull sub_launch;              // records per scatter + partition launch pair
    uint32_t hot_slots;
    ShortFormat fmt;           // short spill entries and directory words
    uint32_t queue_cap;        // deferred entries per CTA in the partition pass
    bool appw_in_smem;
};

bool config_ok(const atrex_agg_config_t* c) {
    if (!c) return false;
    if (c->n_apps == 0 || c->n_phases == 0 || c->n_phases > ATREX_MAX_PHASES) return false;
    if (c->max_keys == 0 || c->max_keys > MAX_KEYS) return false;
    if (c->max_work_rows > (1ull << 30)) return false;
    return true;
}

void compute_layout(const atrex_agg_config_t* c, size_t smem_optin, int n_sms, Layout* L) {
    // Partition geometry: one partition's keys + per-launch accumulators (20 B per slot) and, where entries may be
    // short, the applications' weights must fit one SM's shared memory (10 688 slots beside 4 096 weights and not 11 488:
    // 2^30 records over 16 M keys, whole build +0.5 %).  A key can only live in its hash partition, so a partition is sized for the
    // tail of its load, not for the mean: with m = max_keys / P keys expected, the keys of one
    // (operator, shape) -- up to n_phases of them -- always fall together, which bounds the standard
    // deviation by sqrt(n_phases * m); six of those plus a constant, and never less than 1.3 m (2 m for small tables).
    L->appw_in_smem = c->n_apps <= APPW_SMEM_MAX;
    const bool with_weights = L->appw_in_smem && SCATTER_RING_STAGES == 0;   // (the partition pass multiplies short entries)
    const uint32_t c_max = (uint32_t)((smem_optin - 2048 - (with_weights ? 4 * c->n_apps : 0)) / 20) & ~31u;
    auto slots_for = [&](uint32_t lp) -> ull {
        const ull m = (c->max_keys + (1ull << lp) - 1) >> lp;
        // two slots per key where the smallest number of partitions allows it (probes mostly end at the first
        // pair then: drain of 17 M entries into 0.5 M keys 157 -> 134 us), 1.3 where the table is large
        const ull flat = lp == LP_MIN && 2 * m < c_max ? 2 * m + 1 : m + m * 3 / 10 + 1;
        const ull tail = m + (ull)std::ceil(6.0 * std::sqrt((double)c->n_phases * (double)m)) + 32;
        return flat > tail ? flat : tail;
    };
    L->lp = LP_MIN;
    while (L->lp < LP_MAX && slots_for(L->lp) > c_max) ++L->lp;
    ull per = slots_for(L->lp);
    if (per > c_max || L->lp > LP_MIN) per = c_max;  // big tables: use all of shared memory, lower load factor
    if (per < 128) per = 128;
    L->C = (uint32_t)((per + 31) / 32 * 32);
    L->n_slots = (ull)L->C << L->lp;
    L->n_groups = (uint32_t)n_sms;
    L->sub_launch = c->max_keys >= (1ull << 21) ? (1ull << 27) : (c->max_keys >= (1ull << 16) ? (1ull << 25) : (1ull << 24));
    // room for 4.5 launches' worth of long entries if every record spilled, 6.75 of short ones; a drain is requested when a
    // buffer passes 3/4 of that, which leaves 1.1 and 1.7 full launches of headroom.  A short entry's record takes two where its
    // duration is long: a launch that is mostly such asks from 5/8 on, which leaves room for two entries a record.  (Only
    // where short durations turn into long ones from one launch to the next may a buffer still run over: exact, but
    // record by record.)  At the bench workload (half of the records spill) four or five launches
    // accumulate between drains.
    ull per_buf = (L->sub_launch * 9 / 2) / (((ull)n_sms) << L->lp);
    if (per_buf < 64) per_buf = 64;
    if (per_buf > 32768) per_buf = 32768;   // the scatter pass counts a buffer's entries in 16 bits, with headroom
    L->cap = (uint32_t)((per_buf + 31) / 32 * 32);   // a buffer is a whole number of 128-byte lines
    // entries of one partition whose first look fails wait in a per-CTA queue, one segment per warp:
    // room for a quarter of the partition's worst-case stream, at most 32 K entries (a warp whose
    // segment could not take another batch of 128 settles it first), at least two batches per warp
    {
        ull q = (ull)L->cap * n_sms / 4;
        L->queue_cap = (uint32_t)(q < 8192 ? 8192 : (q > 32768 ? 32768 : q));
    }
    // work table: same partitions as the key table, 1.5 slots per row plus slack for uneven partitions
    L->Cw = c->max_work_rows ? (uint32_t)((((c->max_work_rows * 3 / 2) >> L->lp) + 64 + 31) / 32 * 32) : 0;
    L->work_slots = (ull)L->Cw << L->lp;
    L->hot_slots = scatter_hot_slots(L->lp);   // what the scatter pass's shared memory holds for this partition count
    if (c->flags & ATREX_FLAG_NO_HOT_DIRECTORY) L->hot_slots = 0;
    // Short spill entries: phases and applications take what they need, the operators all that a directory word has left
    // as long as durations keep 20 bits (2 % of log-normal durations around 50 us are longer and take two entries), and
    // eight bits in any case; below 16 bits of duration an entry of 12 bytes would be no worse.
    const auto bits_for = [](uint32_t n) {
        uint32_t b = 0;
        while (b < 32 && (1u << b) < n) ++b;
        return b;
    };
    memset(&L->fmt, 0, sizeof(L->fmt));
    if (with_weights) {
        ShortFormat& f = L->fmt;
        f.phase_bits = bits_for(c->n_phases);
        f.app_bits = bits_for(c->n_apps);
        const uint32_t in_high = L->lp - 1 < DIR_ID_BITS - 1 ? L->lp - 1 : DIR_ID_BITS - 1;
        uint32_t op_bits = DIR_ID_BITS - 1 - f.phase_bits, rest_bits = 0;
        for (;; --op_bits) {
            rest_bits = f.phase_bits + op_bits > in_high ? f.phase_bits + op_bits - in_high : 0;
            f.dur_bits = 32 - rest_bits - f.app_bits;
            if (f.dur_bits >= 20 || op_bits == 8) break;
        }
        f.rest_shift = rest_bits ? 32 - rest_bits : 31;
        f.rest_mask = rest_bits ? ~0u << f.rest_shift : 0u;
        if (f.dur_bits > 31) f.dur_bits = 31;
        f.max_ops = 1u << op_bits;
    }
    size_t o = 0;
    // (control block, spill counts and table are neighbours: a reset clears them in one piece)
    L->off_ctl = o;            o += round_up(sizeof(Control), ALIGN);
    L->off_spill_cnt = o;      o += round_up(((size_t)L->n_groups << L->lp) * 4, ALIGN);
    L->off_keys = o;           o += round_up(L->n_slots * 8, ALIGN);
    L->off_vals = o;           o += round_up(L->n_slots * 16, ALIGN);
    L->off_work = o;           o += round_up(L->work_slots * WORK_SLOT_BYTES, ALIGN);
    L->off_appw = o;           o += round_up((size_t)c->n_apps * 4, ALIGN);
    L->off_hot = o;            o += round_up((size_t)(L->hot_slots ? L->hot_slots : 2) * 8, ALIGN);
    L->off_hot_words = o;      o += round_up((size_t)(L->hot_slots ? L->hot_slots : 2) * 4, ALIGN);
    L->off_hot_img = o;        o += round_up((size_t)L->n_groups * (L->hot_slots ? L->hot_slots : 2) * 16, ALIGN);
    L->off_staging[0] = o;     o += STAGING_BYTES;
    L->off_staging[1] = o;     o += STAGING_BYTES;
    L->off_sel = o;            o += round_up((size_t)SEL_CAP * 32 * c->n_phases, ALIGN);   // one region per phase
    L->off_pick = o;           o += round_up((size_t)TOPK_PICK_MAX * 32 * c->n_phases, ALIGN);
    L->off_hist_all = o;       o += round_up((size_t)2 * c->n_phases * TOPK_BINS * 4, ALIGN);
    L->off_hist_next = o;      o += round_up((size_t)c->n_phases * TOPK_BINS * 4, ALIGN);
    L->off_topk_out = o;       o += round_up((size_t)ATREX_MAX_TOPK * sizeof(atrex_entry_t), ALIGN);
    L->off_hot_scratch = o;    o += round_up(HOT_SCRATCH_BYTES, ALIGN);
    L->off_queue = o;          o += round_up((size_t)L->n_groups * L->queue_cap * 16, ALIGN);
    L->off_spill = o;          o += round_up(((size_t)L->n_groups << L->lp) * L->cap * SPILL_ENTRY_BYTES, ALIGN) + ALIGN;  // + prefetch overrun
    L->total = o;
}

struct DeviceGuard {
    int prev = -1;
    bool switched = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) switched = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() {
        if (switched && prev >= 0) cudaSetDevice(prev);
    }
};

}  // namespace

// What ranking requests worked out, kept until the next finalize: for the last k asked for, every phase's answer
// (in pinned memory); for the last k that took the long way, the sorted selections of the phases that do.
struct TopkCache {
    ull pick_gen = 0;                       // finalize generation the answers belong to (0 = none)
    uint32_t k = 0;                         // k of the answers
    ull sel_gen = 0;                        // the long way
    uint32_t sel_k = 0, sel_mask = 0;       // its phases
    ull total[ATREX_MAX_PHASES] = {};       // candidates selected
};

struct atrex_agg {
    atrex_agg_config_t cfg;
    Layout L;
    int n_sms = 0;
    bool owns_workspace = false;
    unsigned char* ws = nullptr;
    Control* ctl = nullptr;
    ull* keys = nullptr;
    ulonglong2* vals = nullptr;
    uint32_t* spill_cnt = nullptr;
    unsigned char* spill = nullptr;
    ulonglong2* queue = nullptr;
    unsigned char* hot_scratch = nullptr;
    ull* work = nullptr;      // keys, the rows behind them
    uint32_t* d_appw = nullptr;
    ull* hot_keys = nullptr;
    ulonglong2* hot_img = nullptr;   // [n_groups][hot_slots] per-CTA directory sums not yet in the table
    uint32_t img_rows = 0;           // rows that hold sums
    unsigned char* staging[2] = {nullptr, nullptr};
    ull* sel = nullptr;
    atrex_entry_t* topk_out = nullptr;
    Control* h_ctl = nullptr;  // pinned: the host's copy of the control block
    ulonglong2* h_told = nullptr;     // pinned: [CONTROL_WORDS] as the last finalize's kernel tells them
    ulonglong2* h_top_told = nullptr;    // pinned: [n_phases][TOPK_TOLD_K][6] ... the best few of each phase
    size_t pinned_bytes = 0;
    uint32_t* hist_all = nullptr;     // [2][n_phases][TOPK_BINS] first-digit counts: the last totals pass's, and zeros for the next
    uint32_t hist_at = 0;             // which half is the last pass's
    uint32_t* hist_next = nullptr;    // [n_phases][TOPK_BINS] counts of a further digit
    ull wait_seq = 0;                 // number of the last kernel that the host waited for
    ull* pick = nullptr;              // [n_phases][TOPK_PICK_MAX][4] candidates
    atrex_entry_t* h_top = nullptr;   // pinned: [n_phases][TOPK_PICK_K] the best k of each phase, then [n_phases] how many
    TopkDigit* h_digit = nullptr;     // pinned: [n_phases]
    TopkCache topk;
    ull fin_gen = 0;                  // bumped by every successful finalize
    bool hot_ready = false;
    ull* h_long = nullptr;        // pinned: the trace whose entries had to become long, as the partition pass tells it
    ull trace = 1;                // number of this trace: one more with every reset
    bool long_only = false;       // ... its entries have, and the directory was built anew for them
    bool finalized = false;
    bool one_cluster = false;     // finalize and top-k of this (small) table: a launch of one cluster each
    bool spill_pending = false;   // entries may sit in the spill buffers
    ull scatter_seq = 0;          // sequence number of the last scatter launch
    atrex_hw_peaks_t peaks;
    ull n_records = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_ready[2] = {nullptr, nullptr}, ev_free[2] = {nullptr, nullptr};
    int last_cuda_error = 0;
    uint64_t launches = 0;

    // eight odd primes, one per byte, that do not divide m (m even or a power of two times such a number:
    // the strides are then coprime to it)
    static ull strides_for(uint32_t m) {
        ull strides = 0;
        uint32_t n = 0;
        for (uint32_t c = 7; n < 8; c += 2) {
            bool prime = true;
            for (uint32_t d = 3; d * d <= c; d += 2) prime = prime && (c % d != 0);
            if (prime && m % c != 0) strides |= (ull)c << (8 * n++);
        }
        return strides;
    }
    ull key_strides = 0, work_strides = 0;   // worked out once by create
    TableRef table_ref() const {
        TableRef t;
        t.keys = keys;
        t.vals = vals;
        t.lp = L.lp;
        t.C = L.C;
        t.ctl = ctl;
        t.strides = key_strides;
        return t;
    }
    WorkRef work_ref() const {
        WorkRef w;
        w.keys = L.work_slots ? work : nullptr;
        w.rows = (double2*)(work + L.work_slots);
        w.lp = L.lp;
        w.Cw = L.Cw;
        w.strides = work_strides;
        return w;
    }
    int scan_grid(ull n_items, int threads) const {
        ull g = (n_items + threads - 1) / threads;
        ull cap = (ull)n_sms * 8;
        if (g > cap) g = cap;
        return g < 1 ? 1 : (int)g;
    }
};

#define CU(h, call)                                   \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) {                      \
            (h)->last_cuda_error = (int)e_;           \
            return ATREX_ERR_CUDA;                    \
        }                                             \
    } while (0)

static int device_status_to_error(const Control* c) {
    if (c->status & ST_BOUNDS) return ATREX_ERR_BOUNDS;
    if (c->status & ST_TIMEOUT) return ATREX_ERR_TIMEOUT;
    if (c->status & ST_TABLE_FULL) return ATREX_ERR_CAPACITY;
    return ATREX_OK;
}

static int query_sm_count(int device) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || v <= 0) {
        cudaGetLastError();
        return 148;  // B200
    }
    return v;
}

static int query_smem_optin(int device, size_t* out) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) return -1;
    *out = (size_t)v;
    return 0;
}

extern "C" {

uint64_t atrex_agg_workspace_bytes(const atrex_agg_config_t* cfg) {
    if (!config_ok(cfg)) return 0;
    // the directory size depends on the device's shared memory; without a device, size for
    // the sm_100 maximum (the layout only grows with it)
    size_t smem = 232448;
    size_t q;
    if (query_smem_optin(cfg->device, &q) == 0 && q > 0) smem = q;
    Layout L;
    compute_layout(cfg, smem, query_sm_count(cfg->device), &L);
    return L.total;
}

int atrex_agg_create(const atrex_agg_config_t* cfg, atrex_agg_t** out) {
    if (!out) return ATREX_ERR_INVALID;
    *out = nullptr;
    if (!config_ok(cfg) || !cfg->app_weights) return ATREX_ERR_INVALID;
    if (cfg->workspace && ((uintptr_t)cfg->workspace % ALIGN) != 0) return ATREX_ERR_INVALID;
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess || cfg->device < 0 || cfg->device >= n_dev) {
        cudaGetLastError();
        return ATREX_ERR_CUDA;
    }
    atrex_agg* h = new (std::nothrow) atrex_agg;
    if (!h) return ATREX_ERR_NOMEM;
    h->cfg = *cfg;
    h->cfg.app_weights = nullptr;
    DeviceGuard guard(cfg->device);
    size_t smem = 0;
    int rc = ATREX_OK;
    do {
        if (query_smem_optin(cfg->device, &smem) != 0) { rc = ATREX_ERR_CUDA; break; }
        if (cudaDeviceGetAttribute(&h->n_sms, cudaDevAttrMultiProcessorCount, cfg->device) != cudaSuccess) { rc = ATREX_ERR_CUDA; break; }
        compute_layout(cfg, smem, h->n_sms, &h->L);
        if (cfg->workspace) {
            if (cfg->workspace_bytes < h->L.total) { rc = ATREX_ERR_NOMEM; break; }
            h->ws = (unsigned char*)cfg->workspace;
        } else {
            if (cudaMalloc((void**)&h->ws, h->L.total) != cudaSuccess) { cudaGetLastError(); rc = ATREX_ERR_NOMEM; break; }
            h->owns_workspace = true;
        }
        const Layout& L = h->L;
        h->key_strides = atrex_agg::strides_for(L.C / 2);   // in slot pairs
        h->work_strides = atrex_agg::strides_for(L.Cw ? L.Cw / WORK_WAYS : 1);
        h->ctl = (Control*)(h->ws + L.off_ctl);
        h->keys = (ull*)(h->ws + L.off_keys);
        h->vals = (ulonglong2*)(h->ws + L.off_vals);
        h->spill_cnt = (uint32_t*)(h->ws + L.off_spill_cnt);
        h->spill = h->ws + L.off_spill;
        h->queue = (ulonglong2*)(h->ws + L.off_queue);
        h->hot_scratch = h->ws + L.off_hot_scratch;
        h->work = (ull*)(h->ws + L.off_work);
        h->d_appw = (uint32_t*)(h->ws + L.off_appw);
        h->hot_keys = (ull*)(h->ws + L.off_hot);
        h->hot_img = (ulonglong2*)(h->ws + L.off_hot_img);
        h->staging[0] = h->ws + L.off_staging[0];
        h->staging[1] = h->ws + L.off_staging[1];
        h->sel = (ull*)(h->ws + L.off_sel);
        h->topk_out = (atrex_entry_t*)(h->ws + L.off_topk_out);
        h->hist_all = (uint32_t*)(h->ws + L.off_hist_all);
        h->pick = (ull*)(h->ws + L.off_pick);
        h->hist_next = (uint32_t*)(h->ws + L.off_hist_next);
        cudaError_t e = cudaSuccess;
        if (e == cudaSuccess) e = cudaMemset(h->ws + L.off_ctl, 0, L.off_appw - L.off_ctl);  // control, spill counts, table, work
        if (e == cudaSuccess) e = cudaMemcpy(h->d_appw, cfg->app_weights, (size_t)cfg->n_apps * 4, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(h->hist_all, 0, (size_t)2 * cfg->n_phases * TOPK_BINS * 4);
        if (e == cudaSuccess) e = cudaMemset(h->hot_keys, 0, (size_t)(L.hot_slots ? L.hot_slots : 2) * 8);
        // the pinned block: what kernels tell with stamps, every phase's best, how many there are, a digit each, the control block's copy
        const size_t top_bytes = (size_t)cfg->n_phases * (TOPK_PICK_K * sizeof(atrex_entry_t) + 8), digit_bytes = cfg->n_phases * sizeof(TopkDigit);
        const size_t told_bytes = CONTROL_WORDS * 16 + (size_t)cfg->n_phases * TOPK_TOLD_K * 96;
        h->pinned_bytes = told_bytes + top_bytes + digit_bytes + sizeof(Control) + 8;
        if (e == cudaSuccess) e = pinned_alloc((void**)&h->h_told, h->pinned_bytes);
        if (e == cudaSuccess) {
            memset(h->h_told, 0, told_bytes);        // (the block may be another handle's former one: no stamp of its may be left)
            h->h_top_told = h->h_told + CONTROL_WORDS;
            h->h_top = (atrex_entry_t*)((unsigned char*)h->h_told + told_bytes);
            h->h_digit = (TopkDigit*)((unsigned char*)h->h_top + top_bytes);
            h->h_ctl = (Control*)((unsigned char*)h->h_digit + digit_bytes);
            memset(h->h_digit, 0, digit_bytes);
            h->h_long = (ull*)(h->h_ctl + 1);
            *h->h_long = 0;
        }
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking);
        for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
            e = cudaEventCreateWithFlags(&h->ev_ready[i], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_free[i], cudaEventDisableTiming);
        }
        if (e == cudaSuccess) e = ingest_prepare();
        if (e == cudaSuccess) e = finalize_prepare();
        if (e == cudaSuccess) h->one_cluster = finalize_in_one_cluster(L.n_slots);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (e != cudaSuccess) { h->last_cuda_error = (int)e; rc = ATREX_ERR_CUDA; break; }
    } while (0);
    if (rc != ATREX_OK) {
        atrex_agg_destroy(h);
        return rc;
    }
    *out = h;
    return ATREX_OK;
}

void atrex_agg_destroy(atrex_agg_t* h) {
    if (!h) return;
    DeviceGuard guard(h->cfg.device);
    cudaDeviceSynchronize();
    for (int i = 0; i < 2; ++i) {
        if (h->ev_ready[i]) cudaEventDestroy(h->ev_ready[i]);
        if (h->ev_free[i]) cudaEventDestroy(h->ev_free[i]);
    }
    if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
    pinned_free(h->h_told, h->pinned_bytes);
    if (h->owns_workspace && h->ws) cudaFree(h->ws);
    delete h;
}

int atrex_agg_reset(atrex_agg_t* h, void* stream) {
    TraceRange range("atrex_agg_reset");
    if (!h) return ATREX_ERR_INVALID;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    // control block, spill counts (undrained entries are discarded), keys and values
    CU(h, cudaMemsetAsync(h->ctl, 0, h->L.off_work - h->L.off_ctl, s));
    h->img_rows = 0;
    h->spill_pending = false;
    h->hot_ready = false;
    h->long_only = false;
    ++h->trace;
    h->finalized = false;
    h->n_records = 0;
    return ATREX_OK;
}

int atrex_agg_set_work_table(atrex_agg_t* h, const atrex_work_t* rows, uint64_t n, void* stream) {
    TraceRange range("atrex_agg_set_work_table");
    if (!h || (n && !rows) || n > h->cfg.max_work_rows) return ATREX_ERR_INVALID;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    if (h->L.work_slots == 0) return ATREX_OK;
    CU(h, cudaMemsetAsync(h->work, 0, h->L.work_slots * sizeof(ull), s));
    CU(h, cudaMemsetAsync(&h->ctl->work_status, 0, sizeof(ull), s));
    const uint64_t per_piece = STAGING_BYTES / sizeof(atrex_work_t);
    for (uint64_t off = 0; off < n; off += per_piece) {
        uint64_t m = n - off < per_piece ? n - off : per_piece;
        CU(h, cudaMemcpyAsync(h->staging[0], rows + off, m * sizeof(atrex_work_t), cudaMemcpyHostToDevice, s));
        CU(h, launch_work_insert((const atrex_work_t*)h->staging[0], m, h->work_ref(), h->ctl, h->scan_grid(m, 256), s));
        h->launches++;
        CU(h, cudaStreamSynchronize(s));  // the staging buffer and the host rows are reused
    }
    CU(h, cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Control), cudaMemcpyDeviceToHost, s));
    CU(h, cudaStreamSynchronize(s));
    h->finalized = false;
    if (h->h_ctl->work_status != 0) {
        CU(h, cudaMemsetAsync(h->work, 0, h->L.work_slots * sizeof(ull), s));
        CU(h, cudaStreamSynchronize(s));
        return ATREX_ERR_INVALID;
    }
    return ATREX_OK;
}

// The directory sums kept per scatter CTA join the table.
static int fold_directory(atrex_agg* h, cudaStream_t s) {
    if (h->img_rows == 0) return ATREX_OK;
    CU(h, launch_hot_fold(h->hot_keys, h->hot_img, h->img_rows, h->L.hot_slots, h->table_ref(), s));
    h->launches++;
    h->img_rows = 0;
    return ATREX_OK;
}

// Partition pass over the spill buffers.  Unforced, the kernel exits at once unless the scatter
// launch just before it saw a buffer more than 3/4 full; forced (before results are read), it
// drains whatever is there.
static int drain_spill(atrex_agg* h, bool force, cudaStream_t s) {
    if (force && !h->spill_pending) return ATREX_OK;
    if (force) {
        // results are about to be read (the directory's sums before the spilled entries, while the frequent keys' slots are
        // still easy to come by)
        const int rc = fold_directory(h, s);
        if (rc != ATREX_OK) return rc;
    }
    PartitionParams q;
    q.t = h->table_ref();
    q.spill = h->spill;
    q.spill_cnt = h->spill_cnt;
    q.n_groups = h->L.n_groups;
    q.cap = h->L.cap;
    q.short_cap = h->L.cap / 2 * 3;
    q.fmt = h->L.fmt;
    // (A record that does not fit goes to the table by itself, 0.33 ns each of 2.7 M in a call of 2^27 records; the long form
    // takes 60 us more of such a call: as much as one such record of 700.)
    const ull misfits = h->n_records / 512 < (1u << 18) ? 1u << 18 : h->n_records / 512;
    q.misfit_max = (uint32_t)(misfits < 0xFFFFFFFFull ? misfits : 0xFFFFFFFFull);
    q.n_apps = h->cfg.n_apps;
    q.app_w = h->d_appw;
    q.queue = h->queue;
    q.queue_cap = h->L.queue_cap;
    q.force = force ? 1u : 0u;
    q.seq = h->scatter_seq;
    q.told_long = h->h_long;
    q.trace = h->trace;
    CU(h, launch_partition(q, h->n_sms, s));
    h->launches++;
    if (force) h->spill_pending = false;
    return ATREX_OK;
}

static int ingest_launch(atrex_agg* h, const atrex_record_t* recs, uint64_t n, cudaStream_t s) {
    // Small calls go straight into the table (direct.cu).  Measured per 2^20 records: 40 to 65 us that way, 16 to 25
    // by the two-pass route, which costs 110 to 270 us once (directory, drain, fold): made up for after 4 M records.
    // A single call breaks even at 2^17 records once that is spent, at 2^18 where the table is larger than L2.
    // The records so far are those of earlier calls: a call's own pieces are not counted against it, so that every piece
    // of a first host call (2^22 records) goes direct where the table stays in L2.  The link takes 290 us for 2^20 records
    // and hides either route but for the last piece's: counting the pieces takes 25 to 75 us longer at 6 M records, -46
    // to +6 at 12.6 M, 0 to 23 at 20 M, 2 to 150 at 40 M (4 096 to 2^20 keys, uniform, Zipf, one dominant key).
    const bool small_table = h->L.n_slots * 24 <= L2_TABLE_BYTES;
    const bool few_so_far = !h->hot_ready && h->n_records + n <= (1ull << 22);
    const uint64_t direct_max = h->L.hot_slots == 0 ? DIRECT_RECORDS_MAX : (!few_so_far ? 1ull << 17 : (small_table ? 1ull << 22 : 1ull << 18));
    if (n <= direct_max) {
        DirectParams d;
        memset(&d, 0, sizeof(d));
        d.recs = (const uint4*)recs;
        d.n = (uint32_t)n;
        d.n_apps = h->cfg.n_apps;
        d.phase_lim = h->cfg.n_phases << 16;
        d.app_w = h->d_appw;
        d.t = h->table_ref();
        CU(h, launch_direct(d, h->n_sms, s));
        h->launches++;
        return ATREX_OK;
    }
    // Where the entries had to become long, the directory has been empty since: the first call that hears of it builds
    // another, in the form that holds operators of any size, from its own records.  (2^27-record calls, from the second on half of
    // the records with operators that the first did not have: 1 580 to 4 340 us a call without one, 690 with)
    if (h->hot_ready && !h->long_only && *(const volatile ull*)h->h_long == h->trace) {
        const int rc = fold_directory(h, s);
        if (rc != ATREX_OK) return rc;
        h->hot_ready = false;
        h->long_only = true;
    }
    // hot directory from a sample of the first call after create/reset that takes the two-pass route
    if (h->L.hot_slots && !h->hot_ready) {
        HotBuildParams b;
        b.recs = (const uint4*)recs;
        // A record of the sample costs the build 85 ps (2^20: 95 us), a poorer choice the scatter pass up to 4 % where
        // many keys compete: one of 256 records, or one for 16 provisioned keys, whichever is more, from 2^18 on
        // (2^26 records over 2^19 keys 757 -> 729 us with 2^18; 2^30 over 2^24 keys 11.8 ms with 2^20, 12.0 with 2^18)
        ull sample = n / 256 > h->cfg.max_keys / 16 ? n / 256 : h->cfg.max_keys / 16;
        sample = pow2_at_least(sample < HOT_SAMPLE / 4 ? HOT_SAMPLE / 4 : (sample < HOT_SAMPLE ? sample : HOT_SAMPLE));
        b.n_sample = (uint32_t)(n < sample ? n : sample);
        b.stride = n / b.n_sample;
        b.n_apps = h->cfg.n_apps;
        b.n_phases = h->cfg.n_phases;
        b.hot_keys = h->hot_keys;
        b.max_ops = h->long_only ? 0 : h->L.fmt.max_ops;
        b.dur_mask = h->L.fmt.dur_mask();
        b.hot_slots = h->L.hot_slots;
        b.hot_words = (uint32_t*)(h->ws + h->L.off_hot_words);
        b.phase_bits = h->L.fmt.phase_bits;
        for (int words = 0; words < 2; ++words) {
            b.slots[words][0] = scatter_slots(h->L.lp, words != 0);
            b.slots[words][1] = scatter_dominated_slots(h->L.lp, words != 0);
        }
        b.ctl = h->ctl;
        b.sketch = (uint32_t*)h->hot_scratch;
        b.sample = (ull*)(h->hot_scratch + HOT_SAMPLE_OFF);
        b.scratch = (HotBuildScratch*)(h->hot_scratch + HOT_SELECT_OFF);
        b.cand_keys = (ull*)(h->hot_scratch + SKETCH_BYTES);
        b.cand_cnt = (uint32_t*)(h->hot_scratch + SKETCH_BYTES + ((size_t)8 << CAND_BITS));
        b.cand_bits = CAND_BITS;
        CU(h, cudaMemsetAsync(h->hot_scratch, 0, HOT_COUNT_BYTES, s));
        CU(h, launch_hot_build(b, h->n_sms, s));
        h->launches += 6;
        h->hot_ready = true;
    }
    IngestParams p;
    memset(&p, 0, sizeof(p));
    const unsigned char* base = (const unsigned char*)recs;
    uint64_t head = (((uintptr_t)base & 31u) != 0 && n > 0) ? 1 : 0;
    uint64_t n_body = n - head;
    p.recs = recs;
    p.n_recs = n;
    p.body = base + head * 16;
    p.n_pairs = n_body / 2;
    p.n_single = 0;
    if (head) p.single[p.n_single++] = base;
    if (n_body & 1) p.single[p.n_single++] = base + (n - 1) * 16;
    p.n_apps = h->cfg.n_apps;
    p.n_phases = h->cfg.n_phases;
    p.phase_lim = h->cfg.n_phases << 16;
    p.appw_in_smem = h->L.appw_in_smem ? 1u : 0u;
    p.app_w = h->d_appw;
    p.fmt = h->L.fmt;
    p.hot_keys = h->hot_keys;
    p.hot_slots = h->L.hot_slots;
    p.hot_words = (const uint4*)(h->ws + h->L.off_hot_words);
    p.hot_img = h->hot_img;
    p.t = h->table_ref();
    p.spill = h->spill;
    p.spill_cnt = h->spill_cnt;
    p.n_groups = h->L.n_groups;
    p.cap = h->L.cap;
    const ull pairs_per_cta_iter = 2048;
    ull want = (p.n_pairs + pairs_per_cta_iter - 1) / pairs_per_cta_iter;
    int grid = (int)(want < 1 ? 1 : (want > (ull)h->n_sms ? (ull)h->n_sms : want));
    p.drain_above = h->L.cap / 4 * 3;
    p.short_cap = h->L.cap / 2 * 3;       // (the same bytes)
    p.short_drain_above = p.short_cap / 4 * 3;
    p.long_drain_above = p.short_cap / 8 * 5;
    p.seq = ++h->scatter_seq;
    p.img_rows = h->img_rows;
    CU(h, launch_scatter(p, h->hot_ready, grid, s));
    if (h->hot_ready && h->img_rows < (uint32_t)grid) h->img_rows = (uint32_t)grid;
    h->spill_pending = true;
    h->launches++;
    return drain_spill(h, /*force=*/false, s);
}

int atrex_agg_ingest(atrex_agg_t* h, const atrex_record_t* d_records, uint64_t n, void* stream) {
    TraceRange range("atrex_agg_ingest");
    if (!h) return ATREX_ERR_INVALID;
    if (n == 0) return ATREX_OK;
    if (!d_records || ((uintptr_t)d_records & 15u) != 0) return ATREX_ERR_INVALID;
    if (h->n_records + n >= MAX_RECORDS_TOTAL) return ATREX_ERR_STATE;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    h->finalized = false;
    for (uint64_t off = 0; off < n; off += h->L.sub_launch) {
        uint64_t m = n - off < h->L.sub_launch ? n - off : h->L.sub_launch;
        int rc = ingest_launch(h, d_records + off, m, s);
        if (rc != ATREX_OK) return rc;
    }
    h->n_records += n;
    return ATREX_OK;
}

int atrex_agg_ingest_host(atrex_agg_t* h, const atrex_record_t* h_records, uint64_t n, void* stream) {
    TraceRange range("atrex_agg_ingest_host");
    if (!h) return ATREX_ERR_INVALID;
    if (n == 0) return ATREX_OK;
    if (!h_records) return ATREX_ERR_INVALID;
    if (h->n_records + n >= MAX_RECORDS_TOTAL) return ATREX_ERR_STATE;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    h->finalized = false;
    const uint64_t per_piece = STAGING_BYTES / sizeof(atrex_record_t);
    int b = 0;
    for (uint64_t off = 0; off < n; off += per_piece, b ^= 1) {
        uint64_t m = n - off < per_piece ? n - off : per_piece;
        CU(h, cudaStreamWaitEvent(h->copy_stream, h->ev_free[b], 0));
        CU(h, cudaMemcpyAsync(h->staging[b], h_records + off, m * sizeof(atrex_record_t), cudaMemcpyHostToDevice, h->copy_stream));
        CU(h, cudaEventRecord(h->ev_ready[b], h->copy_stream));
        CU(h, cudaStreamWaitEvent(s, h->ev_ready[b], 0));
        int rc = ingest_launch(h, (const atrex_record_t*)h->staging[b], m, s);
        if (rc != ATREX_OK) return rc;
        CU(h, cudaEventRecord(h->ev_free[b], s));
    }
    h->n_records += n;
    return ATREX_OK;
}

int atrex_agg_merge(atrex_agg_t* h, const atrex_entry_t* d_entries, uint64_t n, void* stream) {
    TraceRange range("atrex_agg_merge");
    if (!h) return ATREX_ERR_INVALID;
    if (n == 0) return ATREX_OK;
    if (!d_entries || ((uintptr_t)d_entries & 15u) != 0) return ATREX_ERR_INVALID;
    DeviceGuard guard(h->cfg.device);
    h->finalized = false;
    CU(h, launch_merge(d_entries, n, h->table_ref(), (cudaStream_t)stream));
    h->launches++;
    return ATREX_OK;
}

static GivenTotals given_totals(const uint64_t* total_lo, const uint64_t* total_hi) {
    GivenTotals given;
    memset(&given, 0, sizeof(given));
    if (total_lo) {
        // normalise by the totals over all shards instead of this handle's own
        memcpy(given.lo, total_lo, sizeof(given.lo));
        memcpy(given.hi, total_hi, sizeof(given.hi));
        given.use = 1;
    }
    return given;
}

static uint32_t* hist_half(atrex_agg* h, uint32_t which) { return h->hist_all + (size_t)which * h->cfg.n_phases * TOPK_BINS; }

static int run_totals(atrex_agg* h, const GivenTotals& given, cudaStream_t s) {
    h->hist_at ^= 1u;
    CU(h, launch_totals(h->table_ref(), h->L.n_slots, h->cfg.n_phases, given, hist_half(h, h->hist_at), hist_half(h, h->hist_at ^ 1u), h->n_sms, s));
    h->launches++;
    return ATREX_OK;
}

static FinalizeParams finalize_params(const atrex_agg* h, atrex_entry_t* out, uint64_t cap) {
    FinalizeParams p;
    p.t = h->table_ref();
    p.n_slots = h->L.n_slots;
    p.ctl = h->ctl;
    p.told = h->h_told;
    p.stamp = 0;
    p.work = h->work_ref();
    p.peaks = h->peaks;
    p.out = out;
    p.out_cap = cap;
    return p;
}

static int finalize_impl(atrex_agg_t* h, const atrex_hw_peaks_t* peaks, const uint64_t* total_lo,
                         const uint64_t* total_hi, atrex_entry_t* d_out, uint64_t out_cap, uint64_t* n_out,
                         void* stream);

// Words that a kernel tells (finalize.cu): whether all of them have arrived, and what they say.
static bool all_told(const ulonglong2* words, uint32_t n, uint32_t stamp) {
    const volatile ull* half = (const volatile ull*)words;
    for (uint32_t i = 2 * n; i-- > 0;)
        if (half[i] >> 32 != stamp) return false;
    return true;
}
static void take_told(const ulonglong2* words, uint32_t n, void* out) {
    for (uint32_t i = 0; i < n; ++i) ((ull*)out)[i] = (uint32_t)words[i].x | words[i].y << 32;
}

int atrex_agg_finalize(atrex_agg_t* h, const atrex_hw_peaks_t* peaks, atrex_entry_t* d_out, uint64_t out_cap,
                       uint64_t* n_out, void* stream) {
    return finalize_impl(h, peaks, nullptr, nullptr, d_out, out_cap, n_out, stream);
}

int atrex_agg_finalize_with_totals(atrex_agg_t* h, const atrex_hw_peaks_t* peaks, const uint64_t* total_lo,
                                   const uint64_t* total_hi, atrex_entry_t* d_out, uint64_t out_cap,
                                   uint64_t* n_out, void* stream) {
    if (!total_lo || !total_hi) return ATREX_ERR_INVALID;
    return finalize_impl(h, peaks, total_lo, total_hi, d_out, out_cap, n_out, stream);
}

static int finalize_impl(atrex_agg_t* h, const atrex_hw_peaks_t* peaks, const uint64_t* total_lo,
                         const uint64_t* total_hi, atrex_entry_t* d_out, uint64_t out_cap, uint64_t* n_out,
                         void* stream) {
    TraceRange range("atrex_agg_finalize");
    if (!h || !peaks || !n_out) return ATREX_ERR_INVALID;
    if (d_out && ((uintptr_t)d_out & 15u) != 0) return ATREX_ERR_INVALID;
    if (!d_out) out_cap = 0;
    if (!(std::isfinite(peaks->peak_bw) && peaks->peak_bw > 0)) return ATREX_ERR_INVALID;
    for (int i = 0; i < ATREX_MAX_DTYPES; ++i)
        if (!(std::isfinite(peaks->peak_flops[i]) && peaks->peak_flops[i] > 0)) return ATREX_ERR_INVALID;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    h->peaks = *peaks;
    int rc = drain_spill(h, /*force=*/true, s);
    if (rc != ATREX_OK) return rc;
    const GivenTotals given = given_totals(total_lo, total_hi);
    FinalizeParams fin = finalize_params(h, d_out, out_cap);
    // (the last kernel tells the control block)
    if (h->one_cluster) {
        fin.stamp = (uint32_t)++h->wait_seq;
        h->hist_at ^= 1u;
        CU(h, launch_finalize_small(fin, h->cfg.n_phases, given, hist_half(h, h->hist_at), hist_half(h, h->hist_at ^ 1u), s));
    } else {
        rc = run_totals(h, given, s);
        if (rc != ATREX_OK) return rc;
        fin.stamp = (uint32_t)++h->wait_seq;
        CU(h, launch_emit(fin, h->n_sms, s));
    }
    h->launches++;
    const ulonglong2* const told = h->h_told;
    const uint32_t stamp = fin.stamp;
    CU(h, wait_for_kernel([=] { return all_told(told, CONTROL_WORDS, stamp); }, s));
    if (!all_told(told, CONTROL_WORDS, stamp)) return ATREX_ERR_STATE;   // (cannot happen: the stream is idle)
    take_told(told, CONTROL_WORDS, h->h_ctl);
    *n_out = h->h_ctl->n_out;
    rc = device_status_to_error(h->h_ctl);
    if (rc != ATREX_OK) return rc;
    h->finalized = true;
    h->fin_gen++;
    if (d_out && h->h_ctl->n_out > out_cap) return ATREX_ERR_OUT_TOO_SMALL;
    return ATREX_OK;
}

// The candidates for the best k of all phases in `mask`, sorted, each in its selection region (the long way, see
// finalize.cu).
static int select_phases(atrex_agg* h, uint32_t mask, uint32_t k, cudaStream_t s) {
    TopkCache& cache = h->topk;
    const uint32_t n_phases = h->cfg.n_phases;
    cache.sel_gen = 0;
    TopkAllParams all;
    memset(&all, 0, sizeof(all));
    all.t = h->table_ref();
    all.n_slots = h->L.n_slots;
    all.hist = h->hist_next;
    all.sel = h->sel;
    all.sel_count = h->ctl->sel_count_all;
    all.sel_cap = SEL_CAP;
    // the items to sort stay within what k alone would be padded to
    const ull most = pow2_at_least(k) > TOPK_PICK_MAX ? pow2_at_least(k) : TOPK_PICK_MAX;
    TopkDigitParams digit;
    memset(&digit, 0, sizeof(digit));
    digit.answers = h->h_digit;
    for (uint32_t q = 0; q < n_phases; ++q) {
        if (!((mask >> q) & 1u)) continue;
        cache.total[q] = h->h_ctl->keys_per_phase[q];
        if (cache.total[q] <= k) {
            all.collect_all_mask |= 1u << q;
        } else {
            digit.active_mask |= 1u << q;
            digit.need[q] = k;
        }
    }
    for (uint32_t known = 0; digit.active_mask; ++known) {   // digits known of the phases still active: the first one and `known` - 1 more
        if (known == 0) {
            digit.hist = h->hist_all + (size_t)h->hist_at * n_phases * TOPK_BINS;
        } else {
            if (known > TOPK_DIGITS) return ATREX_ERR_STATE;   // cannot happen: composites are unique
            all.active_mask = digit.active_mask;
            for (uint32_t q = 0, row = 0; q < n_phases; ++q)
                if ((all.active_mask >> q) & 1u) all.row[q] = row++;
            CU(h, cudaMemsetAsync(h->hist_next, 0, (size_t)n_phases * TOPK_BINS * 4, s));
            CU(h, launch_topk_hist(all, h->n_sms, s));
            h->launches++;
            digit.hist = h->hist_next;
        }
        digit.seq = ++h->wait_seq;
        CU(h, launch_topk_digit(digit, n_phases, s));
        h->launches++;
        const volatile TopkDigit* a = h->h_digit;
        const ull want = digit.seq;
        const uint32_t asked = digit.active_mask;
        auto answered = [=] {
            for (uint32_t q = 0; q < n_phases; ++q)
                if (((asked >> q) & 1u) && a[q].seq != want) return false;
            return true;
        };
        CU(h, wait_for_kernel(answered, s));
        if (!answered()) return ATREX_ERR_STATE;               // cannot happen: more than k keys were counted
        for (uint32_t q = 0; q < n_phases; ++q) {
            if (!((asked >> q) & 1u)) continue;
            if (known == 0) all.first[q] = (uint32_t)a[q].bin;
            else all.digit[q][all.n_digits[q]++] = (uint16_t)a[q].bin;
            digit.need[q] -= (uint32_t)a[q].above;
            cache.total[q] = k - digit.need[q] + a[q].in_bin;  // the better ones and those level with the k-th
            if (cache.total[q] <= most) digit.active_mask &= ~(1u << q);
        }
    }
    TopkSortParams sort;
    memset(&sort, 0, sizeof(sort));
    sort.sel = h->sel;
    sort.sel_cap = SEL_CAP;
    CU(h, cudaMemsetAsync(h->ctl->sel_count_all, 0, sizeof(h->ctl->sel_count_all), s));
    for (uint32_t q = 0; q < n_phases; ++q) {
        if (!((mask >> q) & 1u)) continue;
        sort.n_pow2[q] = (uint32_t)pow2_at_least(cache.total[q] < 2 ? 2 : cache.total[q]);
        CU(h, cudaMemsetAsync(h->sel + (size_t)q * SEL_CAP * 4, 0, (size_t)sort.n_pow2[q] * 32, s));   // (the sort wants zeros behind the candidates)
    }
    all.active_mask = mask;
    CU(h, launch_topk_collect_all(all, h->scan_grid(h->L.n_slots, 256 * 4), s));
    CU(h, cudaMemsetAsync(h->ctl->sel_count_all, 0, sizeof(h->ctl->sel_count_all), s));
    CU(h, launch_topk_sort(sort, n_phases, s));
    h->launches += 2;
    cache.sel_gen = h->fin_gen;
    cache.sel_k = k;
    cache.sel_mask = mask;
    return ATREX_OK;
}

int atrex_agg_topk(atrex_agg_t* h, uint32_t phase, uint32_t k, atrex_entry_t* h_out, uint32_t* n_out, void* stream) {
    TraceRange range("atrex_agg_topk");
    if (!h || !n_out || (k && !h_out) || k > ATREX_MAX_TOPK || phase >= h->cfg.n_phases) return ATREX_ERR_INVALID;
    *n_out = 0;
    if (!h->finalized) return ATREX_ERR_STATE;
    if (k == 0) return ATREX_OK;
    if (h->h_ctl->keys_per_phase[phase] == 0) return ATREX_OK;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    TopkCache& cache = h->topk;
    uint32_t long_way = 0;   // the phases that a request of this k cannot answer at once
    for (uint32_t q = 0; q < h->cfg.n_phases; ++q)
        if (h->h_ctl->keys_per_phase[q] != 0) long_way |= 1u << q;
    if (k <= TOPK_PICK_K) {
        // every phase's answer in one go
        ull* const answers = (ull*)(h->h_top + (size_t)h->cfg.n_phases * TOPK_PICK_K);
        if (cache.pick_gen != h->fin_gen || cache.k != k) {
            PickParams p;
            p.fin = finalize_params(h, nullptr, 0);
            p.fin.stamp = (uint32_t)++h->wait_seq;
            p.n_phases = h->cfg.n_phases;
            p.k = k;
            p.hist = h->hist_all + (size_t)h->hist_at * h->cfg.n_phases * TOPK_BINS;
            p.sel = h->pick;
            p.host_top = h->h_top;
            p.host_told = h->h_top_told;
            p.host_n = answers;
            cache.pick_gen = 0;
            const uint32_t n_phases = p.n_phases;
            const uint32_t stamp = p.fin.stamp;
            for (uint32_t q = 0; q < n_phases; ++q) answers[q] = (ull)~stamp << 32;
            CU(h, launch_topk_pick(p, h->one_cluster, h->n_sms, s));
            h->launches += h->one_cluster ? 1 : 2;
            const volatile ull* a = answers;
            const ulonglong2* const rows = k <= TOPK_TOLD_K ? h->h_top_told : nullptr;
            const auto answered = [=] {
                for (uint32_t q = 0; q < n_phases; ++q)
                    if (a[q] >> 32 != stamp || (rows && (uint32_t)a[q] != PICK_NONE && !all_told(rows + (size_t)q * TOPK_TOLD_K * 6, (uint32_t)a[q] * 6, stamp))) return false;
                return true;
            };
            CU(h, wait_for_kernel(answered, s));
            if (!answered()) return ATREX_ERR_STATE;                     // (cannot happen: the stream is idle)
            for (uint32_t q = 0; rows && q < n_phases; ++q)
                if ((uint32_t)a[q] != PICK_NONE) take_told(rows + (size_t)q * TOPK_TOLD_K * 6, (uint32_t)a[q] * 6, h->h_top + (size_t)q * TOPK_PICK_K);
            cache.pick_gen = h->fin_gen;
            cache.k = k;
        }
        const uint32_t m = (uint32_t)((const volatile ull*)answers)[phase];
        if (m != PICK_NONE) {
            memcpy(h_out, h->h_top + (size_t)phase * TOPK_PICK_K, (size_t)m * sizeof(atrex_entry_t));
            *n_out = m;
            return ATREX_OK;
        }
        for (uint32_t q = 0; q < h->cfg.n_phases; ++q)
            if ((uint32_t)((const volatile ull*)answers)[q] != PICK_NONE) long_way &= ~(1u << q);
    }
    if (cache.sel_gen != h->fin_gen || cache.sel_k != k || cache.sel_mask != long_way) {
        const int rc = select_phases(h, long_way, k, s);
        if (rc != ATREX_OK) return rc;
    }
    const ull total = cache.total[phase];
    const uint32_t m = (uint32_t)(total < k ? total : k);
    CU(h, launch_topk_emit(finalize_params(h, h->topk_out, m), h->sel + (size_t)phase * SEL_CAP * 4, m, s));
    h->launches++;
    CU(h, cudaMemcpyAsync(h_out, h->topk_out, (size_t)m * sizeof(atrex_entry_t), cudaMemcpyDeviceToHost, s));
    CU(h, cudaStreamSynchronize(s));
    *n_out = m;
    return ATREX_OK;
}

int atrex_agg_totals(const atrex_agg_t* h, uint64_t* h_lo, uint64_t* h_hi) {
    if (!h || !h_lo || !h_hi) return ATREX_ERR_INVALID;
    if (!h->finalized) return ATREX_ERR_STATE;
    for (int p = 0; p < ATREX_MAX_PHASES; ++p) {
        h_lo[p] = h->h_ctl->total_lo[p];
        h_hi[p] = h->h_ctl->total_hi[p];
    }
    return ATREX_OK;
}

int atrex_agg_stats(atrex_agg_t* h, atrex_stats_t* out, void* stream) {
    TraceRange range("atrex_agg_stats");
    if (!h || !out) return ATREX_ERR_INVALID;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    int rc = drain_spill(h, /*force=*/true, s);
    if (rc != ATREX_OK) return rc;
    rc = run_totals(h, given_totals(nullptr, nullptr), s);
    if (rc != ATREX_OK) return rc;
    CU(h, cudaMemcpyAsync(h->h_ctl, h->ctl, offsetof(Control, acc_lo), cudaMemcpyDeviceToHost, s));
    CU(h, cudaStreamSynchronize(s));
    memset(out, 0, sizeof(*out));
    const Control* c = h->h_ctl;
    out->n_rejected = c->n_rejected;
    out->n_dropped = c->n_dropped;
    for (int p = 0; p < ATREX_MAX_PHASES; ++p) {
        out->total_lo[p] = c->total_lo[p];
        out->total_hi[p] = c->total_hi[p];
        out->keys_per_phase[p] = c->keys_per_phase[p];
        out->n_keys += c->keys_per_phase[p];
        out->n_valid += c->count_per_phase[p];
    }
    out->table_slots = h->L.n_slots;
    out->hot_slots = c->hot_n;
    out->n_spilled = c->n_spilled;
    out->n_overflow = c->n_overflow;
    out->max_spill_fill = c->max_fill;
    out->spill_cap = c->form == FORM_SHORT ? h->L.cap / 2 * 3 : h->L.cap;
    out->n_drains = c->n_drains;
    return device_status_to_error(c);
}

int atrex_agg_hot_directory(atrex_agg_t* h, uint64_t* h_keys, uint32_t cap, uint32_t* n_out, void* stream) {
    if (!h || !n_out || (cap && !h_keys)) return ATREX_ERR_INVALID;
    *n_out = 0;
    if (!h->hot_ready || h->L.hot_slots == 0) return ATREX_OK;
    DeviceGuard guard(h->cfg.device);
    cudaStream_t s = (cudaStream_t)stream;
    ull* image = (ull*)malloc((size_t)h->L.hot_slots * 8);
    if (!image) return ATREX_ERR_NOMEM;
    ull form = FORM_LONG;
    cudaError_t e = cudaMemcpyAsync(image, h->hot_keys, (size_t)h->L.hot_slots * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&form, &h->ctl->form, sizeof(form), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        free(image);
        h->last_cuda_error = (int)e;
        return ATREX_ERR_CUDA;
    }
    uint32_t n = 0;
    for (uint32_t i = 0; form != FORM_LONG_ONLY && i < h->L.hot_slots; ++i) {
        if (image[i] == 0) continue;
        if (n < cap) h_keys[n] = ~image[i];
        ++n;
    }
    free(image);
    *n_out = n;
    return ATREX_OK;
}

const char* atrex_strerror(int status) {
    switch (status) {
        case ATREX_OK: return "ok";
        case ATREX_ERR_INVALID: return "invalid argument";
        case ATREX_ERR_CAPACITY: return "more distinct keys than provisioned";
        case ATREX_ERR_OUT_TOO_SMALL: return "output buffer too small";
        case ATREX_ERR_CUDA: return "CUDA runtime error";
        case ATREX_ERR_TIMEOUT: return "bounded device wait gave up";
        case ATREX_ERR_STATE: return "call not valid in this state";
        case ATREX_ERR_NOMEM: return "workspace too small or allocation failed";
        case ATREX_ERR_TOO_LARGE: return "input larger than the fixed internal buffer";
        case ATREX_ERR_BOUNDS: return "checked build: a kernel index was out of range";
        default: return "unknown status";
    }
}

int atrex_build_has_bounds_checks(void) {
#ifdef ATREX_DEBUG_BOUNDS
    return 1;
#else
    return 0;
#endif
}

int atrex_agg_last_cuda_error(const atrex_agg_t* h) { return h ? h->last_cuda_error : 0; }

uint64_t atrex_agg_launch_count(const atrex_agg_t* h) { return h ? h->launches : 0; }

}  // extern "C"
