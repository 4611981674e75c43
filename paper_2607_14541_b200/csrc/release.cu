// Release artefacts made from a list of aggregated entries: the list in key order, and the
// per-phase ranking with its running share and coverage cut (the construction behind Table 2:
// operators ordered by weight, a "Cum." column beside them).
//
// Both sort (64-bit word, 32-bit entry index) pairs, usually by binning (see "binned sort").  Where the words
// cluster so much that a bin outgrows a CTA's shared memory, a stable least-significant-digit radix sort
// with 8-bit digits takes over (tiles reordered in shared memory, so that every pass writes contiguous
// runs).  For it the ranking order (weighted time descending, key ascending) is a 3-word composite,
// produced word by word, least significant first: key, then ~wt_lo, then ~wt_hi, each word gathered
// through the current permutation.  A digit on which all words agree (the bitwise OR and AND of the words
// match there) is skipped, so a pass is only paid for digits that carry information: 6 of 8 for the key of
// one phase, 3 or fewer for wt_hi.
//
// The running sum is an exact 128-bit prefix sum in rank order (sums of tiles or blocks, a scan of those, a
// local scan), rounded once per row when the share is formed.
#include <cstring>
#include <mutex>

#include "kernels.h"

using namespace atrex;

namespace {

constexpr int SORT_WARPS = 16;                                // 512 threads
constexpr int SORT_ROUNDS = 16;                               // 32 items per warp and round
constexpr uint32_t SORT_TILE = SORT_WARPS * SORT_ROUNDS * 32;  // 8192 items per CTA
constexpr uint32_t SCAN_BLOCK = 1024;
constexpr uint32_t FULL = 0xFFFFFFFFu;

struct ReleaseCtl {       // 256 bytes at the start of the scratch, cleared by every call
    ull counter;          // entries of the phase
    ull word_or, word_and;
    ull total_lo, total_hi;
    ull n_keep, covered_lo, covered_hi;
    ull pad[24];
};
static_assert(sizeof(ReleaseCtl) == 256, "control block is 256 bytes");

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

__device__ __forceinline__ void add128(ull& lo, ull& hi, ull alo, ull ahi) {
    const ull s = lo + alo;
    hi += ahi + (s < lo ? 1ull : 0ull);
    lo = s;
}

// Exact 128-bit sum of two 64-bit halves kept in global memory: the low half's returning add
// tells each adder whether it produced the carry, and carries commute.
__device__ __forceinline__ void atomic_add128(ull* lo, ull* hi, ull alo, ull ahi) {
    const ull old = atomicAdd(lo, alo);
    const ull carry = (old + alo < old) ? 1ull : 0ull;
    if (ahi + carry) atomicAdd(hi, ahi + carry);
}

__device__ __forceinline__ void warp_or_and(ull v_or, ull v_and, ReleaseCtl* ctl) {
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        v_or |= __shfl_xor_sync(FULL, v_or, d);
        v_and &= __shfl_xor_sync(FULL, v_and, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicOr(&ctl->word_or, v_or);
        atomicAnd(&ctl->word_and, v_and);
    }
}

// Sort words for the key order: all entries, word = packed key.
__global__ void __launch_bounds__(256) init_key_words_kernel(const atrex_entry_t* entries, uint32_t n, ull* words,
                                                             uint32_t* idx, ReleaseCtl* ctl) {
    ull v_or = 0, v_and = ~0ull;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const ull key = entries[i].key;
        words[i] = key;
        idx[i] = i;
        v_or |= key;
        v_and &= key;
    }
    warp_or_and(v_or, v_and, ctl);
}

// Entries of `phase` are compacted to (key, index) pairs; their weighted times are summed exactly.
__global__ void __launch_bounds__(256) filter_phase_kernel(const atrex_entry_t* entries, uint32_t n, uint32_t phase,
                                                           ull* words, uint32_t* idx, ReleaseCtl* ctl) {
    ull v_or = 0, v_and = ~0ull, sum_lo = 0, sum_hi = 0;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t n_round = (n + 31u) & ~31u;  // whole warps stay in the loop for the ballots
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_round; i += gridDim.x * blockDim.x) {
        ull key = 0;
        bool mine = false;
        if (i < n) {
            key = entries[i].key;
            mine = (uint32_t)(key >> 48) == phase;
        }
        const uint32_t mask = __ballot_sync(FULL, mine);
        if (mask == 0) continue;
        ull base = 0;
        if (lane == (uint32_t)(__ffs(mask) - 1)) base = atomicAdd(&ctl->counter, (ull)__popc(mask));
        base = __shfl_sync(FULL, base, __ffs(mask) - 1);
        if (mine) {
            const ull pos = base + __popc(mask & ((1u << lane) - 1u));
            words[pos] = key;
            idx[pos] = i;
            v_or |= key;
            v_and &= key;
            add128(sum_lo, sum_hi, entries[i].wt_lo, entries[i].wt_hi);
        }
    }
    warp_or_and(v_or, v_and, ctl);
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const ull olo = __shfl_xor_sync(FULL, sum_lo, d), ohi = __shfl_xor_sync(FULL, sum_hi, d);
        add128(sum_lo, sum_hi, olo, ohi);
    }
    if (lane == 0 && (sum_lo | sum_hi)) atomic_add128(&ctl->total_lo, &ctl->total_hi, sum_lo, sum_hi);
}

// word[r] = ~(wt_lo or wt_hi) of the entry at the current position r: ascending order of the
// complement is descending order of the weighted time.
__global__ void __launch_bounds__(256) gather_wt_words_kernel(const atrex_entry_t* entries, const uint32_t* idx,
                                                              uint32_t m, int high, ull* words, ReleaseCtl* ctl) {
    ull v_or = 0, v_and = ~0ull;
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < m; r += gridDim.x * blockDim.x) {
        const atrex_entry_t* e = entries + idx[r];
        const ull w = ~(high ? e->wt_hi : e->wt_lo);
        words[r] = w;
        v_or |= w;
        v_and &= w;
    }
    warp_or_and(v_or, v_and, ctl);
}

// ---- one radix pass: per-tile digit counts, per-digit exclusive scan over the tiles plus digit
// totals, stable scatter (which adds the scan of the 256 digit totals itself)

__global__ void __launch_bounds__(SORT_WARPS * 32) radix_hist_kernel(const ull* words, uint32_t m, int shift,
                                                                     uint32_t* hist, uint32_t n_tiles) {
    __shared__ uint32_t h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t tile = blockIdx.x * SORT_TILE;
    for (uint32_t j = threadIdx.x; j < SORT_TILE; j += SORT_WARPS * 32) {
        const uint32_t i = tile + j;
        if (i < m) atomicAdd(&h[(uint32_t)(words[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 256) hist[(size_t)threadIdx.x * n_tiles + blockIdx.x] = h[threadIdx.x];
}

// One CTA per digit value: exclusive scan of that digit's counts over the tiles (a contiguous row,
// 1024 at a time with a running carry), and the digit's total to bin_total[digit].
__global__ void __launch_bounds__(SCAN_BLOCK) radix_scan_kernel(uint32_t* hist, uint32_t n_tiles, uint32_t* bin_total) {
    __shared__ uint32_t warp_sum[32];
    uint32_t* row = hist + (size_t)blockIdx.x * n_tiles;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < n_tiles; base += SCAN_BLOCK) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t c = i < n_tiles ? row[i] : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, incl, d);
            if (lane >= (uint32_t)d) incl += o;
        }
        if (lane == 31) warp_sum[w] = incl;
        __syncthreads();
        if (w == 0) {
            uint32_t iv = warp_sum[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(FULL, iv, d);
                if (lane >= (uint32_t)d) iv += o;
            }
            warp_sum[lane] = iv;  // inclusive over warps
        }
        __syncthreads();
        if (i < n_tiles) row[i] = carry + (w ? warp_sum[w - 1] : 0u) + incl - c;
        carry += warp_sum[31];
        __syncthreads();  // warp_sum is reused by the next round
    }
    if (threadIdx.x == 0) bin_total[blockIdx.x] = carry;
}

// Stable: item order inside a tile is (warp, round, lane) = input order; a lane's rank among
// equal digits is (items of earlier warps) + (earlier rounds of its warp) + (lower lanes of its
// round), and tiles are ordered by the scanned (digit, tile) counters.  The tile is first put in
// digit order in shared memory and then written out run by run, so that the global stores are
// contiguous per digit (about 32 items per digit and tile) instead of one scattered 12-byte piece
// per item.
constexpr size_t SCATTER_SMEM = (size_t)SORT_TILE * 12;   // words (8 B) and indices (4 B) of one tile

__global__ void __launch_bounds__(SORT_WARPS * 32) radix_scatter_kernel(const ull* words_in, const uint32_t* idx_in,
                                                                        ull* words_out, uint32_t* idx_out, uint32_t m,
                                                                        int shift, const uint32_t* hist,
                                                                        uint32_t n_tiles, const uint32_t* bin_total) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    ull* s_words = reinterpret_cast<ull*>(sort_smem);                          // [SORT_TILE] the tile in digit order
    uint32_t* s_idx = reinterpret_cast<uint32_t*>(sort_smem + (size_t)SORT_TILE * 8);
    __shared__ uint32_t wh[SORT_WARPS][256];
    __shared__ uint32_t bin_base[256];   // exclusive scan of the digit totals (global)
    __shared__ uint32_t bin_warp[8];
    __shared__ uint32_t tile_base[256];  // first position of digit d inside this tile's digit order
    __shared__ uint32_t tile_warp[8];
    __shared__ uint32_t out_base[256];   // global position of this tile's first item of digit d
    for (uint32_t j = threadIdx.x; j < SORT_WARPS * 256; j += SORT_WARPS * 32) (&wh[0][0])[j] = 0;
    __syncthreads();
    const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    const uint32_t tile_start = blockIdx.x * SORT_TILE;
    const uint32_t first = tile_start + w * (SORT_ROUNDS * 32) + lane;
    uint32_t packed[SORT_ROUNDS];  // digit | rank inside the warp << 9
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const uint32_t i = first + r * 32;
        const bool valid = i < m;
        const uint32_t d = valid ? (uint32_t)(words_in[i] >> shift) & 255u : 256u + lane;  // padding never groups
        const uint32_t same = __match_any_sync(FULL, d);
        const uint32_t base = valid ? wh[w][d] : 0u;
        __syncwarp();
        if (valid && (same & lt) == 0) wh[w][d] = base + __popc(same);
        __syncwarp();
        packed[r] = d | ((base + __popc(same & lt)) << 9);
    }
    __syncthreads();
    uint32_t tile_count = 0;
    if (threadIdx.x < 256) {
        // this digit's items in the tile, per warp -> running offsets; the digit totals -> global bases
#pragma unroll
        for (int k = 0; k < SORT_WARPS; ++k) {
            const uint32_t c = wh[k][threadIdx.x];
            wh[k][threadIdx.x] = tile_count;     // items of this digit in earlier warps
            tile_count += c;
        }
        const uint32_t c = bin_total[threadIdx.x];
        uint32_t incl = c, tincl = tile_count;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, incl, d), to = __shfl_up_sync(FULL, tincl, d);
            if (lane >= (uint32_t)d) {
                incl += o;
                tincl += to;
            }
        }
        if (lane == 31) {
            bin_warp[w] = incl;
            tile_warp[w] = tincl;
        }
        bin_base[threadIdx.x] = incl - c;
        tile_base[threadIdx.x] = tincl - tile_count;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t g = bin_base[threadIdx.x] + hist[(size_t)threadIdx.x * n_tiles + blockIdx.x], t = tile_base[threadIdx.x];
        for (uint32_t k = 0; k < w; ++k) {
            g += bin_warp[k];
            t += tile_warp[k];
        }
        out_base[threadIdx.x] = g;
        tile_base[threadIdx.x] = t;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const uint32_t i = first + r * 32;
        if (i < m) {
            const uint32_t d = packed[r] & 511u;
            const uint32_t at = tile_base[d] + wh[w][d] + (packed[r] >> 9);
            s_words[at] = words_in[i];
            s_idx[at] = idx_in[i];
        }
    }
    __syncthreads();
    const uint32_t tile_n = min(SORT_TILE, m - tile_start);
    for (uint32_t j = threadIdx.x; j < tile_n; j += SORT_WARPS * 32) {
        const ull word = s_words[j];
        const uint32_t d = (uint32_t)(word >> shift) & 255u;
        const uint32_t pos = out_base[d] + (j - tile_base[d]);
        words_out[pos] = word;
        idx_out[pos] = s_idx[j];
    }
}

__global__ void __launch_bounds__(256) gather_entries_kernel(const atrex_entry_t* entries, const uint32_t* idx,
                                                             uint32_t m, atrex_entry_t* out) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < m; r += gridDim.x * blockDim.x)
        out[r] = entries[idx[r]];
}

// ---- exact running sum in rank order

__device__ __forceinline__ void block_scan128(ull& lo, ull& hi, ull (*warp_tot)[2], ull& block_lo, ull& block_hi) {
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const ull olo = __shfl_up_sync(FULL, lo, d), ohi = __shfl_up_sync(FULL, hi, d);
        if (lane >= (uint32_t)d) add128(lo, hi, olo, ohi);
    }
    if (lane == 31) {
        warp_tot[w][0] = lo;
        warp_tot[w][1] = hi;
    }
    __syncthreads();
    if (w == 0) {
        ull tlo = warp_tot[lane][0], thi = warp_tot[lane][1];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const ull olo = __shfl_up_sync(FULL, tlo, d), ohi = __shfl_up_sync(FULL, thi, d);
            if (lane >= (uint32_t)d) add128(tlo, thi, olo, ohi);
        }
        warp_tot[lane][0] = tlo;  // inclusive over warps
        warp_tot[lane][1] = thi;
    }
    __syncthreads();
    if (w > 0) add128(lo, hi, warp_tot[w - 1][0], warp_tot[w - 1][1]);
    block_lo = warp_tot[31][0];
    block_hi = warp_tot[31][1];
}

__global__ void __launch_bounds__(SCAN_BLOCK) rank_block_sums_kernel(const atrex_entry_t* entries, const uint32_t* idx,
                                                                     uint32_t m, ull* bsums) {
    __shared__ ull warp_tot[32][2];
    const uint32_t r = blockIdx.x * SCAN_BLOCK + threadIdx.x;
    ull lo = 0, hi = 0;
    if (r < m) {
        const atrex_entry_t* e = entries + idx[r];
        lo = e->wt_lo;
        hi = e->wt_hi;
    }
    ull blo, bhi;
    block_scan128(lo, hi, warp_tot, blo, bhi);
    if (threadIdx.x == 0) {
        bsums[2 * blockIdx.x] = blo;
        bsums[2 * blockIdx.x + 1] = bhi;
    }
}

// Exclusive scan of the block sums by one CTA, 1024 at a time with a running carry-in.
__global__ void __launch_bounds__(SCAN_BLOCK) rank_scan_sums_kernel(ull* bsums, uint32_t nb) {
    __shared__ ull warp_tot[32][2];
    ull run_lo = 0, run_hi = 0;
    for (uint32_t base = 0; base < nb; base += SCAN_BLOCK) {
        const uint32_t b = base + threadIdx.x;
        ull lo = 0, hi = 0;
        if (b < nb) {
            lo = bsums[2 * b];
            hi = bsums[2 * b + 1];
        }
        const ull own_lo = lo, own_hi = hi;
        ull blo, bhi;
        block_scan128(lo, hi, warp_tot, blo, bhi);
        if (b < nb) {
            // exclusive = carry-in + inclusive - own
            ull elo = lo - own_lo, ehi = hi - own_hi - (lo < own_lo ? 1ull : 0ull);
            add128(elo, ehi, run_lo, run_hi);
            bsums[2 * b] = elo;
            bsums[2 * b + 1] = ehi;
        }
        add128(run_lo, run_hi, blo, bhi);
        __syncthreads();  // warp_tot is reused by the next round
    }
}

__device__ __forceinline__ bool less128(ull alo, ull ahi, ull blo, ull bhi) {
    return ahi < bhi || (ahi == bhi && alo < blo);
}

// Row r of the ranking: the entry, its running share fl(fl(prefix) / fl(T)), and the coverage cut
// (the one row whose exclusive prefix is below the needed sum and whose inclusive prefix reaches it).
__global__ void __launch_bounds__(SCAN_BLOCK) rank_emit_kernel(const atrex_entry_t* entries, const uint32_t* idx,
                                                               uint32_t m, const ull* bsums, ull total_lo, ull total_hi,
                                                               ull need_lo, ull need_hi, atrex_entry_t* out,
                                                               double* cum, uint32_t out_cap, ReleaseCtl* ctl) {
    __shared__ ull warp_tot[32][2];
    const uint32_t r = blockIdx.x * SCAN_BLOCK + threadIdx.x;
    ull lo = 0, hi = 0;
    const atrex_entry_t* e = nullptr;
    if (r < m) {
        e = entries + idx[r];
        lo = e->wt_lo;
        hi = e->wt_hi;
    }
    const ull own_lo = lo, own_hi = hi;
    ull blo, bhi;
    block_scan128(lo, hi, warp_tot, blo, bhi);
    if (r >= m) return;
    add128(lo, hi, bsums[2 * blockIdx.x], bsums[2 * blockIdx.x + 1]);  // inclusive prefix of the whole list
    const ull ex_lo = lo - own_lo, ex_hi = hi - own_hi - (lo < own_lo ? 1ull : 0ull);
    if ((need_lo | need_hi) && less128(ex_lo, ex_hi, need_lo, need_hi) && !less128(lo, hi, need_lo, need_hi)) {
        ctl->n_keep = (ull)r + 1;
        ctl->covered_lo = lo;
        ctl->covered_hi = hi;
    }
    if (r < out_cap) {
        out[r] = *e;
        cum[r] = (total_lo | total_hi) ? __ddiv_rn(u128_to_f64_rn(hi, lo), u128_to_f64_rn(total_hi, total_lo)) : 0.0;
    }
}

// ---- binned sort ----------------------------------------------------------------------------------
// The usual way to both orders.  Every item gets a 64-bit word whose order is the wanted one (ties aside),
// and moves twice: to its bin (up to 2^14 equal ranges of the word), then, a tile of neighbouring bins at a
// time, to its place -- a CTA sorts the tile's items in shared memory and gathers their entries, so that
// the only random traffic is one read of each entry.
//   key order   word = the key's fields in mixed radix, (phase * ops + op) * shapes + shape with the fields'
//               largest values as radices: neighbouring words for neighbouring keys, so the bins fill evenly
//   ranking     word = complement of {bit length of the weighted time, its next 57 bits}: a logarithmic scale
//               on which weights that span many orders of magnitude spread; what the 57 bits leave equal is
//               compared in full
// Nothing is read back in between: the item count, the word range and the bins stay on the device, and the
// grids are sized for the caller's n.  A word distribution that puts too much into one bin for a CTA's
// shared memory (thousands of equal weights, say) raises a flag, the remaining kernels do nothing, and the
// call starts over with the radix sort below.
// 15.6 M entries: key order 2.20 -> 0.86 ms against that radix sort alone (four passes and a gather in
// 48-byte pieces); bound by the DRAM reads of the random gather.
constexpr uint32_t BIN_BITS_MAX = 14, BIN_THREADS = 512;
constexpr uint32_t SHARE_THREADS = 1024;     // counting and moving: one CTA per SM, for long runs
constexpr uint32_t CURSORS_MAX = 1u << 14;
// A tile is the bins that start in one window of 2^log_step positions: 2 048, or 512 where a list is so short that larger tiles would
// leave SMs without one and make every phase of a tile's sort longer (tile kernel, key order of 10 000 entries 12.7 -> 7.9 us, 150 000
// 13.5 -> 9.3, 250 000 13.2 -> 15.4): up to there two tiles per SM are enough.  A ranking, of which the tiles of other phases are empty, takes windows of
// 1 024 up to twice that (whole call with windows of 2 048 / 1 024 / 512: 155 000 entries of one phase 62 / 57 / 61 us, 250 000 62 / 60 / 66, 299 000
// 66 / 63 / 70; a phase of two of 250 000 62 / 55 / 59; from 310 000 on no better than 2 048).
constexpr uint32_t TILE_LOG_STEP = 11, MIDDLE_LOG_STEP = 10, SMALL_LOG_STEP = 9;
constexpr uint64_t SMALL_LIST_MAX = 150000, MIDDLE_RANKING_MAX = 300000;
constexpr uint32_t TILE_GROUP = 64;         // tiles whose weighted times are summed
constexpr uint32_t TILE_CAP = 6144;         // ... and has at most this many items
constexpr uint32_t TILE_LOCAL_BINS = 4096, SMALL_LOCAL_BINS = 1024, TILE_THREADS = 512, TILE_HELD = 5, GATHER_LOADS = 6;
constexpr uint32_t TILE_CLASH_MAX = 24;     // larger local bins are crowded: some are sorted by a warp or the CTA each,
constexpr uint32_t TILE_CROWDED = 32;       // more of them send the tile to the comparison network
constexpr uint32_t TILE_SMALL_CROWD = 64;   // sorted by a warp each, side by side, which takes 12 us; the whole CTA takes 4 for one,
constexpr uint32_t TILE_CROWDED_FEW = 3;    // so that so many are sorted one after the other
// From so many items on, half of them alike in their leading bits, a local bin has ties: by insertion every comparison would read two
// entries, so a warp sorts it (tile kernel of a ranking by insertion / now: 100 groups of 8 equal weights in one tile of 75 000 entries 66 / 36 us,
// 100 of 24 116 / 50; every weight 8 times, 700 000 entries 187 / 126, 3 million 617 / 415, 24 times 1 780 / 496; up to 32 of those bins by the whole CTA
// one after the other, the rest by insertion: 229, 178, 366, 1 213 and 2 074).
constexpr uint32_t TILE_TIES = 8;
constexpr size_t TILE_SMEM = (size_t)TILE_CAP * 8 + TILE_LOCAL_BINS * 4;    // (what it leaves of two CTAs is L1 for the gather; with
// more than 1 KB of static shared memory beside it less is left: 10 % slower)
constexpr uint32_t COUNT_SORT_MAX = 8192;   // up to here one kernel ranks every key by counting

struct BinCtl {                  // at the start of the scratch, cleared by every call (with the bins behind it)
    ull counter;                 // items (entries of the phase)
    ull max_word, max_nword;     // largest word and largest complement of a word
    ull max_phase, max_op, max_shape;
    ull total_lo, total_hi;
    ull need_lo, need_hi;        // coverage cut: smallest sufficient prefix sum
    ull overflow;                // a bin (or the total) is too large: nothing more is done
    ull pad[5];
};
static_assert(sizeof(BinCtl) == 128, "half of the control block");

// CTAs of a call's last kernel that are through, by the call's report slot; back at 0 after the last one
__device__ uint32_t g_finished[REPORT_SLOTS];

// The last act of every CTA of a call's last kernel (all of its threads): the last CTA tells the host, which
// notices that several microseconds before the stream counts as idle.
__device__ __forceinline__ void finish_call(BinReport* report, uint32_t slot) {
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicInc(&g_finished[slot], gridDim.x - 1) == gridDim.x - 1) {
        __threadfence_system();
        *(volatile ull*)&report->done = 1;
    }
}

struct BinSort {                 // what the kernels share
    BinCtl* ctl;
    BinReport* report;
    const atrex_entry_t* entries;
    ull* words;                  // [n] raw words: keys (key order), words (ranking)
    uint32_t* idx;               // [n] (ranking) entry of each word
    ulonglong2* ranked_wt;       // [n] (ranking) in the place of both once they are read: the ranked rows' weighted times
    ull* items;                  // [n] in bin order: leading 32 bits of the word's place in the range, then the entry
    uint32_t* bins;              // [1 << bits] counts, then each bin's cursor number
    uint32_t* cursors;           // [n_cursors] where the next item of a tile (by_tile) or bin goes
    uint32_t* tile_start;        // [tiles + 1]
    uint32_t n_cursors;
    uint32_t log_step;           // a tile's window of positions
    bool by_tile;                // items of a tile lie in any order, not bin by bin
    ulonglong2* tile_sum;        // (ranking) [tiles] weighted time
    ulonglong2* group_sum;       // (ranking) ... of TILE_GROUP tiles
    uint32_t n;                  // upper bound of the item count
    uint32_t bits;
    bool ranking;
    uint32_t slot;               // the report's number
    uint32_t turns;              // parts of the cursors that step 4 serves one after the other
};

__host__ __device__ __forceinline__ uint32_t tiles_of(const BinSort& b, uint32_t items) { return (uint32_t)(((uint64_t)items + (1u << b.log_step) - 1) >> b.log_step); }
__device__ __forceinline__ uint32_t item_count(const BinSort& b) { return b.ranking ? (uint32_t)b.ctl->counter : b.n; }

__device__ __forceinline__ ull rank_word(ull lo, ull hi) {
    if ((lo | hi) == 0) return ~0ull;
    const int e = hi ? 128 - __clzll((long long)hi) : 64 - __clzll((long long)lo);
    // the 57 bits below the leading one
    ull m;
    if (e >= 58) {
        const int s = e - 58;
        m = s == 0 ? lo : (s < 64 ? (lo >> s) | (hi << (64 - s)) : hi >> (s - 64));
    } else {
        m = lo << (58 - e);
    }
    return ~(((ull)e << 57) | (m & ((1ull << 57) - 1)));
}

// Word of a key once the fields' largest values are known.
struct KeyRadix {
    ull ops, shapes;
    __device__ __forceinline__ explicit KeyRadix(const BinCtl* c) : ops(c->max_op + 1), shapes(c->max_shape + 1) {}
    __device__ __forceinline__ ull word(ull key) const {
        return ((key >> 48) * ops + ((key >> 32) & 0xFFFFu)) * shapes + (key & 0xFFFFFFFFull);
    }
};

// The words' range cut into equal bins, and into 2^32 steps for the items (all of it, where it is no wider).
struct BinRange {
    ull low, scale;
    uint32_t last;
    int shift;
    __device__ __forceinline__ BinRange(const BinSort& b, const KeyRadix& r) {
        low = b.ranking ? ~b.ctl->max_nword : 0ull;
        const ull span = b.ranking ? b.ctl->max_word - low : (b.ctl->max_phase + 1) * r.ops * r.shapes - 1;
        const int len = 64 - __clzll((long long)span);
        shift = len > 32 ? len - 32 : 0;
        last = (1u << b.bits) - 1u;
        // bin = floor(place * bins / (span + 1)) up to rounding, which keeps the order of the bins
        const double s = ldexp((double)(1u << b.bits), 64) / ((double)span + 1.0);
        scale = s >= 18446744073709549568.0 ? ~0ull : (ull)s;
    }
    __device__ __forceinline__ uint32_t bin(ull word) const { return min(last, (uint32_t)__umul64hi(word - low, scale)); }
    __device__ __forceinline__ ull item(ull word, uint32_t entry) const { return ((word - low) >> shift) << 32 | entry; }
};

template <typename T>
__device__ __forceinline__ T block_reduce(T v, T (*op)(T, T), T* s_part) {   // result in thread 0
#pragma unroll
    for (int d = 16; d; d >>= 1) v = op(v, __shfl_xor_sync(FULL, v, d));
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < (blockDim.x >> 5) ? s_part[threadIdx.x] : s_part[0];
#pragma unroll
        for (int d = 16; d; d >>= 1) v = op(v, __shfl_xor_sync(FULL, v, d));
    }
    __syncthreads();
    return v;
}
__device__ __forceinline__ ull max_ull(ull a, ull b) { return a > b ? a : b; }

// 0. the control block, the sums of groups of tiles and the bins behind it cleared (a kernel in the chain: a memset breaks it, 3 us each side)
__global__ void __launch_bounds__(BIN_THREADS) bin_clear_kernel(uint4* at, uint32_t n) {
    grid_dependency_wait();
    const uint32_t i = blockIdx.x * BIN_THREADS + threadIdx.x;
    if (i < n) at[i] = make_uint4(0, 0, 0, 0);
    grid_dependents_launch();
}

// 1a. (key order) the keys side by side, and the largest value of each field
__global__ void __launch_bounds__(BIN_THREADS) bin_keys_kernel(const BinSort b) {
    __shared__ ull s_part[32];
    grid_dependency_wait();
    ull mp = 0, mo = 0, ms = 0;
    const uint32_t stride = gridDim.x * BIN_THREADS;
    for (uint32_t i0 = blockIdx.x * BIN_THREADS + threadIdx.x; i0 < b.n; i0 += 4 * stride) {
        ull key[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) key[u] = i0 + u * stride < b.n ? b.entries[i0 + u * stride].key : 0ull;
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            if (i0 + u * stride >= b.n) continue;
            b.words[i0 + u * stride] = key[u];
            mp = max_ull(mp, key[u] >> 48);
            mo = max_ull(mo, (key[u] >> 32) & 0xFFFFu);
            ms = max_ull(ms, key[u] & 0xFFFFFFFFull);
        }
    }
    grid_dependents_launch();
    mp = block_reduce(mp, max_ull, s_part);
    mo = block_reduce(mo, max_ull, s_part);
    ms = block_reduce(ms, max_ull, s_part);
    if (threadIdx.x == 0) {
        atomicMax(&b.ctl->max_phase, mp);
        atomicMax(&b.ctl->max_op, mo);
        atomicMax(&b.ctl->max_shape, ms);
    }
}

// 1b. (ranking) the phase's entries: words and indices side by side in any order, word range, exact total.  Bound by the entries' DRAM
//     reads, 4.4 TB/s (weights asked for once the phase was known: 3.1 M entries 38 us, now 34; 15 M 154, now 130; the next round's lines
//     prefetched into L2 as well: 40 and 140; a list in key order, where most warps have nothing to take, one phase of eight of 12 M 100 and 100).
__global__ void __launch_bounds__(BIN_THREADS) bin_phase_kernel(const BinSort b, uint32_t phase) {
    constexpr uint32_t PER = 4;
    __shared__ ull s_part[32];
    __shared__ uint32_t s_warp[BIN_THREADS / 32], s_base;
    grid_dependency_wait();
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    ull top = 0, ntop = 0, sum_lo = 0, sum_hi = 0;
    for (uint32_t t0 = blockIdx.x * (BIN_THREADS * PER); t0 < b.n; t0 += gridDim.x * (BIN_THREADS * PER)) {
        bool mine[PER];
        uint32_t place[PER], run = 0;
        ull lo[PER], hi[PER];
#pragma unroll
        for (uint32_t u = 0; u < PER; ++u) {   // (the weights are asked for with the keys: the lines are the same, mostly)
            const uint32_t i = t0 + u * BIN_THREADS + threadIdx.x;
            mine[u] = i < b.n && (uint32_t)(b.entries[i].key >> 48) == phase;
            lo[u] = i < b.n ? b.entries[i].wt_lo : 0ull;
            hi[u] = i < b.n ? b.entries[i].wt_hi : 0ull;
        }
#pragma unroll
        for (uint32_t u = 0; u < PER; ++u) {
            const uint32_t votes = __ballot_sync(FULL, mine[u]);
            place[u] = run + __popc(votes & ((1u << lane) - 1u));
            run += __popc(votes);
        }
        if (lane == 0) s_warp[w] = run;
        __syncthreads();
        if (threadIdx.x < 32) {
            const uint32_t c = lane < BIN_THREADS / 32 ? s_warp[lane] : 0u;
            uint32_t incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(FULL, incl, d);
                if (lane >= (uint32_t)d) incl += o;
            }
            if (lane == 31) s_base = incl ? (uint32_t)atomicAdd(&b.ctl->counter, (ull)incl) : 0u;
            if (lane < BIN_THREADS / 32) s_warp[lane] = incl - c;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t u = 0; u < PER; ++u) {
            if (!mine[u]) continue;
            const uint32_t i = t0 + u * BIN_THREADS + threadIdx.x, pos = s_base + s_warp[w] + place[u];
            const ull word = rank_word(lo[u], hi[u]);
            b.words[pos] = word;
            b.idx[pos] = i;
            top = max_ull(top, word);
            ntop = max_ull(ntop, ~word);
            add128(sum_lo, sum_hi, lo[u], hi[u]);
        }
        __syncthreads();   // s_warp and s_base are reused
    }
    grid_dependents_launch();
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const ull olo = __shfl_xor_sync(FULL, sum_lo, d), ohi = __shfl_xor_sync(FULL, sum_hi, d);
        add128(sum_lo, sum_hi, olo, ohi);
    }
    if (lane == 0 && (sum_lo | sum_hi)) atomic_add128(&b.ctl->total_lo, &b.ctl->total_hi, sum_lo, sum_hi);
    top = block_reduce(top, max_ull, s_part);
    ntop = block_reduce(ntop, max_ull, s_part);
    if (threadIdx.x == 0) {
        atomicMax(&b.ctl->max_word, top);
        atomicMax(&b.ctl->max_nword, ntop);
    }
}

// The share of the items that CTA blockIdx.x counts (step 2) and moves (step 4).
__device__ __forceinline__ void bin_share(uint32_t m, uint32_t& first, uint32_t& end) {
    const uint32_t share = (m + gridDim.x - 1) / gridDim.x;
    first = min(m, blockIdx.x * share);
    end = min(m, first + share);
}

// Counts the CTA's items per place(bin).
template <typename Place>
__device__ __forceinline__ void bin_count_share(const BinSort& b, const BinRange& range, const KeyRadix& radix, uint32_t first, uint32_t end,
                                                uint32_t* s_bins, Place place) {
    for (uint32_t i = first + threadIdx.x; i < end; i += 4 * SHARE_THREADS) {   // four loads per thread in flight
        ull w[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) w[u] = i + u * SHARE_THREADS < end ? b.words[i + u * SHARE_THREADS] : 0ull;
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
            if (i + u * SHARE_THREADS < end) atomicAdd(&s_bins[place(range.bin(b.ranking ? w[u] : radix.word(w[u])))], 1u);
    }
}

// 2. items per bin
__global__ void __launch_bounds__(SHARE_THREADS) bin_count_kernel(const BinSort b) {
    extern __shared__ __align__(16) uint32_t s_bins[];
    for (uint32_t i = threadIdx.x; i < 1u << b.bits; i += SHARE_THREADS) s_bins[i] = 0;
    __syncthreads();
    grid_dependency_wait();
    uint32_t first, end;
    bin_share(item_count(b), first, end);
    const KeyRadix radix(b.ctl);
    const BinRange range(b, radix);
    bin_count_share(b, range, radix, first, end, s_bins, [](uint32_t bin) { return bin; });
    grid_dependents_launch();
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 1u << b.bits; i += SHARE_THREADS)
        if (s_bins[i]) atomicAdd(&b.bins[i], s_bins[i]);
}

// 3. where each bin and each tile starts; a bin that no tile can hold ends the attempt (one CTA)
//    (ranking) and the sum that the coverage cut needs: the smallest k with 10^6 * prefix_k >= ppm * T, i.e.
//    prefix_k >= ceil(ppm * T / 10^6)
__global__ void __launch_bounds__(1024) bin_scan_kernel(const BinSort b, uint32_t coverage_ppm) {
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_max;
    grid_dependency_wait();
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, m = item_count(b);
    const uint32_t n_bins = 1u << b.bits, per = (n_bins + 1023) / 1024, first = threadIdx.x * per;
    if (threadIdx.x == 0) s_max = 0;
    if (b.ranking && threadIdx.x == 1023) {       // (while the others wait for the bins)
        BinReport* r = b.report;
        BinCtl* ctl = b.ctl;
        r->counter = ctl->counter;
        r->total_lo = ctl->total_lo;
        r->total_hi = ctl->total_hi;
        const unsigned __int128 total = ((unsigned __int128)ctl->total_hi << 64) | ctl->total_lo;
        const unsigned __int128 need = ((unsigned __int128)coverage_ppm * total + 999999u) / 1000000u;   // (not asked for, where that wraps)
        ctl->need_lo = (ull)need;
        ctl->need_hi = (ull)(need >> 64);
    }
    __syncthreads();
    uint32_t c[1u << (BIN_BITS_MAX - 10)];
    uint32_t sum = 0, most = 0;
#pragma unroll
    for (uint32_t u = 0; u < 1u << (BIN_BITS_MAX - 10); u += 4) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (u < per && first + u < n_bins) {
            if (per >= 4) {
                v = *reinterpret_cast<const uint4*>(b.bins + first + u);
            } else {
                v.x = b.bins[first];
                if (per == 2) v.y = b.bins[first + 1];
            }
        }
        c[u] = v.x; c[u + 1] = v.y; c[u + 2] = v.z; c[u + 3] = v.w;
    }
#pragma unroll
    for (uint32_t u = 0; u < 1u << (BIN_BITS_MAX - 10); ++u) {
        sum += c[u];
        most = max(most, c[u]);
    }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(FULL, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_warp[w] = incl;
    atomicMax(&s_max, most);
    __syncthreads();
    if (w == 0) {
        uint32_t v = s_warp[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, v, d);
            if (lane >= (uint32_t)d) v += o;
        }
        s_warp[lane] = v;
    }
    __syncthreads();
    uint32_t at = incl - sum + (w ? s_warp[w - 1] : 0u);
    // tile j starts at the first bin start at or beyond j * 2^log_step (tile 0 at 0)
    const uint32_t n_tiles = tiles_of(b, b.n);
#pragma unroll
    for (uint32_t u = 0; u < 1u << (BIN_BITS_MAX - 10); ++u) {
        if (u >= per || first + u >= n_bins) continue;
        // (a bin belongs to the tile whose window it starts in)
        b.bins[first + u] = b.by_tile ? at >> b.log_step : first + u;
        if (!b.by_tile) b.cursors[first + u] = at;
        const uint32_t next = at + c[u];
        for (uint32_t j = (at >> b.log_step) + 1; j <= next >> b.log_step; ++j) {
            b.tile_start[j] = next;
            if (b.by_tile && j < b.n_cursors) b.cursors[j] = next;
        }
        at = next;
    }
    if (threadIdx.x == 0) {
        b.tile_start[0] = 0;
        if (b.by_tile) b.cursors[0] = 0;
        for (uint32_t j = (m >> b.log_step) + 1; j <= n_tiles; ++j) b.tile_start[j] = m;
        const bool overflow = s_max + (1u << b.log_step) > TILE_CAP;
        b.report->overflow = overflow;
        const bool too_large = b.ranking && (b.ctl->total_hi >> 44) != 0;      // T * 10^6 must fit 128 bits
        b.report->too_large = too_large;
        b.ctl->overflow = overflow || too_large;
    }
}

// 4. items to their tiles (or bins, where there are more tiles than a CTA can keep cursors for), in any order
//    within: the CTA counts its share once more, reserves a range at each cursor with one global atomic, and
//    writes.  Cursors per tile make for runs twice as long as cursors per bin, which keeps the partly written
//    sectors of all CTAs within L2.  From 2 048 cursors on those would take 40 MB and more: the CTAs go over their
//    shares twice, for one half of the cursors each time (15 M items: 396 -> 300 us; three and four times: the same).
__global__ void __launch_bounds__(SHARE_THREADS) bin_scatter_kernel(const BinSort b) {
    extern __shared__ __align__(16) uint32_t s_cursor[];                       // [n_cursors]
    uint16_t* s_place = reinterpret_cast<uint16_t*>(s_cursor + b.n_cursors);   // [1 << bits]
    for (uint32_t i = threadIdx.x; i < b.n_cursors; i += SHARE_THREADS) s_cursor[i] = 0;
    grid_dependency_wait();
    if (b.ctl->overflow) return;
    for (uint32_t i = threadIdx.x; i < 1u << b.bits; i += SHARE_THREADS) s_place[i] = (uint16_t)b.bins[i];
    __syncthreads();
    uint32_t first, end;
    bin_share(item_count(b), first, end);
    const KeyRadix radix(b.ctl);
    const BinRange range(b, radix);
    bin_count_share(b, range, radix, first, end, s_cursor, [&](uint32_t bin) { return (uint32_t)s_place[bin]; });
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < b.n_cursors; i += SHARE_THREADS)
        if (s_cursor[i]) s_cursor[i] = atomicAdd(&b.cursors[i], s_cursor[i]);
    __syncthreads();
    const uint32_t span = (b.n_cursors + b.turns - 1) / b.turns;
    for (uint32_t turn = 0; turn < b.turns; ++turn) {
        for (uint32_t i0 = first + threadIdx.x; i0 < end; i0 += 4 * SHARE_THREADS) {
            ull w[4];
            uint32_t idx[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * SHARE_THREADS;
                w[u] = i < end ? b.words[i] : 0ull;
                idx[u] = b.ranking && i < end ? b.idx[i] : i;
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                if (i0 + u * SHARE_THREADS >= end) continue;
                if (!b.ranking) w[u] = radix.word(w[u]);
                const uint32_t to = s_place[range.bin(w[u])];
                if (to - turn * span >= span) continue;
                const uint32_t pos = atomicAdd(&s_cursor[to], 1u);
                b.items[pos] = range.item(w[u], idx[u]);
            }
        }
    }
}

// Order of two items: by their leading bits; equal ones by what those leave out.
__device__ __forceinline__ bool item_less(const atrex_entry_t* entries, bool ranking, ull x, ull y) {
    if ((x ^ y) >> 32) return x < y;
    const atrex_entry_t *a = entries + (uint32_t)x, *c = entries + (uint32_t)y;
    if (ranking) {
        if (a->wt_hi != c->wt_hi) return a->wt_hi > c->wt_hi;
        if (a->wt_lo != c->wt_lo) return a->wt_lo > c->wt_lo;
    }
    if (a->key != c->key) return a->key < c->key;
    return x < y;               // equal keys keep their input order
}

// Every comparator of this form of the bitonic network puts the smaller element at the lower position, so that
// positions at or beyond n can be left out (whole CTA).
template <typename Less, typename Swap>
__device__ __forceinline__ void bitonic(uint32_t n, Less less, Swap swap) {
    const int bits = n > 1 ? 32 - __clz((int)(n - 1)) : 0;
    for (int k = 1; k <= bits; ++k) {
        for (int j = k - 1; j >= 0; --j) {
            for (uint32_t t = threadIdx.x; t < 1u << (bits - 1); t += blockDim.x) {
                const uint32_t lo = (t >> j) << (j + 1) | (t & ((1u << j) - 1u)), in = (1u << k) - 1u;
                const uint32_t hi = j == k - 1 ? (lo | in) - (lo & in) : lo + (1u << j);
                if (hi < n && less(hi, lo)) swap(hi, lo);
            }
            __syncthreads();
        }
    }
}

// A crowded local bin, the n items at s_item[b0], in order (whole CTA).  They are cut into bins once more, between the
// smallest and the largest of what their leading bits left out -- the weighted times' 57 bits, or the keys where those are all
// alike --, bins that are still crowded again, and so on.  Items that nothing tells apart but their entries' order, and more than CROWD_MAX, go
// through the network, which reads entries at every comparison.  `s_bins`: CROWD_BINS + CROWD_MAX / 2 words.  (1.6 M rows, 1 600
// of them at the clamp of their weights: the tile that held those went through a network as a whole, kernel 90 us, now 80 with the weighted
// times written for the shares; 7.5 M rows, 7 500 of them: 572, now 367)
constexpr uint32_t CROWD_BINS = 2048, CROWD_MAX = 4096, CROWD_CLASH_MAX = 64, CROWD_SEGMENTS = 32;
__device__ __forceinline__ void sort_crowded_bin(const atrex_entry_t* entries, bool ranking, ull* s_item, uint32_t b0, uint32_t n, uint32_t* s_bins) {
    __shared__ ull s_range[2];
    __shared__ uint32_t s_warp[32], s_segments;
    __shared__ uint16_t s_from[CROWD_SEGMENTS], s_size[CROWD_SEGMENTS];
    uint16_t* s_list = reinterpret_cast<uint16_t*>(s_bins + CROWD_BINS);
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    auto by_network = [&](uint32_t from, uint32_t size) {
        bitonic(size, [&](uint32_t a, uint32_t b) { return item_less(entries, ranking, s_item[from + a], s_item[from + b]); },
                [&](uint32_t a, uint32_t b) { const ull x = s_item[from + a]; s_item[from + a] = s_item[from + b]; s_item[from + b] = x; });
    };
    __syncthreads();                 // (the local bins have been read, and the segments of the call before this one)
    if (threadIdx.x == 0) {
        s_segments = 1;
        s_from[0] = (uint16_t)b0;
        s_size[0] = (uint16_t)n;
    }
    __syncthreads();
    for (uint32_t k = 0; k < min(s_segments, CROWD_SEGMENTS); ++k) {       // (the same for every thread)
        const uint32_t from = s_from[k], size = s_size[k];
        ull* item = s_item + from;
        const atrex_entry_t* one = entries + (uint32_t)item[0];
        bool differ = false;
        for (uint32_t i = threadIdx.x; ranking && i < size; i += TILE_THREADS) {
            const atrex_entry_t* e = entries + (uint32_t)item[i];
            differ |= e->wt_lo != one->wt_lo || e->wt_hi != one->wt_hi;
        }
        const bool by_key = __syncthreads_or(differ) == 0;
        auto word = [&](uint32_t i) {
            const atrex_entry_t* e = entries + (uint32_t)item[i];
            return by_key ? e->key : rank_word(e->wt_lo, e->wt_hi);
        };
        if (threadIdx.x < 2) s_range[threadIdx.x] = 0;
        for (uint32_t i = threadIdx.x; i < CROWD_BINS; i += TILE_THREADS) s_bins[i] = 0;
        __syncthreads();
        ull top = 0, ntop = 0;
        for (uint32_t i = threadIdx.x; i < size; i += TILE_THREADS) {
            const ull x = word(i);
            top = max_ull(top, x);
            ntop = max_ull(ntop, ~x);
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            top = max_ull(top, __shfl_xor_sync(FULL, top, d));
            ntop = max_ull(ntop, __shfl_xor_sync(FULL, ntop, d));
        }
        if (lane == 0) {
            atomicMax(&s_range[0], top);
            atomicMax(&s_range[1], ntop);
        }
        __syncthreads();
        const ull low = ~s_range[1];
        if (s_range[0] == low || size > CROWD_MAX) {
            by_network(from, size);
            continue;
        }
        const int len = 64 - __clzll((long long)(s_range[0] - low)), shift = len > 11 ? len - 11 : 0;
        static_assert(CROWD_BINS == 1u << 11, "bits of a bin");
        auto bin_of = [&](uint32_t i) { return (uint32_t)((word(i) - low) >> shift); };
        for (uint32_t i = threadIdx.x; i < size; i += TILE_THREADS) atomicAdd(&s_bins[bin_of(i)], 1u);
        __syncthreads();
        constexpr uint32_t PER = CROWD_BINS / TILE_THREADS;
        uint32_t c[PER], sum = 0;
#pragma unroll
        for (uint32_t u = 0; u < PER; ++u) sum += c[u] = s_bins[threadIdx.x * PER + u];
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, incl, d);
            if (lane >= (uint32_t)d) incl += o;
        }
        if (lane == 31) s_warp[w] = incl;
        __syncthreads();
        uint32_t at = incl - sum;
        for (uint32_t j = 0; j < w; ++j) at += s_warp[j];
#pragma unroll
        for (uint32_t u = 0; u < PER; ++u) {
            s_bins[threadIdx.x * PER + u] = at;
            if (c[u] > CROWD_CLASH_MAX) {
                const uint32_t next = atomicAdd(&s_segments, 1u);
                if (next < CROWD_SEGMENTS) {
                    s_from[next] = (uint16_t)(from + at);
                    s_size[next] = (uint16_t)c[u];
                }
            }
            at += c[u];
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < size; i += TILE_THREADS) s_list[atomicAdd(&s_bins[bin_of(i)], 1u)] = (uint16_t)i;
        __syncthreads();
        // a bin's counter now stands at its end; every item's place in its bin, and all items there (they are held for a moment)
        ull held[CROWD_MAX / TILE_THREADS];
        uint32_t place[CROWD_MAX / TILE_THREADS];
#pragma unroll
        for (uint32_t u = 0; u < CROWD_MAX / TILE_THREADS; ++u) {
            const uint32_t at = u * TILE_THREADS + threadIdx.x;
            if (at >= size) continue;
            const uint32_t i = s_list[at], d = bin_of(i), begin = d ? s_bins[d - 1] : 0u, end = s_bins[d];
            held[u] = item[i];
            place[u] = at;                               // (in a bin that is still crowded: for now)
            if (end - begin <= CROWD_CLASH_MAX) {
                place[u] = begin;
                for (uint32_t j = begin; j < end; ++j) place[u] += j != at && item_less(entries, ranking, item[s_list[j]], held[u]) ? 1u : 0u;
            }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t u = 0; u < CROWD_MAX / TILE_THREADS; ++u)
            if (u * TILE_THREADS + threadIdx.x < size) item[place[u]] = held[u];
        __syncthreads();
    }
    if (s_segments > CROWD_SEGMENTS) by_network(b0, n);
}

// A crowded local bin of up to 64 items by one warp: every lane counts the items before its own two.
__device__ __forceinline__ void sort_small_bin(const atrex_entry_t* entries, bool ranking, ull* s_item, uint32_t n) {
    const uint32_t lane = threadIdx.x & 31u;
    ull item[2], hi[2], lo[2], key[2];
    uint32_t before[2] = {0, 0};
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u) {
        const bool in = u * 32 + lane < n;
        item[u] = in ? s_item[u * 32 + lane] : ~0ull;
        const atrex_entry_t* e = entries + (in ? (uint32_t)item[u] : 0u);
        hi[u] = in && ranking ? e->wt_hi : 0ull;
        lo[u] = in && ranking ? e->wt_lo : 0ull;
        key[u] = in ? e->key : 0ull;
    }
#pragma unroll
    for (uint32_t v = 0; v < 2; ++v) {
        for (uint32_t j = 0; j < 32 && v * 32 + j < n; ++j) {
            const ull y = __shfl_sync(FULL, item[v], j), y_hi = __shfl_sync(FULL, hi[v], j), y_lo = __shfl_sync(FULL, lo[v], j),
                      y_key = __shfl_sync(FULL, key[v], j);
#pragma unroll
            for (uint32_t u = 0; u < 2; ++u) {
                bool less = y < item[u];            // equal keys keep their input order
                if (!((y ^ item[u]) >> 32)) {
                    if (y_key != key[u]) less = y_key < key[u];
                    if (y_lo != lo[u]) less = y_lo > lo[u];
                    if (y_hi != hi[u]) less = y_hi > hi[u];
                }
                before[u] += less ? 1u : 0u;
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u)
        if (u * 32 + lane < n) s_item[before[u]] = item[u];
}

// Crowded local bins of up to TILE_SMALL_CROWD items, a warp each (the others go on).
__device__ __forceinline__ void sort_small_crowds(const atrex_entry_t* entries, bool ranking, ull* s_item, const uint32_t* s_local, const uint16_t* s_bin,
                                                  uint32_t crowded) {
    for (uint32_t k = threadIdx.x >> 5; k < crowded; k += TILE_THREADS / 32) {
        const uint32_t d = s_bin[k], b0 = d ? s_local[d - 1] : 0u, n = s_local[d] - b0;
        if (n <= TILE_SMALL_CROWD) sort_small_bin(entries, ranking, s_item + b0, n);
    }
}

// A tile's other crowded local bins, and those with ties: bit u of `tied` is a thread's bin u * TILE_THREADS + threadIdx.x (whole CTA, behind a
// barrier; the local bins are not needed any more).  A function of its own, as in place it costs every tile registers.
__device__ __noinline__ void sort_crowds(const atrex_entry_t* entries, bool ranking, ull* s_item, uint32_t* s_local, const uint16_t* s_bin, uint32_t crowded,
                                         uint32_t tied, bool any_tied) {
    constexpr uint32_t WARPS = TILE_THREADS / 32, WORDS = TILE_LOCAL_BINS / 32;
    static_assert(WARPS == 16 && WORDS == 4 * 32, "a word's bins go to two lots of sixteen warps, a lane looks at four words");
    __shared__ uint32_t s_tied[WORDS];                   // a bit for every local bin
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    uint32_t begin = 0, size = 0;                        // of the lane's crowded bin
    if (lane < crowded) {
        const uint32_t d = s_bin[lane];
        begin = d ? s_local[d - 1] : 0u;
        size = s_local[d] - begin;
    }
    if (any_tied) {
#pragma unroll
        for (uint32_t u = 0; u < TILE_LOCAL_BINS / TILE_THREADS; ++u) {
            const uint32_t votes = __ballot_sync(FULL, tied >> u & 1u);
            if (lane == 0) s_tied[u * WARPS + w] = votes;
        }
        __syncthreads();
        // bins next to one another go to different warps: groups of ties come side by side
#pragma unroll
        for (uint32_t v = 0; v < 4; ++v) {
            const uint32_t word = v * 32 + lane, own = s_tied[word] & 0x00010001u << ((w + word) & 15u);
            for (uint32_t todo = __ballot_sync(FULL, own != 0); todo; todo &= todo - 1) {
                const uint32_t src = __ffs(todo) - 1;
                for (uint32_t bits = __shfl_sync(FULL, own, src); bits; bits &= bits - 1) {
                    const uint32_t d = (v * 32 + src) * 32 + __ffs(bits) - 1, b0 = d ? s_local[d - 1] : 0u;
                    sort_small_bin(entries, ranking, s_item + b0, s_local[d] - b0);
                }
            }
        }
    }
    const uint32_t sorted = crowded > TILE_CROWDED_FEW ? TILE_SMALL_CROWD : 0u;
    for (uint32_t k = 0; k < crowded; ++k) {
        const uint32_t b0 = __shfl_sync(FULL, begin, k), n = __shfl_sync(FULL, size, k);
        if (n > sorted) sort_crowded_bin(entries, ranking, s_item, b0, n, s_local);
    }
}

// Sorts n <= TILE_CAP items whose leading bits lie in [low, high] into s_item.  `each(f)` calls f with each of
// this thread's items (twice).  Each item goes to one of as many local bins of equal width as a tile usually has items, or twice as many, so that
// a thread puts a bin in order by insertion; a few crowded local bins (hundreds of equal weights, say) are
// sorted on their own, those with ties by a warp each; many crowded ones send the whole tile through a bitonic network, with absent
// items behind the last one.
// (Every item's place counted by a thread of its own instead: 3.1 M entries 107.5 -> 111 us.)
template <uint32_t LOCAL_BINS, typename Each>
__device__ __forceinline__ void sort_tile(const atrex_entry_t* entries, bool ranking, uint32_t n, uint32_t low, uint32_t high, Each each, ull* s_item,
                                          uint32_t* s_local) {
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_crowded;
    __shared__ uint16_t s_bin[TILE_CROWDED];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int len = 32 - __clz((int)(high - low));
    constexpr int BITS = LOCAL_BINS == 4096 ? 12 : 10;
    static_assert(LOCAL_BINS == 1u << BITS, "bits of a local bin");
    const int shift = len > BITS ? len - BITS : 0;
    for (uint32_t i = threadIdx.x; i < LOCAL_BINS; i += blockDim.x) s_local[i] = 0;
    if (threadIdx.x == 0) s_crowded = 0;
    __syncthreads();
    each([&](ull item) {
        const uint32_t d = ((uint32_t)(item >> 32) - low) >> shift;
        if (atomicAdd(&s_local[d], 1u) == TILE_CLASH_MAX) {
            const uint32_t at = atomicAdd(&s_crowded, 1u);
            if (at < TILE_CROWDED) s_bin[at] = (uint16_t)d;
        }
    });
    __syncthreads();
    // exclusive scan of the local bins: each thread a run of them
    const uint32_t per = LOCAL_BINS / blockDim.x, first = threadIdx.x * per;
    uint32_t sum = 0;
    for (uint32_t u = 0; u < per; ++u) sum += s_local[first + u];
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(FULL, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        uint32_t v = lane < n_warps ? s_warp[lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, v, d);
            if (lane >= (uint32_t)d) v += o;
        }
        s_warp[lane] = v;
    }
    __syncthreads();
    uint32_t at = incl - sum + (w ? s_warp[w - 1] : 0u);
    for (uint32_t u = 0; u < per; ++u) {
        const uint32_t c = s_local[first + u];
        s_local[first + u] = at;
        at += c;
    }
    __syncthreads();
    each([&](ull item) { s_item[atomicAdd(&s_local[((uint32_t)(item >> 32) - low) >> shift], 1u)] = item; });
    __syncthreads();
    const uint32_t crowded = s_crowded;   // (nothing adds to it behind the first barrier)
    // (a bin's cursor now stands at its end, its predecessor's at its start)
    if (crowded <= TILE_CROWDED) {
        if (crowded > TILE_CROWDED_FEW) sort_small_crowds(entries, ranking, s_item, s_local, s_bin, crowded);   // (beside the insertion)
        uint32_t tied = 0;                               // (a thread has eight local bins at most)
        for (uint32_t d = threadIdx.x; d < LOCAL_BINS; d += TILE_THREADS) {
            const uint32_t b0 = d ? s_local[d - 1] : 0u, b1 = s_local[d];
            if (b1 - b0 > TILE_CLASH_MAX) continue;
            if (b1 - b0 >= TILE_TIES) {                  // leading bits alike: every comparison would read two entries
                uint32_t ties = 0;
                for (uint32_t i = b0 + 1; i < b1; ++i) ties += (s_item[i] ^ s_item[b0]) >> 32 ? 0u : 1u;
                if (ties >= TILE_TIES / 2) {
                    tied |= 1u << (d / TILE_THREADS);
                    continue;
                }
            }
            for (uint32_t i = b0 + 1; i < b1; ++i) {
                const ull item = s_item[i];
                uint32_t j = i;
                while (j > b0 && item_less(entries, ranking, item, s_item[j - 1])) {
                    s_item[j] = s_item[j - 1];
                    --j;
                }
                s_item[j] = item;
            }
        }
        const bool any_tied = __syncthreads_or(tied) != 0;
        if (any_tied || crowded != 0) sort_crowds(entries, ranking, s_item, s_local, s_bin, crowded, tied, any_tied);
    } else {
        bitonic(n, [&](uint32_t a, uint32_t b) { return item_less(entries, ranking, s_item[a], s_item[b]); },
                [&](uint32_t a, uint32_t b) { const ull x = s_item[a]; s_item[a] = s_item[b]; s_item[b] = x; });
    }
    __syncthreads();
}

// Entries of the sorted items to out[first .. first + n), as far as out_cap: three lanes to an entry, so that
// the stores are contiguous and an entry's read is three 16-byte pieces of one or two lines (8-byte pieces
// where a caller's buffer is only 8-byte aligned).
// (each(row, lo, hi): the weighted time of a row)
template <typename Weight>
__device__ __forceinline__ void gather_tile(const atrex_entry_t* entries, const ull* s_item, uint32_t n, atrex_entry_t* out, uint32_t first,
                                            uint32_t out_cap, Weight each) {
    const uint32_t rows = first < out_cap ? min(n, out_cap - first) : 0u;
    if ((((uintptr_t)entries | (uintptr_t)out) & 15u) == 0) {
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>(entries);
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(out + first);
        for (uint32_t i = threadIdx.x; i < rows * 3; i += GATHER_LOADS * blockDim.x) {
            ulonglong2 v[GATHER_LOADS];
#pragma unroll
            for (uint32_t u = 0; u < GATHER_LOADS; ++u) {
                const uint32_t x = i + u * blockDim.x;
                if (x < rows * 3) v[u] = __ldg(src + (size_t)(uint32_t)s_item[x / 3] * 3 + x % 3);
            }
#pragma unroll
            for (uint32_t u = 0; u < GATHER_LOADS; ++u)
            {
                const uint32_t x = i + u * blockDim.x;
                if (x >= rows * 3) continue;
                __stcs(dst + x, v[u]);
                if (x % 3 == 1) each(x / 3, v[u].x, v[u].y);
            }
        }
    } else {
        const ull* src = reinterpret_cast<const ull*>(entries);
        ull* dst = reinterpret_cast<ull*>(out + first);
        for (uint32_t i = threadIdx.x; i < rows * 6; i += blockDim.x) {
            const size_t at = (size_t)(uint32_t)s_item[i / 6] * 6 + i % 6;
            const ull v = src[at];
            dst[i] = v;
            if (i % 6 == 2) each(i / 6, v, src[at + 1]);
        }
    }
}

// 5. a tile's items in order, their entries gathered; (ranking) the weighted times of the rows and their sum.  A kernel per order: in one for
//    both, what only the other needs costs the key order 2 % and more (15 M entries: tile kernel 565 us, now 548).
template <uint32_t LOCAL_BINS, bool RANKING>
__global__ void __launch_bounds__(TILE_THREADS) bin_tile_kernel(const BinSort b, atrex_entry_t* out, uint32_t out_cap) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ull* s_item = reinterpret_cast<ull*>(smem_raw);
    uint32_t* s_local = reinterpret_cast<uint32_t*>(s_item + TILE_CAP);
    __shared__ ull s_sum[2];
    __shared__ uint32_t s_range[2];
    grid_dependency_wait();
    const bool overflow = b.ctl->overflow;
    // the last tile first: at both ends of a ranking the words lie uneven, which takes a tile twice as long
    const uint32_t n_tiles = tiles_of(b, RANKING ? (uint32_t)b.ctl->counter : b.n);
    const uint32_t tile = blockIdx.x >= n_tiles ? blockIdx.x : (blockIdx.x ? blockIdx.x - 1 : n_tiles - 1);
    const uint32_t first = overflow ? 0u : b.tile_start[tile], n = overflow ? 0u : b.tile_start[tile + 1] - first;
    if (n == 0) {
        if (!RANKING) finish_call(b.report, b.slot);
        else if (!overflow && threadIdx.x == 0) b.tile_sum[tile] = make_ulonglong2(0, 0);
        return;
    }
    // the items are read once, all of a thread's at a time (a tile rarely has more than TILE_HELD per thread)
    ull held[TILE_HELD];
#pragma unroll
    for (uint32_t u = 0; u < TILE_HELD; ++u) {
        const uint32_t i = u * TILE_THREADS + threadIdx.x;
        held[u] = i < n ? __ldcs(b.items + first + i) : 0ull;
    }
    auto each = [&](auto f) {
#pragma unroll
        for (uint32_t u = 0; u < TILE_HELD; ++u)
            if (u * TILE_THREADS + threadIdx.x < n) f(held[u]);
        for (uint32_t i = TILE_HELD * TILE_THREADS + threadIdx.x; i < n; i += TILE_THREADS) f(b.items[first + i]);
    };
    uint32_t top = 0, ntop = 0;
    each([&](ull item) {
        const uint32_t w = (uint32_t)(item >> 32);
        top = max(top, w);
        ntop = max(ntop, ~w);
    });
    if (threadIdx.x == 0) s_range[0] = s_range[1] = 0;
    __syncthreads();
    top = __reduce_max_sync(FULL, top);
    ntop = __reduce_max_sync(FULL, ntop);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_range[0], ntop);
        atomicMax(&s_range[1], top);
    }
    __syncthreads();
    sort_tile<LOCAL_BINS>(b.entries, RANKING, n, ~s_range[0], s_range[1], each, s_item, s_local);
    grid_dependents_launch();
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0;
    ulonglong2 sum = make_ulonglong2(0, 0);
    if constexpr (!RANKING) {
        gather_tile(b.entries, s_item, n, out, first, out_cap, [](uint32_t, ull, ull) {});
        finish_call(b.report, b.slot);
        return;
    }
    // (the shares read a row's weighted time from where the words and indices were: the ranked rows themselves would have to come from
    // memory once more)
    auto weight = [&](uint32_t row, ull lo, ull hi) {
        add128(sum.x, sum.y, lo, hi);
        b.ranked_wt[first + row] = make_ulonglong2(lo, hi);
    };
    gather_tile(b.entries, s_item, n, out, first, out_cap, weight);
    for (uint32_t i = threadIdx.x; i < n; i += TILE_THREADS) {   // rows that are not wanted
        if (first + i < out_cap) continue;
        const atrex_entry_t* e = b.entries + (uint32_t)s_item[i];
        weight(i, e->wt_lo, e->wt_hi);
    }
    __syncthreads();   // s_sum is cleared
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const ull olo = __shfl_xor_sync(FULL, sum.x, d), ohi = __shfl_xor_sync(FULL, sum.y, d);
        add128(sum.x, sum.y, olo, ohi);
    }
    if ((threadIdx.x & 31) == 0 && (sum.x | sum.y)) atomic_add128(&s_sum[0], &s_sum[1], sum.x, sum.y);
    __syncthreads();
    if (threadIdx.x == 0) {
        b.tile_sum[tile] = make_ulonglong2(s_sum[0], s_sum[1]);
        ull* group = reinterpret_cast<ull*>(b.group_sum + tile / TILE_GROUP);
        atomic_add128(group, group + 1, s_sum[0], s_sum[1]);
    }
}

// 6. (ranking) running share of each row, and the row at the coverage cut.  A CTA takes a run of tiles and adds up for itself what lies
//    before it, group by group and then tile by tile (a scan of the tiles in a launch of its own took 11 us).  A thread takes four rows
//    one behind the other, so that one scan over the warp serves 128 of them; the shares go out through shared memory, side by side.
//    Bound by latency and instructions (a row's share is sixty): with the scan of the tiles, 1.6 M rows 46 us while a lane took
//    a row, every 1 024 rows three barriers, and the ranked rows were read back; now 26 behind the tiles.  7.5 M rows 155, now 88.
constexpr uint32_t CUM_THREADS = 512, CUM_ROWS = 4, CUM_CTAS = 2;
__global__ void __launch_bounds__(CUM_THREADS, CUM_CTAS) bin_share_kernel(const BinSort b, double* cum, uint32_t out_cap) {
    __shared__ ulonglong2 s_part[CUM_THREADS / 32];
    __shared__ double s_cum[CUM_THREADS * CUM_ROWS];
    grid_dependency_wait();
    const ull total_lo = b.ctl->total_lo, total_hi = b.ctl->total_hi, need_lo = b.ctl->need_lo, need_hi = b.ctl->need_hi, overflow = b.ctl->overflow;
    const uint32_t n_tiles = tiles_of(b, item_count(b)), run = (n_tiles + gridDim.x - 1) / gridDim.x;
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, tile = min(n_tiles, blockIdx.x * run), group = tile / TILE_GROUP;
    if (overflow) {
        finish_call(b.report, b.slot);
        return;
    }
    const uint32_t first = b.tile_start[tile], end = b.tile_start[min(n_tiles, tile + run)];
    const double total = u128_to_f64_rn(total_hi, total_lo);
    // sums of the warps (in each one's last lane): of those before this one, and of all
    auto all_warps = [&](ull lo, ull hi, ull& before_lo, ull& before_hi, ull& all_lo, ull& all_hi) {
        if (lane == 31) s_part[w] = make_ulonglong2(lo, hi);
        __syncthreads();
        const ulonglong2 v = lane < CUM_THREADS / 32 ? s_part[lane] : make_ulonglong2(0, 0);
        before_lo = lane < w ? v.x : 0ull, before_hi = lane < w ? v.y : 0ull, all_lo = v.x, all_hi = v.y;
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const ull olo = __shfl_xor_sync(FULL, before_lo, d), ohi = __shfl_xor_sync(FULL, before_hi, d);
            add128(before_lo, before_hi, olo, ohi);
            const ull alo = __shfl_xor_sync(FULL, all_lo, d), ahi = __shfl_xor_sync(FULL, all_hi, d);
            add128(all_lo, all_hi, alo, ahi);
        }
    };
    ull run_lo = 0, run_hi = 0;
    if (first < end) {
        ull lo = 0, hi = 0, unused_lo, unused_hi;
        for (uint32_t g = threadIdx.x; g < group; g += CUM_THREADS) add128(lo, hi, b.group_sum[g].x, b.group_sum[g].y);
        for (uint32_t t = group * TILE_GROUP + threadIdx.x; t < tile; t += CUM_THREADS) add128(lo, hi, b.tile_sum[t].x, b.tile_sum[t].y);
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const ull olo = __shfl_xor_sync(FULL, lo, d), ohi = __shfl_xor_sync(FULL, hi, d);
            add128(lo, hi, olo, ohi);
        }
        all_warps(lo, hi, unused_lo, unused_hi, run_lo, run_hi);
        __syncthreads();
    }
    for (uint32_t base = first; base < end; base += CUM_ROWS * CUM_THREADS) {
        const uint32_t r0 = base + threadIdx.x * CUM_ROWS;
        ull lo[CUM_ROWS], hi[CUM_ROWS];
#pragma unroll
        for (uint32_t u = 0; u < CUM_ROWS; ++u) {
            lo[u] = hi[u] = 0;
            if (r0 + u < end) {
                const ulonglong2 wt = b.ranked_wt[r0 + u];
                lo[u] = wt.x;
                hi[u] = wt.y;
            }
        }
        ull own_lo = 0, own_hi = 0;
#pragma unroll
        for (uint32_t u = 0; u < CUM_ROWS; ++u) add128(own_lo, own_hi, lo[u], hi[u]);
        ull at_lo = own_lo, at_hi = own_hi;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const ull olo = __shfl_up_sync(FULL, at_lo, d), ohi = __shfl_up_sync(FULL, at_hi, d);
            if (lane >= (uint32_t)d) add128(at_lo, at_hi, olo, ohi);
        }
        ull before_lo, before_hi, all_lo, all_hi;
        all_warps(at_lo, at_hi, before_lo, before_hi, all_lo, all_hi);
        add128(at_lo, at_hi, before_lo, before_hi);
        add128(at_lo, at_hi, run_lo, run_hi);                    // up to and with this thread's rows
        const bool reaches = (need_lo | need_hi) && !less128(at_lo, at_hi, need_lo, need_hi);
        at_hi -= own_hi + (at_lo < own_lo ? 1ull : 0ull);        // up to them
        at_lo -= own_lo;
        const bool cut_here = reaches && less128(at_lo, at_hi, need_lo, need_hi);
        add128(run_lo, run_hi, all_lo, all_hi);
#pragma unroll
        for (uint32_t u = 0; u < CUM_ROWS; ++u) {
            const ull ex_lo = at_lo, ex_hi = at_hi;
            add128(at_lo, at_hi, lo[u], hi[u]);                  // inclusive prefix of the whole list
            if (cut_here && r0 + u < end && less128(ex_lo, ex_hi, need_lo, need_hi) && !less128(at_lo, at_hi, need_lo, need_hi)) {
                b.report->n_keep = (ull)r0 + u + 1;
                b.report->covered_lo = at_lo;
                b.report->covered_hi = at_hi;
                __threadfence_system();
            }
            s_cum[threadIdx.x * CUM_ROWS + u] = (total_lo | total_hi) ? __ddiv_rn(u128_to_f64_rn(at_hi, at_lo), total) : 0.0;
        }
        __syncthreads();                                         // (s_part may be written again, too)
        const uint32_t rows = min(end, out_cap) > base ? min(min(end, out_cap) - base, CUM_ROWS * CUM_THREADS) : 0u;
        for (uint32_t i = threadIdx.x; i < rows; i += CUM_THREADS) cum[base + i] = s_cum[i];
        __syncthreads();
    }
    finish_call(b.report, b.slot);
}

// Key order of up to COUNT_SORT_MAX entries in one kernel: an entry's place is the number of keys before its own.
// Every CTA reads all keys (32 bytes of L2 each: 1 us of an SM's bandwidth for 4 096) and places 32 U entries, a
// lane each (U of them), every warp counting over its own sixteenth of the keys.  Bound by latency: 4 096 entries
// in 9 us (sorted by one CTA in shared memory: 16), the call 15 us, 8 000 entries 24 (binned sort: 37).  (Keys read
// once per cluster of eight and handed round through distributed shared memory: slower, 4 096 remote stores into
// each SM take 10 us.)
constexpr uint32_t COUNT_THREADS = 512, COUNT_LOADS = 8;
template <uint32_t U>
__global__ void __launch_bounds__(COUNT_THREADS) count_sort_kernel(const atrex_entry_t* entries, uint32_t n, atrex_entry_t* out, BinReport* report, uint32_t slot) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ull* s_key = reinterpret_cast<ull*>(smem_raw);   // [n, rounded up to an even number]
    __shared__ uint32_t s_place[32 * U];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, base = blockIdx.x * 32 * U;
    for (uint32_t i = threadIdx.x; i < 32 * U; i += COUNT_THREADS) s_place[i] = 0;
    grid_dependency_wait();
    for (uint32_t i0 = threadIdx.x; i0 < n; i0 += COUNT_LOADS * COUNT_THREADS) {
        ull key[COUNT_LOADS];
#pragma unroll
        for (uint32_t u = 0; u < COUNT_LOADS; ++u) key[u] = i0 + u * COUNT_THREADS < n ? entries[i0 + u * COUNT_THREADS].key : 0ull;
#pragma unroll
        for (uint32_t u = 0; u < COUNT_LOADS; ++u)
            if (i0 + u * COUNT_THREADS < n) s_key[i0 + u * COUNT_THREADS] = key[u];
    }
    if (threadIdx.x == 0 && (n & 1u)) s_key[n] = ~0ull;   // (before nothing)
    grid_dependents_launch();
    __syncthreads();
    ull mine[U];
    uint32_t before[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
        mine[u] = base + u * 32 + lane < n ? s_key[base + u * 32 + lane] : 0ull;
        before[u] = 0;
    }
    // equal keys keep their input order: those at lower positions count too
    const uint32_t per = ((n + COUNT_THREADS / 32 - 1) / (COUNT_THREADS / 32) + 1) & ~1u, first = min((n + 1) & ~1u, w * per), end = min((n + 1) & ~1u, first + per);
    const uint32_t own = min(max(base, first), end), behind = min(max(base + 32 * U, first), end);   // (all of these are even)
    const ulonglong2* pair = reinterpret_cast<const ulonglong2*>(s_key);
#pragma unroll 8
    for (uint32_t i = first / 2; i < own / 2; ++i) {
        const ulonglong2 key = pair[i];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) before[u] += (key.x <= mine[u] ? 1u : 0u) + (key.y <= mine[u] ? 1u : 0u);
    }
    for (uint32_t i = own; i < behind; ++i) {
        const ull key = s_key[i];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) before[u] += key < mine[u] || (key == mine[u] && i < base + u * 32 + lane) ? 1u : 0u;
    }
#pragma unroll 8
    for (uint32_t i = behind / 2; i < end / 2; ++i) {
        const ulonglong2 key = pair[i];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) before[u] += (key.x < mine[u] ? 1u : 0u) + (key.y < mine[u] ? 1u : 0u);
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u)
        if (before[u]) atomicAdd(&s_place[u * 32 + lane], before[u]);
    __syncthreads();
    const ull* src = reinterpret_cast<const ull*>(entries + base);
    ull* dst = reinterpret_cast<ull*>(out);
    for (uint32_t x = threadIdx.x; x < min(32 * U, n - base) * 6; x += COUNT_THREADS) dst[(size_t)s_place[x / 6] * 6 + x % 6] = src[x];
    finish_call(report, slot);
}

// A phase of a list of up to COUNT_RANK_MAX entries ranked in one kernel: an entry's place is the number of the phase's entries before
// it, and the running sum before it the sum of theirs.  Every CTA reads all entries, puts the phase's side by side and places 32 of
// them, a lane each, every warp counting over its own sixteenth.  Bound by the comparisons, some twenty instructions each (whole call,
// one phase of two, in seven launches before: 100 entries 41 -> 18 us, 2 000 45 -> 23, 4 096 51 -> 30; all of one phase 4 096 52 -> 43.  Twice as
// many entries are twice the CTAs and twice the comparisons of each: no gain in one phase).
constexpr uint32_t COUNT_RANK_MAX = 4096;
__global__ void __launch_bounds__(COUNT_THREADS) count_rank_kernel(const atrex_entry_t* entries, uint32_t n, uint32_t phase, uint32_t coverage_ppm,
                                                                   atrex_entry_t* out, double* cum, uint32_t out_cap, BinReport* report, uint32_t slot) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ulonglong2* s_wt = reinterpret_cast<ulonglong2*>(smem_raw);        // [n] the phase's entries in input order
    ull* s_key = reinterpret_cast<ull*>(s_wt + n);
    uint16_t* s_at = reinterpret_cast<uint16_t*>(s_key + n);
    constexpr uint32_t WARPS = COUNT_THREADS / 32, EACH = COUNT_RANK_MAX / COUNT_THREADS, WORDS = COUNT_RANK_MAX / 32;
    __shared__ ulonglong2 s_sum[WARPS][32];
    __shared__ uint32_t s_count[WARPS][32], s_place[32], s_start[WORDS], s_counted;
    __shared__ ull s_total[2];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, base = blockIdx.x * 32;
    if (threadIdx.x < 2) s_total[threadIdx.x] = 0;
    grid_dependency_wait();
    ull key[EACH], lo[EACH], hi[EACH], total_lo = 0, total_hi = 0;
#pragma unroll
    for (uint32_t u = 0; u < EACH; ++u) {
        const uint32_t i = u * COUNT_THREADS + threadIdx.x;
        key[u] = i < n ? entries[i].key : ~0ull;
        lo[u] = i < n ? entries[i].wt_lo : 0ull;
        hi[u] = i < n ? entries[i].wt_hi : 0ull;
    }
    grid_dependents_launch();
    uint32_t votes[EACH];
#pragma unroll
    for (uint32_t u = 0; u < EACH; ++u) {
        const bool mine = (uint32_t)(key[u] >> 48) == phase;
        votes[u] = __ballot_sync(FULL, mine);
        if (lane == 0) s_start[u * WARPS + w] = __popc(votes[u]);
        if (mine) add128(total_lo, total_hi, lo[u], hi[u]);
    }
    __syncthreads();
    if (w == 0) {                                        // where each word's entries start
        static_assert(WORDS == 128, "four words a lane");
        uint32_t c[4], own = 0;
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) own += c[j] = s_start[lane * 4 + j];
        uint32_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, incl, d);
            if (lane >= (uint32_t)d) incl += o;
        }
        uint32_t at = incl - own;
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            s_start[lane * 4 + j] = at;
            at += c[j];
        }
        if (lane == 31) s_counted = incl;
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const ull olo = __shfl_xor_sync(FULL, total_lo, d), ohi = __shfl_xor_sync(FULL, total_hi, d);
        add128(total_lo, total_hi, olo, ohi);
    }
    if (lane == 0 && (total_lo | total_hi)) atomic_add128(&s_total[0], &s_total[1], total_lo, total_hi);
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < EACH; ++u) {
        if ((votes[u] & (1u << lane)) == 0) continue;
        const uint32_t at = s_start[u * WARPS + w] + __popc(votes[u] & ((1u << lane) - 1u));
        s_wt[at] = make_ulonglong2(lo[u], hi[u]);
        s_key[at] = key[u];
        s_at[at] = (uint16_t)(u * COUNT_THREADS + threadIdx.x);
    }
    __syncthreads();
    const uint32_t m = s_counted, own = base + lane;
    const ulonglong2 mine = own < m ? s_wt[own] : make_ulonglong2(0, 0);
    const ull my_key = own < m ? s_key[own] : 0ull, my_lo = mine.x, my_hi = mine.y;
    const uint32_t per = (m + WARPS - 1) / WARPS, first = base < m ? min(m, w * per) : m, end = min(m, first + per);
    uint32_t before = 0;
    ull sum_lo = 0, sum_hi = 0;
#pragma unroll 4
    for (uint32_t j = first; j < end; ++j) {
        const ulonglong2 x = s_wt[j];
        bool less = x.y > my_hi || (x.y == my_hi && x.x > my_lo);
        if (x.x == my_lo && x.y == my_hi) less = s_key[j] < my_key || (s_key[j] == my_key && j < own);    // equal keys keep their input order
        before += less ? 1u : 0u;
        add128(sum_lo, sum_hi, less ? x.x : 0ull, less ? x.y : 0ull);
    }
    s_count[w][lane] = before;
    s_sum[w][lane] = make_ulonglong2(sum_lo, sum_hi);
    __syncthreads();
    total_lo = s_total[0];
    total_hi = s_total[1];
    const bool too_large = (total_hi >> 44) != 0;        // T * 10^6 must fit 128 bits
    if (w == 0) {
        uint32_t place = 0;
        ull ex_lo = 0, ex_hi = 0;
#pragma unroll
        for (uint32_t k = 0; k < WARPS; ++k) {
            place += s_count[k][lane];
            add128(ex_lo, ex_hi, s_sum[k][lane].x, s_sum[k][lane].y);
        }
        const bool ranked = own < m && !too_large;
        s_place[lane] = ranked && place < out_cap ? place : ~0u;
        if (ranked) {
            // the smallest k with 10^6 * prefix_k >= ppm * T, i.e. prefix_k >= ceil(ppm * T / 10^6)
            const unsigned __int128 total = ((unsigned __int128)total_hi << 64) | total_lo;
            const unsigned __int128 need = ((unsigned __int128)coverage_ppm * total + 999999u) / 1000000u;
            const unsigned __int128 ex = ((unsigned __int128)ex_hi << 64) | ex_lo, in = ex + (((unsigned __int128)my_hi << 64) | my_lo);
            if (need != 0 && ex < need && in >= need) {
                report->n_keep = (ull)place + 1;
                report->covered_lo = (ull)in;
                report->covered_hi = (ull)(in >> 64);
                __threadfence_system();
            }
            if (place < out_cap) cum[place] = total != 0 ? __ddiv_rn(u128_to_f64_rn((ull)(in >> 64), (ull)in), u128_to_f64_rn(total_hi, total_lo)) : 0.0;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 32) {
        report->counter = s_counted;
        report->total_lo = total_lo;
        report->total_hi = total_hi;
        report->too_large = too_large;
        __threadfence_system();
    }
    __syncthreads();
    const ull* src = reinterpret_cast<const ull*>(entries);
    ull* dst = reinterpret_cast<ull*>(out);
    for (uint32_t x = threadIdx.x; x < 32 * 6; x += COUNT_THREADS)
        if (s_place[x / 6] != ~0u) dst[(size_t)s_place[x / 6] * 6 + x % 6] = src[(size_t)s_at[base + x / 6] * 6 + x % 6];
    finish_call(report, slot);
}

// ---- host side

struct Scratch {
    ReleaseCtl* ctl;
    ull* words[2];
    uint32_t* idx[2];
    uint32_t* hist;
    uint32_t* bin_total;
    ull* bsums;
};

constexpr uint64_t align256(uint64_t x) { return (x + 255u) & ~(uint64_t)255u; }

constexpr uint64_t scratch_bytes_for(uint64_t n) {
    const uint64_t tiles = (n + SORT_TILE - 1) / SORT_TILE, blocks = (n + SCAN_BLOCK - 1) / SCAN_BLOCK;
    return sizeof(ReleaseCtl) + 2 * align256(n * 8) + 2 * align256(n * 4) + align256(tiles * 256 * 4) +
           1024 + align256(blocks * 16) + 256;
}

Scratch carve(void* base, uint64_t n) {
    const uint64_t tiles = (n + SORT_TILE - 1) / SORT_TILE;
    unsigned char* p = (unsigned char*)base;
    Scratch s;
    s.ctl = (ReleaseCtl*)p;
    p += sizeof(ReleaseCtl);
    for (int b = 0; b < 2; ++b) {
        s.words[b] = (ull*)p;
        p += align256(n * 8);
    }
    for (int b = 0; b < 2; ++b) {
        s.idx[b] = (uint32_t*)p;
        p += align256(n * 4);
    }
    s.hist = (uint32_t*)p;
    p += align256(tiles * 256 * 4);
    s.bin_total = (uint32_t*)p;
    p += 1024;
    s.bsums = (ull*)p;
    return s;
}

int grid_for(uint64_t n, int block) {
    uint64_t g = (n + block - 1) / block;
    return (int)(g < 1 ? 1 : (g > 148 * 8 ? 148 * 8 : g));
}

// Reads back the control block (synchronises the stream).
int read_ctl(const Scratch& sc, ReleaseCtl* host, cudaStream_t s) {
    if (cudaMemcpyAsync(host, sc.ctl, sizeof(ReleaseCtl), cudaMemcpyDeviceToHost, s) != cudaSuccess) return ATREX_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? ATREX_OK : ATREX_ERR_CUDA;
}

int reset_or_and(const Scratch& sc, cudaStream_t s) {
    const ull init[2] = {0ull, ~0ull};
    return cudaMemcpyAsync(&sc.ctl->word_or, init, sizeof(init), cudaMemcpyHostToDevice, s) == cudaSuccess ? ATREX_OK
                                                                                                             : ATREX_ERR_CUDA;
}

// Kernels that keep a whole tile in shared memory: their dynamic shared-memory limit is raised once per
// device (the caller has made the entries' device current).
int prepare_sort_kernels(int* n_sms) {
    static std::mutex lock;
    static int prepared[64];   // the device's SM count, once done
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ATREX_ERR_CUDA;
    std::lock_guard<std::mutex> hold(lock);
    if (prepared[dev] == 0) {
        int v = 0;
        if (cudaFuncSetAttribute(radix_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCATTER_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(bin_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 << BIN_BITS_MAX) != cudaSuccess ||
            cudaFuncSetAttribute(bin_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(4 * CURSORS_MAX + (2 << BIN_BITS_MAX))) != cudaSuccess ||
            cudaFuncSetAttribute(bin_tile_kernel<TILE_LOCAL_BINS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(bin_tile_kernel<TILE_LOCAL_BINS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(bin_tile_kernel<SMALL_LOCAL_BINS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(bin_tile_kernel<SMALL_LOCAL_BINS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(count_rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(COUNT_RANK_MAX * 26)) != cudaSuccess ||
            cudaFuncSetAttribute(count_sort_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(COUNT_SORT_MAX * 8)) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return ATREX_ERR_CUDA;
        }
        prepared[dev] = v;
    }
    *n_sms = prepared[dev];
    return ATREX_OK;
}

// Sorts the m pairs in buffer `cur` by the digits of the word on which the words differ.
// Returns the buffer that holds the result, or a negative status.
int sort_by_word(const Scratch& sc, int cur, uint32_t m, ull differing_bits, cudaStream_t s) {
    const uint32_t tiles = (m + SORT_TILE - 1) / SORT_TILE;
    for (int shift = 0; shift < 64; shift += 8) {
        if (((differing_bits >> shift) & 255u) == 0) continue;
        radix_hist_kernel<<<tiles, SORT_WARPS * 32, 0, s>>>(sc.words[cur], m, shift, sc.hist, tiles);
        radix_scan_kernel<<<256, SCAN_BLOCK, 0, s>>>(sc.hist, tiles, sc.bin_total);
        radix_scatter_kernel<<<tiles, SORT_WARPS * 32, SCATTER_SMEM, s>>>(sc.words[cur], sc.idx[cur], sc.words[cur ^ 1],
                                                                sc.idx[cur ^ 1], m, shift, sc.hist, tiles,
                                                                sc.bin_total);
        if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
        cur ^= 1;
    }
    return cur;
}

// How many tiles, bins and cursors a list of n entries gets, and the bytes that these take in front of the items.
struct BinSizes {
    uint32_t log_step, bits, n_cursors;
    bool by_tile;
    uint64_t tiles, group_bytes, bin_bytes, cursor_bytes;
    constexpr BinSizes(uint64_t n, bool ranking)
        : log_step(n <= SMALL_LIST_MAX ? SMALL_LOG_STEP : ranking && n <= MIDDLE_RANKING_MAX ? MIDDLE_LOG_STEP : TILE_LOG_STEP), bits(4), n_cursors(0), by_tile(false),
          tiles((n + (1ull << log_step) - 1) >> log_step), group_bytes(ranking ? (tiles + TILE_GROUP - 1) / TILE_GROUP * 16 : 0), bin_bytes(0), cursor_bytes(0) {
        // about 256 items per bin, a thousand beyond 2^12 bins (more open ranges than that cost the scattered writes), 64 or
        // 128 for small tiles
        while (bits < BIN_BITS_MAX && ((log_step < TILE_LOG_STEP ? (n <= 65536 ? 64ull : 128ull) : bits < 12 ? 256ull : 1024ull) << bits) < n) ++bits;
        by_tile = tiles <= CURSORS_MAX;
        n_cursors = by_tile ? (uint32_t)tiles : 1u << bits;
        bin_bytes = 4ull << bits;
        cursor_bytes = 4ull * ((n_cursors + 3) & ~3u);
    }
    constexpr uint64_t control_bytes() const { return align256(sizeof(BinCtl) + group_bytes + bin_bytes + cursor_bytes + tiles * 16 + (tiles + 1) * 4); }
    // items, words, and room for the ranked weighted times
    constexpr uint64_t bytes(uint64_t n) const { return control_bytes() + 2 * align256(n * 8) + n * 8; }
};
// (the scratch's size is the radix sort's, whose digit counts take more than the control area: on both sides of every line above)
constexpr bool bins_fit(uint64_t n) { return BinSizes(n, false).bytes(n) <= scratch_bytes_for(n) && BinSizes(n, true).bytes(n) <= scratch_bytes_for(n); }
static_assert(bins_fit(1) && bins_fit(COUNT_RANK_MAX + 1) && bins_fit(COUNT_SORT_MAX + 1) && bins_fit(65536) && bins_fit(65537) && bins_fit(SMALL_LIST_MAX) &&
                  bins_fit(SMALL_LIST_MAX + 1) && bins_fit(MIDDLE_RANKING_MAX) && bins_fit(MIDDLE_RANKING_MAX + 1) && bins_fit(1u << 20) && bins_fit((1u << 20) + 1) &&
                  bins_fit(1u << 22) && bins_fit((1u << 22) + 1) && bins_fit((uint64_t)CURSORS_MAX << TILE_LOG_STEP) &&
                  bins_fit(((uint64_t)CURSORS_MAX << TILE_LOG_STEP) + 1) && bins_fit(ATREX_RELEASE_MAX_ENTRIES), "the binned sort's use of the scratch");

// The scratch as the binned sort uses it.
BinSort carve_bins(void* base, const atrex_entry_t* entries, uint64_t n, bool ranking, const ReportSlot& slot) {
    unsigned char* p = (unsigned char*)base;
    BinSort b;
    const BinSizes z(n, ranking);
    b.log_step = z.log_step;
    b.bits = z.bits;
    b.n_cursors = z.n_cursors;
    b.by_tile = z.by_tile;
    b.turns = b.n_cursors >= 2048 ? 2 : 1;
    b.ctl = (BinCtl*)p;
    b.report = slot.get();
    b.slot = slot.number();
    b.entries = entries;
    b.n = (uint32_t)n;
    b.ranking = ranking;
    p += sizeof(BinCtl);
    b.group_sum = (ulonglong2*)p; p += z.group_bytes;
    b.bins = (uint32_t*)p;       p += z.bin_bytes;
    b.cursors = (uint32_t*)p;    p += z.cursor_bytes;
    b.tile_sum = (ulonglong2*)p; p += z.tiles * 16;
    b.tile_start = (uint32_t*)p;
    p = (unsigned char*)base + z.control_bytes();
    b.words = (ull*)p;           p += align256(n * 8);
    b.idx = (uint32_t*)p;        p += align256(n * 8);
    b.items = (ull*)p;
    b.ranked_wt = (ulonglong2*)b.words;
    return b;
}

cudaError_t launch_clear(const BinSort& b, cudaStream_t s) {
    const BinSizes z(b.n, b.ranking);
    const uint32_t n = (uint32_t)((sizeof(BinCtl) + z.group_bytes + z.bin_bytes) / 16);
    return launch_chained(bin_clear_kernel, (n + BIN_THREADS - 1) / BIN_THREADS, BIN_THREADS, 0, s, (uint4*)b.ctl, n);
}

// Steps 2 to 5, behind the kernel that made the words.
cudaError_t launch_bins(const BinSort& b, uint32_t coverage_ppm, atrex_entry_t* out, uint64_t out_cap, int n_sms, cudaStream_t s) {
    const uint32_t bytes = 4u << b.bits, tiles = tiles_of(b, b.n);
    uint32_t grid = (b.n + 4095) / 4096;
    if (grid > (uint32_t)n_sms) grid = (uint32_t)n_sms;
    cudaError_t e = launch_chained(bin_count_kernel, grid, SHARE_THREADS, bytes, s, b);
    if (e == cudaSuccess) e = launch_chained(bin_scan_kernel, 1, 1024, 0, s, b, coverage_ppm);
    if (e == cudaSuccess) e = launch_chained(bin_scatter_kernel, grid, SHARE_THREADS, b.n_cursors * 4 + (2u << b.bits), s, b);
    auto* tile = b.log_step < TILE_LOG_STEP ? (b.ranking ? bin_tile_kernel<SMALL_LOCAL_BINS, true> : bin_tile_kernel<SMALL_LOCAL_BINS, false>)
                                              : (b.ranking ? bin_tile_kernel<TILE_LOCAL_BINS, true> : bin_tile_kernel<TILE_LOCAL_BINS, false>);
    if (e == cudaSuccess) e = launch_chained(tile, tiles, TILE_THREADS, TILE_SMEM, s, b, out, (uint32_t)(out_cap < b.n ? out_cap : b.n));
    return e;
}

int check_device_pointer(const void* p, int* dev) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess || attr.type != cudaMemoryTypeDevice) {
        cudaGetLastError();
        return ATREX_ERR_INVALID;
    }
    *dev = attr.device;
    return ATREX_OK;
}

}  // namespace

extern "C" uint64_t atrex_release_scratch_bytes(uint64_t n) {
    if (n > ATREX_RELEASE_MAX_ENTRIES) return 0;
    return scratch_bytes_for(n < 1 ? 1 : n);
}

extern "C" int atrex_entries_sort_by_key(const atrex_entry_t* d_entries, uint64_t n, atrex_entry_t* d_out,
                                         void* d_scratch, uint64_t scratch_bytes, void* stream) {
    if (n > ATREX_RELEASE_MAX_ENTRIES) return ATREX_ERR_TOO_LARGE;
    if (n == 0) return ATREX_OK;
    if (!d_entries || !d_out || !d_scratch || d_entries == d_out) return ATREX_ERR_INVALID;
    if (((uintptr_t)d_entries & 7u) || ((uintptr_t)d_out & 7u) || ((uintptr_t)d_scratch & 255u)) return ATREX_ERR_INVALID;
    if (scratch_bytes < scratch_bytes_for(n)) return ATREX_ERR_NOMEM;
    int dev = 0;
    if (check_device_pointer(d_entries, &dev) != ATREX_OK) return ATREX_ERR_INVALID;
    DeviceGuard guard(dev);
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t m = (uint32_t)n;
    int n_sms = 0;
    if (prepare_sort_kernels(&n_sms) != ATREX_OK) return ATREX_ERR_CUDA;
    if (n <= COUNT_SORT_MAX) {   // (above, counting takes longer than the binned sort's launches)
        ReportSlot report(s);
        if (!report.get()) return ATREX_ERR_NOMEM;
        const uint32_t per_cta = n <= 4096 ? 32 : 64, grid = (m + per_cta - 1) / per_cta;
        auto* kernel = n <= 4096 ? count_sort_kernel<1> : count_sort_kernel<2>;
        if (launch_chained(kernel, grid, COUNT_THREADS, (size_t)(m + 1) / 2 * 16, s, d_entries, m, d_out, report.get(), report.number()) != cudaSuccess)
            return ATREX_ERR_CUDA;
        return report.wait() == cudaSuccess ? ATREX_OK : ATREX_ERR_CUDA;
    }
    {
        ReportSlot report(s);
        if (!report.get()) return ATREX_ERR_NOMEM;
        const BinSort b = carve_bins(d_scratch, d_entries, n, false, report);
        if (launch_clear(b, s) != cudaSuccess) return ATREX_ERR_CUDA;
        const uint32_t want = (m + 4 * BIN_THREADS - 1) / (4 * BIN_THREADS), most = 4u * (uint32_t)n_sms;
        if (launch_chained(bin_keys_kernel, want < most ? want : most, BIN_THREADS, 0, s, b) != cudaSuccess ||
            launch_bins(b, 0, d_out, n, n_sms, s) != cudaSuccess || report.wait() != cudaSuccess)
            return ATREX_ERR_CUDA;
        if (!((volatile BinReport*)report.get())->overflow) return ATREX_OK;
    }

    const Scratch sc = carve(d_scratch, n);
    if (cudaMemsetAsync(sc.ctl, 0, sizeof(ReleaseCtl), s) != cudaSuccess) return ATREX_ERR_CUDA;
    if (reset_or_and(sc, s) != ATREX_OK) return ATREX_ERR_CUDA;
    init_key_words_kernel<<<grid_for(n, 256), 256, 0, s>>>(d_entries, m, sc.words[0], sc.idx[0], sc.ctl);
    if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
    ReleaseCtl host;
    if (read_ctl(sc, &host, s) != ATREX_OK) return ATREX_ERR_CUDA;
    const int cur = sort_by_word(sc, 0, m, host.word_or ^ host.word_and, s);
    if (cur < 0) return cur;
    gather_entries_kernel<<<grid_for(n, 256), 256, 0, s>>>(d_entries, sc.idx[cur], m, d_out);
    if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? ATREX_OK : ATREX_ERR_CUDA;
}

extern "C" int atrex_entries_rank(const atrex_entry_t* d_entries, uint64_t n, uint32_t phase, uint32_t coverage_ppm,
                                  atrex_entry_t* d_ranked, double* d_cum_share, uint64_t out_cap,
                                  atrex_rank_result_t* h_result, void* d_scratch, uint64_t scratch_bytes,
                                  void* stream) {
    if (!h_result) return ATREX_ERR_INVALID;
    *h_result = atrex_rank_result_t{};
    if (n > ATREX_RELEASE_MAX_ENTRIES) return ATREX_ERR_TOO_LARGE;
    if (phase >= ATREX_MAX_PHASES || coverage_ppm > 1000000u) return ATREX_ERR_INVALID;
    if (n == 0) return ATREX_OK;
    if (!d_entries || !d_scratch || (out_cap && (!d_ranked || !d_cum_share))) return ATREX_ERR_INVALID;
    if (((uintptr_t)d_entries & 7u) || ((uintptr_t)d_ranked & 7u) || ((uintptr_t)d_cum_share & 7u) ||
        ((uintptr_t)d_scratch & 255u) || (const void*)d_entries == (const void*)d_ranked)
        return ATREX_ERR_INVALID;
    if (scratch_bytes < scratch_bytes_for(n)) return ATREX_ERR_NOMEM;
    int dev = 0;
    if (check_device_pointer(d_entries, &dev) != ATREX_OK) return ATREX_ERR_INVALID;
    DeviceGuard guard(dev);
    cudaStream_t s = (cudaStream_t)stream;
    int n_sms = 0;
    if (prepare_sort_kernels(&n_sms) != ATREX_OK) return ATREX_ERR_CUDA;
    {
        ReportSlot slot(s);
        if (!slot.get()) return ATREX_ERR_NOMEM;
        const uint32_t cap = (uint32_t)(out_cap < n ? out_cap : n);
        cudaError_t e;
        if (n <= COUNT_RANK_MAX) {
            e = launch_chained(count_rank_kernel, ((uint32_t)n + 31) / 32, COUNT_THREADS, (size_t)n * 26, s, d_entries, (uint32_t)n, phase, coverage_ppm,
                               d_ranked, d_cum_share, cap, slot.get(), slot.number());
        } else {
            const BinSort b = carve_bins(d_scratch, d_entries, n, true, slot);
            const uint32_t want = ((uint32_t)n + 4 * BIN_THREADS - 1) / (4 * BIN_THREADS), most = 4u * (uint32_t)n_sms, tiles = tiles_of(b, (uint32_t)n);
            e = launch_clear(b, s);
            if (e == cudaSuccess) e = launch_chained(bin_phase_kernel, want < most ? want : most, BIN_THREADS, 0, s, b, phase);
            if (e == cudaSuccess) e = launch_bins(b, coverage_ppm, d_ranked, cap, n_sms, s);
            if (e == cudaSuccess)
                e = launch_chained(bin_share_kernel, tiles < CUM_CTAS * (uint32_t)n_sms ? tiles : CUM_CTAS * (uint32_t)n_sms, CUM_THREADS, 0, s, b, d_cum_share, cap);
        }
        if (e != cudaSuccess || slot.wait() != cudaSuccess) return ATREX_ERR_CUDA;
        const volatile BinReport* r = slot.get();
        if (r->too_large || !r->overflow) {
            h_result->n_phase = r->counter;
            h_result->total_lo = r->total_lo;
            h_result->total_hi = r->total_hi;
            if (r->too_large) return ATREX_ERR_TOO_LARGE;
            h_result->n_keep = r->n_keep;
            h_result->covered_lo = r->covered_lo;
            h_result->covered_hi = r->covered_hi;
            return ATREX_OK;
        }
    }

    const Scratch sc = carve(d_scratch, n);
    // 1. the phase's entries as (key, index) pairs, their count and exact total
    if (cudaMemsetAsync(sc.ctl, 0, sizeof(ReleaseCtl), s) != cudaSuccess) return ATREX_ERR_CUDA;
    if (reset_or_and(sc, s) != ATREX_OK) return ATREX_ERR_CUDA;
    filter_phase_kernel<<<grid_for(n, 256), 256, 0, s>>>(d_entries, (uint32_t)n, phase, sc.words[0], sc.idx[0], sc.ctl);
    if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
    ReleaseCtl host;
    if (read_ctl(sc, &host, s) != ATREX_OK) return ATREX_ERR_CUDA;
    const uint32_t m = (uint32_t)host.counter;
    const ull total_lo = host.total_lo, total_hi = host.total_hi;
    h_result->n_phase = m;
    h_result->total_lo = total_lo;
    h_result->total_hi = total_hi;
    if (m == 0) return ATREX_OK;
    if ((total_hi >> 44) != 0) return ATREX_ERR_TOO_LARGE;  // T * 10^6 must fit 128 bits

    // 2. least significant word first: key ascending, then ~wt_lo, then ~wt_hi
    int cur = sort_by_word(sc, 0, m, host.word_or ^ host.word_and, s);
    if (cur < 0) return cur;
    for (int high = 0; high < 2; ++high) {
        if (reset_or_and(sc, s) != ATREX_OK) return ATREX_ERR_CUDA;
        gather_wt_words_kernel<<<grid_for(m, 256), 256, 0, s>>>(d_entries, sc.idx[cur], m, high, sc.words[cur], sc.ctl);
        if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
        if (read_ctl(sc, &host, s) != ATREX_OK) return ATREX_ERR_CUDA;
        cur = sort_by_word(sc, cur, m, host.word_or ^ host.word_and, s);
        if (cur < 0) return cur;
    }

    // 3. exact running sum, shares, coverage cut: the smallest k with 10^6 * prefix_k >= ppm * T,
    //    i.e. prefix_k >= ceil(ppm * T / 10^6)
    typedef unsigned __int128 u128;
    const u128 total = ((u128)total_hi << 64) | total_lo;
    const u128 need = ((u128)coverage_ppm * total + 999999u) / 1000000u;
    const uint32_t blocks = (m + SCAN_BLOCK - 1) / SCAN_BLOCK;
    rank_block_sums_kernel<<<blocks, SCAN_BLOCK, 0, s>>>(d_entries, sc.idx[cur], m, sc.bsums);
    rank_scan_sums_kernel<<<1, SCAN_BLOCK, 0, s>>>(sc.bsums, blocks);
    rank_emit_kernel<<<blocks, SCAN_BLOCK, 0, s>>>(d_entries, sc.idx[cur], m, sc.bsums, total_lo, total_hi, (ull)need,
                                                   (ull)(need >> 64), d_ranked, d_cum_share,
                                                   (uint32_t)(out_cap < m ? out_cap : m), sc.ctl);
    if (cudaGetLastError() != cudaSuccess) return ATREX_ERR_CUDA;
    if (read_ctl(sc, &host, s) != ATREX_OK) return ATREX_ERR_CUDA;
    h_result->n_keep = host.n_keep;
    h_result->covered_lo = host.covered_lo;
    h_result->covered_hi = host.covered_hi;
    return ATREX_OK;
}
