// Finalize: per-phase totals (Eq. 2's D^phi), per-key weights (Eq. 3 normalised per phase),
// roofline times (Eq. 1), compaction, and the ranked top-k (Table 2).
//
// All floating-point results come from explicit round-to-nearest intrinsics on exact
// integers, so they have one correct bit pattern: fl(fl(wt) / fl(T)) and
// fmax(fl(F) / P, fl(M) / beta).
#include <cstddef>

#include "atrex_dev.cuh"
#include "kernels.h"

namespace atrex {

constexpr int FIN_THREADS = 256;

// A word for the host in pinned memory: both halves carry the stamp of the answer they belong to and are stored whole, so
// that the host sees for itself what has arrived.  (A flag behind the words has to wait for a fence of the system first, which is
// a round trip over the link: 2 us of an answer.)
__device__ __forceinline__ void tell(ulonglong2* to, ull word, uint32_t stamp) {
    const ull mark = (ull)stamp << 32;
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(to), "l"(mark | (uint32_t)word), "l"(mark | (word >> 32)) : "memory");
}
constexpr uint32_t TOT_ILP = 6;

struct SlotView {
    ull key, count, lo, hi;
    bool live;
};

__device__ __forceinline__ SlotView load_slot(const TableRef& t, ull i) {
    SlotView v;
    ull sk = t.keys[i];
    v.live = sk != 0;
    v.key = ~sk;
    v.lo = v.count = v.hi = 0;
    if (v.live) {
        ulonglong2 x = t.vals[i];
        v.lo = x.x;
        v.count = x.y & COUNT_MASK;
        v.hi = x.y >> HI_SHIFT;
    }
    return v;
}

__device__ __forceinline__ uint32_t topk_first_digit(ull lo, ull hi) {
    if ((lo | hi) == 0) return 0;
    const int e = hi ? 128 - __clzll((long long)hi) : 64 - __clzll((long long)lo);      // 1 .. 88
    uint32_t m;
    if (e > 69) m = (uint32_t)(hi >> (e - 70));
    else if (e > 64) m = (uint32_t)((hi << (70 - e)) | (lo >> (e - 6)));
    else m = (uint32_t)(e >= 6 ? lo >> (e - 6) : lo << (6 - e));
    return ((uint32_t)e << 5) | (m & 31u);
}
constexpr uint32_t FIRST_BINS = (88 << 5) + 32;
static_assert(FIRST_BINS <= TOPK_BINS && FIRST_BINS % 4 == 0, "first digits fit the histogram");

// ---- per-phase totals -------------------------------------------------------------------
// Each thread keeps private per-phase 128-bit sums in its own shared-memory column; columns are added per
// CTA and folded into accumulators in the control block with a carry-aware pair of atomics.  The last CTA
// moves the accumulators to their place and clears them (and the emit kernel's output count), so that no
// launch is spent on clearing.  On the way the keys are counted by the first digit of the top-k selection (per
// phase, for the top-k), which saves that call a pass over the table; the next pass's counters are
// cleared here.  Bound by DRAM (525 MB: 91 us), given 512 threads per SM or more: shared memory holds that many up to eight
// phases (16 M keys, whole finalize: five phases 650 -> 569 us, eight 650 -> 582; with one CTA of 256 threads before).
__device__ __forceinline__ bool last_cta(ull* done) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(done, 1ull) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    return s_last;
}

constexpr uint32_t TOT_THREADS = 256, TOT_WIDE_FROM = 7;       // (from seven phases on one CTA per SM, of twice as many threads)
constexpr uint32_t totals_threads(uint32_t n_phases) { return n_phases < TOT_WIDE_FROM ? TOT_THREADS : 2 * TOT_THREADS; }
constexpr size_t totals_smem(uint32_t n_phases) { return (size_t)n_phases * (totals_threads(n_phases) * 28 + FIRST_BINS * 4); }

template <uint32_t THREADS>
__global__ void __launch_bounds__(THREADS) totals_kernel(TableRef tab, ull n_slots, uint32_t n_phases, const __grid_constant__ GivenTotals given,
                                                             uint32_t* hist, uint32_t* next_hist) {
    Control* ctl = tab.ctl;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t t = threadIdx.x;
    ull* s_lo = reinterpret_cast<ull*>(smem_raw);                                    // [n_phases][THREADS] each
    ull* s_hi = s_lo + n_phases * THREADS;
    ull* s_cnt = s_hi + n_phases * THREADS;
    uint32_t* s_nk = reinterpret_cast<uint32_t*>(s_cnt + n_phases * THREADS);
    uint32_t* s_hist = s_nk + n_phases * THREADS;                                    // [n_phases][FIRST_BINS]
    for (uint32_t i = t; i < n_phases * THREADS; i += THREADS) {
        s_lo[i] = 0; s_hi[i] = 0; s_cnt[i] = 0; s_nk[i] = 0;
    }
    for (uint32_t i = t; i < n_phases * FIRST_BINS; i += THREADS) s_hist[i] = 0;
    __syncthreads();
    grid_dependency_wait();
    for (uint32_t i = blockIdx.x * THREADS + t; i < n_phases * TOPK_BINS / 4; i += gridDim.x * THREADS)
        reinterpret_cast<uint4*>(next_hist)[i] = make_uint4(0, 0, 0, 0);
    // six slots per thread in flight
    const ull stride = (ull)gridDim.x * THREADS;
    for (ull i0 = (ull)blockIdx.x * THREADS + t; i0 < n_slots; i0 += stride * TOT_ILP) {
        ull sk[TOT_ILP];
        ulonglong2 x[TOT_ILP];
#pragma unroll
        for (int u = 0; u < TOT_ILP; ++u) sk[u] = i0 + u * stride < n_slots ? tab.keys[i0 + u * stride] : 0ull;
#pragma unroll
        for (int u = 0; u < TOT_ILP; ++u) x[u] = i0 + u * stride < n_slots ? tab.vals[i0 + u * stride] : make_ulonglong2(0, 0);  // unconditional: no wait for the keys
#pragma unroll
        for (int u = 0; u < TOT_ILP; ++u) {
            if (sk[u] == 0) continue;
            const uint32_t p = (uint32_t)(~sk[u] >> 48) & (ATREX_MAX_PHASES - 1);
            const ull hi = x[u].y >> HI_SHIFT;
            if (p >= n_phases) {   // (rare: a merged entry of a phase that records of this handle cannot have)
                const ull old = atomicAdd(&ctl->acc_lo[p], x[u].x);
                atomicAdd(&ctl->acc_hi[p], hi + (old + x[u].x < old ? 1ull : 0ull));
                atomicAdd(&ctl->acc_count[p], x[u].y & COUNT_MASK);
                atomicAdd(&ctl->acc_keys[p], 1ull);
                continue;
            }
            const uint32_t at = p * THREADS + t;
            const ull o = s_lo[at], n = o + x[u].x;
            s_lo[at] = n;
            s_hi[at] += hi + (n < o ? 1ull : 0ull);
            s_cnt[at] += x[u].y & COUNT_MASK;
            s_nk[at] += 1;
            atomicAdd(&s_hist[p * FIRST_BINS + topk_first_digit(x[u].x, hi)], 1u);
        }
    }
    grid_dependents_launch();
    __syncthreads();
    for (uint32_t p = 0; p < n_phases; ++p)
        for (uint32_t i = t; i < FIRST_BINS; i += THREADS)
            if (s_hist[p * FIRST_BINS + i] != 0) atomicAdd(&hist[p * TOPK_BINS + i], s_hist[p * FIRST_BINS + i]);
    const uint32_t lane = t & 31;
    for (uint32_t p = t >> 5; p < n_phases; p += THREADS / 32) {   // a warp per phase
        ull lo = 0, hi = 0, cnt = 0, nk = 0;
        for (uint32_t j = p * THREADS + lane; j < (p + 1) * THREADS; j += 32) {
            const ull n = lo + s_lo[j];
            hi += s_hi[j] + (n < lo ? 1ull : 0ull);
            lo = n;
            cnt += s_cnt[j];
            nk += s_nk[j];
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const ull olo = __shfl_xor_sync(0xFFFFFFFFu, lo, d), ohi = __shfl_xor_sync(0xFFFFFFFFu, hi, d), n = lo + olo;
            hi += ohi + (n < lo ? 1ull : 0ull);
            lo = n;
            cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, d);
            nk += __shfl_xor_sync(0xFFFFFFFFu, nk, d);
        }
        if (lane == 0 && nk != 0) {
            const ull old = atomicAdd(&ctl->acc_lo[p], lo);
            atomicAdd(&ctl->acc_hi[p], hi + (old + lo < old ? 1ull : 0ull));
            atomicAdd(&ctl->acc_count[p], cnt);
            atomicAdd(&ctl->acc_keys[p], nk);
        }
    }
    if (!last_cta(&ctl->tot_done)) return;
    if (t < ATREX_MAX_PHASES) {
        ctl->total_lo[t] = given.use ? given.lo[t] : ld_relaxed(&ctl->acc_lo[t]);
        ctl->total_hi[t] = given.use ? given.hi[t] : ld_relaxed(&ctl->acc_hi[t]);
        ctl->keys_per_phase[t] = ld_relaxed(&ctl->acc_keys[t]);
        ctl->count_per_phase[t] = ld_relaxed(&ctl->acc_count[t]);
        ctl->acc_lo[t] = ctl->acc_hi[t] = ctl->acc_keys[t] = ctl->acc_count[t] = 0;
    }
    if (t == 0) ctl->tot_done = ctl->n_out = 0;
}

// ---- per-key results ----------------------------------------------------------------------
// The work table is probed a bucket of four keys at a time (one 32-byte load), from bucket to bucket by double hashing
// (strides coprime to the partition's bucket count): the longest of a warp's 32 probe sequences is what the warp waits for.
// Slot by slot it was eight loads; with linear probing several times that.  Buckets fill from the first way on.
constexpr ull WORK_PAIR = 0x0000FFFFFFFFFFFFull;
__device__ __forceinline__ uint32_t work_stride(const WorkRef& w, uint32_t h) {
    return (uint32_t)(w.strides >> (8 * ((h >> 3) & 7u))) & 0xFFu;
}
__device__ __forceinline__ uint32_t work_start(const WorkRef& w, uint32_t h) { return __umulhi(h * 0x85EBCA6Bu, w.Cw / WORK_WAYS); }
__device__ __forceinline__ uint32_t work_next(const WorkRef& w, uint32_t bucket, uint32_t advance) {
    bucket += advance;
    while (bucket >= w.Cw / WORK_WAYS) bucket -= w.Cw / WORK_WAYS;    // (a small table's stride may be longer than the table)
    return bucket;
}
struct WorkKeys {
    ull k[WORK_WAYS];
};
__device__ __forceinline__ WorkKeys load_work_keys(const ull* bucket) {
    WorkKeys x;
    asm("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(x.k[0]), "=l"(x.k[1]), "=l"(x.k[2]), "=l"(x.k[3]) : "l"(bucket));
    return x;
}
// The way that holds `pair`, WORK_WAYS if none does; `dtype` is set where one does.
__device__ __forceinline__ uint32_t work_way(const WorkKeys& x, ull pair, uint32_t& dtype) {
    uint32_t way = WORK_WAYS;
#pragma unroll
    for (uint32_t i = 0; i < WORK_WAYS; ++i) {
        if (((x.k[i] ^ (WORK_USED | pair)) & (WORK_USED | WORK_PAIR)) != 0) continue;
        way = i;
        dtype = (uint32_t)(x.k[i] >> 48) & (ATREX_MAX_DTYPES - 1);
    }
    return way;
}
__device__ __forceinline__ double roofline_of(const double2& work, uint32_t dtype, const atrex_hw_peaks_t& pk) {
    return fmax(__ddiv_rn(work.x, pk.peak_flops[dtype]), __ddiv_rn(work.y, pk.peak_bw));
}
__device__ __forceinline__ double roofline_time(const WorkRef& w, const atrex_hw_peaks_t& pk, ull key) {
    const double qnan = __longlong_as_double(0x7FF8000000000000ll);
    if (w.keys == nullptr) return qnan;
    const uint32_t h = hash32(key & WORK_PAIR), first = part_of(h, w.lp) * w.Cw, advance = work_stride(w, h);
    uint32_t bucket = work_start(w, h);
    for (uint32_t probe = 0; probe < w.Cw / WORK_WAYS; ++probe) {
        const uint32_t at = first + bucket * WORK_WAYS;
        const WorkKeys x = load_work_keys(w.keys + at);
        uint32_t dtype = 0;
        const uint32_t way = work_way(x, key & WORK_PAIR, dtype);
        if (way != WORK_WAYS) return roofline_of(w.rows[at + way], dtype, pk);
        if (x.k[WORK_WAYS - 1] == 0) break;
        bucket = work_next(w, bucket, advance);
    }
    return qnan;
}

__device__ __forceinline__ atrex_entry_t make_entry(const SlotView& v, const double* dT, const bool* zeroT,
                                                    const FinalizeParams& p) {
    atrex_entry_t e;
    e.key = v.key;
    e.count = v.count;
    e.wt_lo = v.lo;
    e.wt_hi = v.hi;
    int ph = (int)(v.key >> 48) & (ATREX_MAX_PHASES - 1);
    e.phase_weight = zeroT[ph] ? 0.0 : __ddiv_rn(u128_to_f64_rn(v.hi, v.lo), dT[ph]);
    e.roofline_s = roofline_time(p.work, p.peaks, v.key);
    return e;
}

__device__ __forceinline__ void store_entry(atrex_entry_t* dst, const atrex_entry_t& e) {
    ulonglong2* q = reinterpret_cast<ulonglong2*>(dst);
    q[0] = make_ulonglong2(e.key, e.count);
    q[1] = make_ulonglong2(e.wt_lo, e.wt_hi);
    q[2] = make_ulonglong2((ull)__double_as_longlong(e.phase_weight), (ull)__double_as_longlong(e.roofline_s));
}

// Row `row` of phase q's best, for the host.
__device__ __forceinline__ void tell_row(const PickParams& p, uint32_t q, uint32_t row, const atrex_entry_t& e) {
    if (p.k > TOPK_TOLD_K) {
        store_entry(p.host_top + (size_t)q * TOPK_PICK_K + row, e);
        return;
    }
    ulonglong2* to = p.host_told + ((size_t)q * TOPK_TOLD_K + row) * 6;
    const ull words[6] = {e.key, e.count, e.wt_lo, e.wt_hi, (ull)__double_as_longlong(e.phase_weight), (ull)__double_as_longlong(e.roofline_s)};
#pragma unroll
    for (int i = 0; i < 6; ++i) tell(to + i, words[i], p.fin.stamp);
}
// ... and how many rows there are, PICK_NONE: not answered this way (one thread; all rows stored before)
__device__ __forceinline__ void tell_count(const PickParams& p, uint32_t q, uint32_t n) {
    if (p.k > TOPK_TOLD_K) __threadfence_system();      // (rows without stamps)
    *(volatile ull*)&p.host_n[q] = (ull)p.fin.stamp << 32 | n;   // the host waits for this word
}

__device__ __forceinline__ void load_phase_totals(const Control* ctl, double* dT, bool* zeroT) {
    if (threadIdx.x < ATREX_MAX_PHASES) {
        ull lo = ctl->total_lo[threadIdx.x], hi = ctl->total_hi[threadIdx.x];
        dT[threadIdx.x] = u128_to_f64_rn(hi, lo);
        zeroT[threadIdx.x] = (lo | hi) == 0;
    }
    __syncthreads();
}

// Each warp looks at 128 slots per round (four coalesced rows), queues the live ones in shared
// memory and then works through the queue with all lanes busy: at a table load of a third, the
// divisions and the work-table probe run on full warps instead of one lane in three.  A lane probes for two
// entries side by side (four need more registers than four CTAs per SM have, and three CTAs are slower), and the entries
// go out through shared memory in whole lines.  Bound by latency and instructions at half occupancy (3.1 M keys
// of 5.8 M slots: 121 -> 97 us, DRAM 45 %; 15 M of 21.9 M: 540 -> 475; one entry at a time over the same buckets 155, four
// 113; five CTAs of 48 registers: 2 % more on the whole refresh).
constexpr int EMIT_ILP = 4;
constexpr int EMIT_PROBES = 2;
constexpr int EMIT_WARPS = FIN_THREADS / 32;

__global__ void __launch_bounds__(FIN_THREADS) emit_kernel(const __grid_constant__ FinalizeParams p) {
    __shared__ double dT[ATREX_MAX_PHASES];
    __shared__ bool zeroT[ATREX_MAX_PHASES];
    __shared__ ull q_key[EMIT_WARPS][32 * EMIT_ILP];
    __shared__ ulonglong2 q_val[EMIT_WARPS][32 * EMIT_ILP];
    __shared__ ulonglong2 s_out[EMIT_WARPS][32 * 3];
    grid_dependency_wait();
    load_phase_totals(p.ctl, dT, zeroT);
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    const ull stride = (ull)gridDim.x * blockDim.x;
    const ull rounds = (p.n_slots + stride * EMIT_ILP - 1) / (stride * EMIT_ILP);  // uniform: warps stay converged
    for (ull r = 0; r < rounds; ++r) {
        uint32_t total = 0;
        {
            ull sk[EMIT_ILP];
            ulonglong2 xv[EMIT_ILP];
#pragma unroll
            for (int u = 0; u < EMIT_ILP; ++u) {
                const ull i = (r * EMIT_ILP + u) * stride + (ull)blockIdx.x * blockDim.x + threadIdx.x;
                sk[u] = i < p.n_slots ? p.t.keys[i] : 0ull;
                xv[u] = i < p.n_slots ? p.t.vals[i] : make_ulonglong2(0, 0);  // with the key, not after it
            }
#pragma unroll
            for (int u = 0; u < EMIT_ILP; ++u) {
                const unsigned live = __ballot_sync(0xFFFFFFFFu, sk[u] != 0);
                if (sk[u] != 0) {
                    const uint32_t at = total + __popc(live & ((1u << lane) - 1u));
                    q_key[w][at] = ~sk[u];
                    q_val[w][at] = xv[u];
                }
                total += __popc(live);
            }
        }
        if (total == 0) continue;
        ull base = 0;
        if (lane == 0) base = atomicAdd(&p.ctl->n_out, (ull)total);
        __syncwarp();
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        for (uint32_t j0 = 0; j0 < total; j0 += 32 * EMIT_PROBES) {
            // The entries' rows of the work table: the partition's first slot, the bucket, stride (once found: slot and type).
            uint32_t slot[EMIT_PROBES], bucket[EMIT_PROBES], advance[EMIT_PROBES], pending = 0, known = 0;
#pragma unroll
            for (int u = 0; u < EMIT_PROBES; ++u) {
                slot[u] = bucket[u] = advance[u] = 0;
                if (p.work.keys != nullptr && j0 + lane + 32u * u < total) {
                    const uint32_t h = hash32(q_key[w][j0 + lane + 32u * u]);
                    slot[u] = part_of(h, p.work.lp) * p.work.Cw;
                    bucket[u] = work_start(p.work, h);
                    advance[u] = work_stride(p.work, h);
                    pending |= 1u << u;
                }
            }
            for (uint32_t probe = 0; probe < p.work.Cw && __any_sync(0xFFFFFFFFu, pending != 0); ++probe) {
                WorkKeys x[EMIT_PROBES];
#pragma unroll
                for (int u = 0; u < EMIT_PROBES; ++u)
                    if (pending & (1u << u)) x[u] = load_work_keys(p.work.keys + (slot[u] + bucket[u] * WORK_WAYS));
#pragma unroll
                for (int u = 0; u < EMIT_PROBES; ++u) {
                    if (!(pending & (1u << u))) continue;
                    uint32_t dtype = 0;
                    const uint32_t way = work_way(x[u], q_key[w][j0 + lane + 32u * u] & WORK_PAIR, dtype);
                    if (way != WORK_WAYS) {
                        pending &= ~(1u << u);
                        known |= 1u << u;
                        slot[u] += bucket[u] * WORK_WAYS + way;
                        advance[u] = dtype;
                    } else if (x[u].k[WORK_WAYS - 1] == 0) {
                        pending &= ~(1u << u);
                    } else {
                        bucket[u] = work_next(p.work, bucket[u], advance[u]);
                    }
                }
            }
            double2 work[EMIT_PROBES];
#pragma unroll
            for (int u = 0; u < EMIT_PROBES; ++u) work[u] = known & (1u << u) ? p.work.rows[slot[u]] : make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < EMIT_PROBES; ++u) {
                const uint32_t j1 = j0 + 32u * u, j = j1 + lane;
                if (j1 >= total) break;
                if (j < total) {
                    const ull key = q_key[w][j];
                    const ulonglong2 x = q_val[w][j];
                    const int ph = (int)(key >> 48) & (ATREX_MAX_PHASES - 1);
                    const double weight = zeroT[ph] ? 0.0 : __ddiv_rn(u128_to_f64_rn(x.y >> HI_SHIFT, x.x), dT[ph]);
                    const double roofline = known & (1u << u) ? roofline_of(work[u], advance[u], p.peaks) : __longlong_as_double(0x7FF8000000000000ll);
                    s_out[w][3 * lane] = make_ulonglong2(key, x.y & COUNT_MASK);
                    s_out[w][3 * lane + 1] = make_ulonglong2(x.x, x.y >> HI_SHIFT);
                    s_out[w][3 * lane + 2] = make_ulonglong2((ull)__double_as_longlong(weight), (ull)__double_as_longlong(roofline));
                }
                __syncwarp();
                const ull at = base + j1;
                const uint32_t fit = at >= p.out_cap ? 0u : (uint32_t)min(p.out_cap - at, (ull)min(total - j1, 32u));
                ulonglong2* to = reinterpret_cast<ulonglong2*>(p.out + at);
#pragma unroll
                for (uint32_t k = lane; k < 96; k += 32)
                    if (k < 3 * fit) to[k] = s_out[w][k];
                __syncwarp();
            }
        }
    }
    grid_dependents_launch();
    if (!last_cta(&p.ctl->emit_done)) return;
    // the host's copy of the counters and totals, straight to pinned memory
    if (threadIdx.x < CONTROL_WORDS) tell(p.told + threadIdx.x, ld_relaxed(reinterpret_cast<const ull*>(p.ctl) + threadIdx.x), p.stamp);
    if (threadIdx.x == 0) p.ctl->emit_done = 0;
}

// ---- work table ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) work_insert_kernel(const atrex_work_t* rows, ull n, WorkRef w, Control* ctl) {
    for (ull i = (ull)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (ull)gridDim.x * blockDim.x) {
        atrex_work_t r = rows[i];
        if (r.dtype >= ATREX_MAX_DTYPES) {
            atomicOr(&ctl->work_status, ST_WORK_DTYPE);
            continue;
        }
        const ull pair = ((ull)r.op_id << 32) | (ull)r.shape_id;
        const uint32_t h = hash32(pair), first = part_of(h, w.lp) * w.Cw, advance = work_stride(w, h);
        uint32_t bucket = work_start(w, h);
        bool done = false;
        for (uint32_t probe = 0; probe < w.Cw && !done; ++probe) {
            const uint32_t at = first + bucket * WORK_WAYS + probe % WORK_WAYS;
            const ull old = atomicCAS(&w.keys[at], 0ull, WORK_USED | (ull)r.dtype << 48 | pair);
            if (old == 0) {
                w.rows[at] = make_double2(__ull2double_rn(r.flops), __ull2double_rn(r.bytes));
                done = true;
            } else if ((old & WORK_PAIR) == pair) {
                atomicOr(&ctl->work_status, ST_WORK_DUP);
                done = true;
            } else if (probe % WORK_WAYS == WORK_WAYS - 1) {
                bucket = work_next(w, bucket, advance);
            }
        }
        if (!done) atomicOr(&ctl->work_status, ST_WORK_FULL);
    }
}

// ---- top-k, the usual way -----------------------------------------------------------------
// All phases at once, without a word from the host in between: a first digit on a logarithmic scale (bit
// length and the five bits below the leading one: 3 % steps) is counted per phase; the digit of each
// phase's k-th key is found; the keys at or above it are collected; one CTA per phase ranks them exactly and
// writes the best k to pinned host memory.  Weights that span orders of magnitude leave a few dozen
// candidates beside the winners.  (Digits on a linear scale below the phase total's highest bit put every
// key of a flat trace into the lowest one: 26 000 candidates in one CTA's global-memory sort took 4 ms.)
//
// Every collecting CTA finds the digits for itself, a quarter of a phase's bins to a warp at a time: a
// microsecond, where a kernel of its own before this one cost four.
constexpr uint32_t QUARTER = TOPK_BINS / 4;

// Keys in one quarter of phase q's bins, quarter 0 the highest (one warp); v[u] = lane's four bins of step u, the
// highest bins in step 0 and lane 0.
__device__ __forceinline__ uint32_t load_quarter(const PickParams& p, uint32_t q, uint32_t quarter, uint4 (&v)[8]) {
    const uint4* hist = reinterpret_cast<const uint4*>(p.hist + (size_t)q * TOPK_BINS) + (TOPK_BINS - quarter * QUARTER) / 4 - 1 - (threadIdx.x & 31u);
    uint32_t sum = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = *(hist - 32 * u);
#pragma unroll
    for (int u = 0; u < 8; ++u) sum += v[u].x + v[u].y + v[u].z + v[u].w;
    return __reduce_add_sync(0xFFFFFFFFu, sum);
}

// the digit of phase q's k-th key, which lies in this quarter, `above` keys in higher ones (one warp)
__device__ __forceinline__ uint32_t digit_in_quarter(const PickParams& p, uint32_t q, uint32_t quarter, uint32_t above) {
    const uint32_t lane = threadIdx.x & 31u;
    uint4 v[8];
    load_quarter(p, q, quarter, v);
    uint32_t found = PICK_NONE;
#pragma unroll
    for (uint32_t u = 0; u < 8; ++u) {
        const uint32_t own = v[u].x + v[u].y + v[u].z + v[u].w, all = __reduce_add_sync(0xFFFFFFFFu, own);
        if (above < p.k && above + all >= p.k) {
            uint32_t incl = own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= (uint32_t)d) incl += o;
            }
            const uint32_t src = __ffs(__ballot_sync(0xFFFFFFFFu, above + incl >= p.k)) - 1;
            uint32_t at = above + incl - own + v[u].w, digit = TOPK_BINS - 1 - quarter * QUARTER - 4 * (32 * u + lane);
            if (at < p.k) { at += v[u].z; --digit; }
            if (at < p.k) { at += v[u].y; --digit; }
            if (at < p.k) { at += v[u].x; --digit; }
            found = __shfl_sync(0xFFFFFFFFu, at <= TOPK_PICK_MAX ? digit : PICK_NONE, src);
        }
        above += all;
    }
    return found;
}

// the digit of every phase's k-th key (all threads of a CTA; PICK_NONE: too many keys to rank this way)
__device__ __forceinline__ void find_digits(const PickParams& p, uint32_t* s_bin, uint32_t* s_sum) {
    const uint32_t warp = threadIdx.x >> 5;
    for (uint32_t i = warp; i < 4 * p.n_phases; i += blockDim.x / 32) {
        uint4 v[8];
        const uint32_t sum = load_quarter(p, i / 4, i % 4, v);
        if ((threadIdx.x & 31u) == 0) s_sum[i] = sum;
    }
    __syncthreads();
    if (warp < ATREX_MAX_PHASES) {
        uint32_t digit = PICK_NONE;
        if (warp < p.n_phases) {
            uint32_t above = 0, quarter = 0;
            while (quarter < 4 && above + s_sum[4 * warp + quarter] < p.k) above += s_sum[4 * warp + quarter++];
            if (quarter < 4) digit = digit_in_quarter(p, warp, quarter, above);
            else digit = above <= TOPK_PICK_MAX ? 0u : PICK_NONE;              // fewer than k keys: all of them
        }
        if ((threadIdx.x & 31u) == 0) s_bin[warp] = digit;
    }
    __syncthreads();
}

// the keys at or above that digit
__global__ void __launch_bounds__(FIN_THREADS) topk_collect_kernel(const __grid_constant__ PickParams p) {
    __shared__ uint32_t s_bin[ATREX_MAX_PHASES], s_sum[4 * ATREX_MAX_PHASES];
    static_assert(FIN_THREADS / 32 >= ATREX_MAX_PHASES, "a warp per phase");
    grid_dependency_wait();
    find_digits(p, s_bin, s_sum);
    if (blockIdx.x == 0 && threadIdx.x < ATREX_MAX_PHASES) p.fin.ctl->pick_bin[threadIdx.x] = s_bin[threadIdx.x];
    const TableRef& tab = p.fin.t;
    constexpr int ILP = 4;
    const ull stride = (ull)gridDim.x * FIN_THREADS, n_slots = p.fin.n_slots;
    for (ull i0 = (ull)blockIdx.x * FIN_THREADS + threadIdx.x; i0 < n_slots; i0 += stride * ILP) {
        ull sk[ILP];
        ulonglong2 x[ILP];
#pragma unroll
        for (int u = 0; u < ILP; ++u) {
            const ull i = i0 + u * stride;
            sk[u] = i < n_slots ? tab.keys[i] : 0ull;
            x[u] = i < n_slots ? tab.vals[i] : make_ulonglong2(0, 0);
        }
#pragma unroll
        for (int u = 0; u < ILP; ++u) {
            if (sk[u] == 0) continue;
            const uint32_t q = (uint32_t)(~sk[u] >> 48) & (ATREX_MAX_PHASES - 1);
            const ull hi = x[u].y >> HI_SHIFT;
            if (topk_first_digit(x[u].x, hi) < s_bin[q]) continue;      // (PICK_NONE: never)
            const ull pos = atomicAdd(&p.fin.ctl->sel_count_all[q], 1ull);
            if (pos < TOPK_PICK_MAX) {
                ull* dst = p.sel + ((ull)q * TOPK_PICK_MAX + pos) * 4;
                dst[0] = hi; dst[1] = x[u].x; dst[2] = ~sk[u]; dst[3] = i0 + u * stride;
            }
        }
    }
    grid_dependents_launch();
}

// The weighted time's place on a logarithmic scale, 4 096 steps to a doubling (19 bits).
constexpr int FINE_BITS = 12;
__device__ __forceinline__ uint32_t fine_digit(ull lo, ull hi) {
    if ((lo | hi) == 0) return 0;
    const int e = hi ? 128 - __clzll((long long)hi) : 64 - __clzll((long long)lo);      // 1 .. 88
    const ull top = e > 64 ? (hi << (128 - e)) | (e < 128 ? lo >> (e - 64) : 0ull) : lo << (64 - e);   // leading one at bit 63
    return ((uint32_t)e << FINE_BITS) | ((uint32_t)(top >> (63 - FINE_BITS)) & ((1u << FINE_BITS) - 1u));
}

// n candidates ranked: fine(a) is the place of one on a scale that agrees with before(a, b), which compares two of them; swap(a, b)
// exchanges them, emit(row, a) takes one of the best k (all threads of a CTA of THREADS)
constexpr uint32_t RANK_BINS = 2048, RANK_BIN_MAX = 32, RANK_BINS_FROM = 128;
struct RankBins {
    uint32_t count[RANK_BINS];             // of a bin, then where it starts
    uint32_t warp[32], low, high;
    uint16_t order[TOPK_PICK_MAX];         // candidates bin by bin
};
template <uint32_t THREADS, typename Fine, typename Before, typename Swap, typename Emit>
__device__ __forceinline__ void rank_candidates(RankBins& s, uint32_t n, uint32_t best, Fine fine, Before before, Swap swap, Emit emit) {
    const uint32_t t = threadIdx.x, lane = t & 31u, w = t >> 5;
    // More than a few: spread over bins between the smallest and the largest weighted time; a candidate counts those before
    // it in its own bin only.  (Some 900 candidates in each of four phases of a small table, the best 512: whole kernel 48 ->
    // 28.5 us, 55 barriers of a bitonic network before; the best 512 of 4 M keys 48 -> 22.5.  The best 100 of 85 000 keys, where every
    // candidate counted all others: 21.7 -> 19.4.)
    if (n > RANK_BINS_FROM) {
        constexpr uint32_t EACH = TOPK_PICK_MAX / THREADS, BINS = RANK_BINS / THREADS;
        if (t == 0) { s.low = ~0u; s.high = 0; }
        for (uint32_t i = t; i < RANK_BINS; i += THREADS) s.count[i] = 0;
        __syncthreads();
        uint32_t digit[EACH], place[EACH], least = ~0u, most = 0;
#pragma unroll
        for (uint32_t u = 0; u < EACH; ++u) {
            const uint32_t i = u * THREADS + t;
            if (i >= n) continue;
            digit[u] = fine(i);
            least = min(least, digit[u]);
            most = max(most, digit[u]);
        }
        least = __reduce_min_sync(0xFFFFFFFFu, least);
        most = __reduce_max_sync(0xFFFFFFFFu, most);
        if (lane == 0) {
            atomicMin(&s.low, least);
            atomicMax(&s.high, most);
        }
        __syncthreads();
        const uint32_t low = s.low, high = s.high;
        bool crowded = false;
#pragma unroll
        for (uint32_t u = 0; u < EACH; ++u) {
            if (u * THREADS + t >= n) continue;
            digit[u] = (high - digit[u]) * RANK_BINS / (high - low + 1);          // (below 2^30)
            place[u] = atomicAdd(&s.count[digit[u]], 1u);
            crowded = crowded || place[u] >= RANK_BIN_MAX;
        }
        if (!__syncthreads_or(crowded)) {
            uint32_t c[BINS], own = 0;
#pragma unroll
            for (uint32_t i = 0; i < BINS; ++i) own += c[i] = s.count[t * BINS + i];
            uint32_t incl = own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= (uint32_t)d) incl += o;
            }
            if (lane == 31) s.warp[w] = incl;
            __syncthreads();
            uint32_t at = __reduce_add_sync(0xFFFFFFFFu, lane < w ? s.warp[lane] : 0u) + incl - own;
#pragma unroll
            for (uint32_t i = 0; i < BINS; ++i) {
                s.count[t * BINS + i] = at;
                at += c[i];
            }
            __syncthreads();
#pragma unroll
            for (uint32_t u = 0; u < EACH; ++u)
                if (u * THREADS + t < n) s.order[s.count[digit[u]] + place[u]] = (uint16_t)(u * THREADS + t);
            __syncthreads();
#pragma unroll
            for (uint32_t u = 0; u < EACH; ++u) {
                const uint32_t i = u * THREADS + t;
                if (i >= n) continue;
                const uint32_t first = s.count[digit[u]], end = digit[u] + 1 < RANK_BINS ? s.count[digit[u] + 1] : n;
                uint32_t row = first;
                for (uint32_t j = first; j < end; ++j) row += before(s.order[j], i) ? 1u : 0u;
                if (row < best) emit(row, i);
            }
            return;
        }
        // (many alike: as follows)
    }
    if (n <= 512) {     // every candidate counts those before it
        if (threadIdx.x < n) {
            uint32_t row = 0;
            for (uint32_t j = 0; j < n; ++j) row += before(j, threadIdx.x) ? 1u : 0u;
            if (row < best) emit(row, threadIdx.x);
        }
        return;
    }
    // bitonic network over positions 0 .. n - 1 (every comparator puts the better one first, so that
    // positions beyond n can be left out)
    for (uint32_t k = 2; k / 2 < n; k <<= 1) {
        for (uint32_t j = k >> 1; j; j >>= 1) {
            for (uint32_t t = threadIdx.x; t < n; t += blockDim.x) {
                const uint32_t lo = (t / j) * 2 * j + (t & (j - 1));
                const uint32_t hi = j == k >> 1 ? (lo | (k - 1)) - (lo & (k - 1)) : lo + j;
                if (hi < n && before(hi, lo)) swap(lo, hi);
            }
            __syncthreads();
        }
    }
    for (uint32_t i = threadIdx.x; i < min(n, best); i += blockDim.x) emit(i, i);
}
template <typename T>
__device__ __forceinline__ void exchange(T& a, T& b) {
    const T x = a;
    a = b;
    b = x;
}

// the candidates of each phase ranked: weighted time descending, key ascending (one CTA per phase)
constexpr uint32_t RANK_THREADS = 512;
__global__ void __launch_bounds__(RANK_THREADS) topk_rank_kernel(const __grid_constant__ PickParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ull* s_hi = reinterpret_cast<ull*>(smem_raw);
    ull* s_lo = s_hi + TOPK_PICK_MAX;
    ull* s_key = s_lo + TOPK_PICK_MAX;
    uint32_t* s_at = reinterpret_cast<uint32_t*>(s_key + TOPK_PICK_MAX);
    __shared__ double dT[ATREX_MAX_PHASES];
    __shared__ bool zeroT[ATREX_MAX_PHASES];
    grid_dependency_wait();
    const uint32_t q = blockIdx.x;
    if (p.fin.ctl->pick_bin[q] == PICK_NONE) {
        if (threadIdx.x == 0) tell_count(p, q, PICK_NONE);
        return;
    }
    load_phase_totals(p.fin.ctl, dT, zeroT);
    const uint32_t n = (uint32_t)p.fin.ctl->sel_count_all[q];      // <= TOPK_PICK_MAX by the plan
    const ull* sel = p.sel + (size_t)q * TOPK_PICK_MAX * 4;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        s_hi[i] = sel[4 * i];
        s_lo[i] = sel[4 * i + 1];
        s_key[i] = sel[4 * i + 2];
        s_at[i] = (uint32_t)sel[4 * i + 3];
    }
    __syncthreads();
    auto before = [&](uint32_t a, uint32_t b) {
        if (s_hi[a] != s_hi[b]) return s_hi[a] > s_hi[b];
        if (s_lo[a] != s_lo[b]) return s_lo[a] > s_lo[b];
        return s_key[a] < s_key[b];
    };
    auto emit = [&](uint32_t row, uint32_t i) {
        const SlotView v = load_slot(p.fin.t, s_at[i]);
        tell_row(p, q, row, make_entry(v, dT, zeroT, p.fin));
    };
    __shared__ RankBins s_bins;
    rank_candidates<RANK_THREADS>(s_bins, n, p.k, [&](uint32_t a) { return fine_digit(s_lo[a], s_hi[a]); }, before, [&](uint32_t a, uint32_t b) {
        exchange(s_hi[a], s_hi[b]);
        exchange(s_lo[a], s_lo[b]);
        exchange(s_key[a], s_key[b]);
        exchange(s_at[a], s_at[b]);
    }, emit);
    __syncthreads();
    if (threadIdx.x == 0) {
        p.fin.ctl->sel_count_all[q] = 0;   // (for the next request)
        tell_count(p, q, min(n, p.k));
    }
}

// ---- top-k, the long way ------------------------------------------------------------------
// For k above TOPK_PICK_K, and where more than TOPK_PICK_MAX keys share the first digit of the k-th.
// A most-significant-digit radix select narrows the table down to little more than the k best keys, which a CTA per
// phase sorts.  The first digit is the logarithmic one that the totals pass has counted already; where too many keys
// share it, 12-bit digits of the rest follow, one pass over the table each, for all phases at once.  Every phase
// that a request of this k would take this way is selected and sorted with the first one asked for: the
// table is read once or twice instead of twice per phase (16 M keys, k = 1 500: two phases 1 483 -> 375 us, eight 4 844 ->
// 562).  Sorting twice as many items costs more than a further pass, so digits are added until the items'
// padded number is that of k alone.
//
// Ranking composite, larger = better: bits 56..143 hold the 88-bit weighted time, bits 0..55
// the complemented key (so the smaller key wins a tie).  Unique per key.
struct Composite {
    ull c[3];  // c[2] = bits 128..143
};

__device__ __forceinline__ Composite composite_of(ull key, ull lo, ull hi) {
    Composite x;
    x.c[0] = ((~key) & 0x00FFFFFFFFFFFFFFull) | (lo << 56);
    x.c[1] = (lo >> 8) | (hi << 56);
    x.c[2] = hi >> 8;
    return x;
}

// Leading bits of the composite that keys of one first digit share: all above the weighted time's bit length e, and
// six from there on.
__device__ __forceinline__ int shared_bits(uint32_t first) { return 94 - max((int)(first >> 5), 6); }

// Digit d (most significant first) of the composite shifted left by `shift` bits.
__device__ __forceinline__ uint32_t digit_of(const Composite& x, int d, int shift) {
    int off = 144 - 12 * (d + 1) - shift;
    if (off < 0) return (uint32_t)(x.c[0] << (-off)) & 0xFFFu;  // last, partial digit
    int wi = off >> 6, sh = off & 63;
    ull v = x.c[wi] >> sh;
    if (sh > 52 && wi < 2) v |= x.c[wi + 1] << (64 - sh);
    return (uint32_t)v & 0xFFFu;
}

// A key of phase q against the digits known so far -- -1: below, 0: equal on all of them, +1: above
__device__ __forceinline__ int compare_known(const TopkAllParams& p, uint32_t q, ull key, ull lo, ull hi, Composite& x) {
    const uint32_t first = topk_first_digit(lo, hi);
    if (first != p.first[q]) return first > p.first[q] ? 1 : -1;
    x = composite_of(key, lo, hi);
    const int shift = shared_bits(first);
    for (uint32_t d = 0; d < p.n_digits[q]; ++d) {
        const uint32_t a = digit_of(x, (int)d, shift), b = p.digit[q][d];
        if (a != b) return a > b ? 1 : -1;
    }
    return 0;
}

// f(phase, key, lo, hi, slot) for every live slot of an active phase, four slots per thread in flight
template <typename F>
__device__ __forceinline__ void each_active(const TopkAllParams& p, F f) {
    constexpr int ILP = 4;
    const ull stride = (ull)gridDim.x * blockDim.x;
    for (ull i0 = (ull)blockIdx.x * blockDim.x + threadIdx.x; i0 < p.n_slots; i0 += stride * ILP) {
        ull sk[ILP];
        ulonglong2 x[ILP];
#pragma unroll
        for (int u = 0; u < ILP; ++u) sk[u] = i0 + u * stride < p.n_slots ? p.t.keys[i0 + u * stride] : 0ull;
#pragma unroll
        for (int u = 0; u < ILP; ++u) {
            x[u] = i0 + u * stride < p.n_slots ? p.t.vals[i0 + u * stride] : make_ulonglong2(0, 0);  // no wait for the keys
        }
#pragma unroll
        for (int u = 0; u < ILP; ++u) {
            const uint32_t q = (uint32_t)(~sk[u] >> 48) & (ATREX_MAX_PHASES - 1);
            if (sk[u] != 0 && ((p.active_mask >> q) & 1u)) f(q, ~sk[u], x[u].x, x[u].y >> HI_SHIFT, i0 + u * stride);
        }
    }
}

// Counts of the next digit of the active phases' keys that are level with the known ones (shared memory: a row each).
constexpr int TOPK_HIST_THREADS = 1024;
__global__ void __launch_bounds__(TOPK_HIST_THREADS) topk_hist_kernel(const __grid_constant__ TopkAllParams p) {
    extern __shared__ uint32_t s_hist[];
    const uint32_t rows = __popc(p.active_mask);
    for (uint32_t i = threadIdx.x; i < rows * TOPK_BINS; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
    each_active(p, [&](uint32_t q, ull key, ull lo, ull hi, ull) {
        Composite x;
        if (compare_known(p, q, key, lo, hi, x) == 0) atomicAdd(&s_hist[p.row[q] * TOPK_BINS + digit_of(x, (int)p.n_digits[q], shared_bits(p.first[q]))], 1u);
    });
    __syncthreads();
    for (uint32_t q = 0; q < ATREX_MAX_PHASES; ++q) {
        if (!((p.active_mask >> q) & 1u)) continue;
        for (uint32_t i = threadIdx.x; i < TOPK_BINS; i += blockDim.x) {
            const uint32_t c = s_hist[p.row[q] * TOPK_BINS + i];
            if (c) atomicAdd(&p.hist[(size_t)q * TOPK_BINS + i], c);
        }
    }
}

// The digit of each active phase's wanted key (a CTA per phase, four bins to a thread, the highest first), told to the host.
__global__ void __launch_bounds__(TOPK_BINS / 4) topk_digit_kernel(const __grid_constant__ TopkDigitParams p) {
    __shared__ uint32_t s_warp[32];
    const uint32_t q = blockIdx.x, t = threadIdx.x, lane = t & 31u, w = t >> 5, need = p.need[q];
    grid_dependency_wait();
    if (!((p.active_mask >> q) & 1u)) return;
    const uint4 v = reinterpret_cast<const uint4*>(p.hist + (size_t)q * TOPK_BINS)[TOPK_BINS / 4 - 1 - t];
    const uint32_t own = v.x + v.y + v.z + v.w;
    uint32_t incl = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        uint32_t c = s_warp[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, c, d);
            if (lane >= (uint32_t)d) c += o;
        }
        s_warp[lane] = c;
    }
    __syncthreads();
    if (w) incl += s_warp[w - 1];
    uint32_t above = incl - own;
    if (above >= need || incl < need) return;          // (exactly one thread goes on)
    uint32_t bin = TOPK_BINS - 1 - 4 * t, in_bin = v.w;
    if (above + in_bin < need) { above += in_bin; --bin; in_bin = v.z; }
    if (above + in_bin < need) { above += in_bin; --bin; in_bin = v.y; }
    if (above + in_bin < need) { above += in_bin; --bin; in_bin = v.x; }
    volatile TopkDigit* a = p.answers + q;
    a->bin = bin;
    a->above = above;
    a->in_bin = in_bin;
    __threadfence_system();
    a->seq = p.seq;                                    // the host waits for this word
}

// Candidates of all active phases in one pass, each into its own selection region.
__global__ void __launch_bounds__(FIN_THREADS) topk_collect_all_kernel(const __grid_constant__ TopkAllParams p) {
    each_active(p, [&](uint32_t q, ull key, ull lo, ull hi, ull slot) {
        Composite x;
        if (!((p.collect_all_mask >> q) & 1u) && compare_known(p, q, key, lo, hi, x) < 0) return;
        x = composite_of(key, lo, hi);
        const ull pos = atomicAdd(&p.sel_count[q], 1ull);
        if (pos < p.sel_cap) {
            ull* dst = p.sel + ((ull)q * p.sel_cap + pos) * 4;
            dst[0] = x.c[2]; dst[1] = x.c[1]; dst[2] = x.c[0]; dst[3] = slot;
        }
    });
}

__device__ __forceinline__ bool sel_less(const ull* a, const ull* b) {
    if (a[0] != b[0]) return a[0] < b[0];
    if (a[1] != b[1]) return a[1] < b[1];
    return a[2] < b[2];
}

// Bitonic sort, descending by composite, of each phase's n (power of two) 32-byte items in global memory,
// by a CTA per phase.  Padding items are all-zero and sink to the end.
__global__ void __launch_bounds__(1024) topk_sort_kernel(const __grid_constant__ TopkSortParams p) {
    const uint32_t n = p.n_pow2[blockIdx.x];
    ull* sel = p.sel + (size_t)blockIdx.x * p.sel_cap * 4;
    for (uint32_t k = 2; k <= n; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
                uint32_t l = i ^ j;
                if (l > i) {
                    ull* a = sel + (ull)i * 4;
                    ull* b = sel + (ull)l * 4;
                    bool descending = (i & k) == 0;
                    bool swap = descending ? sel_less(a, b) : sel_less(b, a);
                    if (swap) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            ull t = a[q]; a[q] = b[q]; b[q] = t;
                        }
                    }
                }
            }
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(FIN_THREADS) topk_emit_kernel(FinalizeParams p, const ull* sel, uint32_t n) {
    __shared__ double dT[ATREX_MAX_PHASES];
    __shared__ bool zeroT[ATREX_MAX_PHASES];
    load_phase_totals(p.ctl, dT, zeroT);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        SlotView v = load_slot(p.t, sel[(ull)i * 4 + 3]);
        store_entry(p.out + i, make_entry(v, dT, zeroT, p));
    }
}

// ---- launchers ----------------------------------------------------------------------------
constexpr size_t PICK_SMEM = (size_t)TOPK_PICK_MAX * 28;

// ---- small tables --------------------------------------------------------------------------
// Up to 65 536 slots (some 25 000 keys) one cluster of 8 or 16 CTAs, four slots to a thread, does in one launch what takes
// two above, and keeps the table in registers in between: the CTAs' sums and counts meet through distributed shared memory and
// cluster barriers, where kernels of many CTAs pay for atomics to one address, a fence and a word counted per CTA, and the
// next launch.  Latency-bound (4 001 records over 2 phases, whole build 71.8 ->
// 66.3 us; 2^20 over 4 096 keys 103.9 -> 96.3).
constexpr uint32_t SMALL_THREADS = 1024, SMALL_ILP = 4, SMALL_CTA_SLOTS = SMALL_THREADS * SMALL_ILP, SMALL_CTAS_MAX = 16;
constexpr uint32_t SMALL_PIECES = 7;                     // a phase's sums: weighted time in four pieces of 22 bits, count in two of 20, keys
constexpr uint32_t SMALL_SUMS = ATREX_MAX_PHASES * SMALL_PIECES;
constexpr size_t FINALIZE_SMALL_SMEM = SMALL_CTA_SLOTS * 24;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// (the aligned forms are for whole warps: lanes that took different ways come together first)
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote_addr(const void* p, uint32_t rank) {   // of the same variable in another CTA of the cluster
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ ull remote_u64(const ull* p, uint32_t rank) {
    ull v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(remote_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t remote_u32(const uint32_t* p, uint32_t rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote_addr(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ ull warp_sum(ull v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    return v;
}

__global__ void __launch_bounds__(SMALL_THREADS) finalize_small_kernel(const __grid_constant__ FinalizeParams p, uint32_t n_phases,
                                                                       const __grid_constant__ GivenTotals given, uint32_t* hist, uint32_t* next_hist) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ulonglong2* const q_val = reinterpret_cast<ulonglong2*>(smem_raw);              // [SMALL_CTA_SLOTS] the CTA's live slots side by side
    ull* const q_key = reinterpret_cast<ull*>(q_val + SMALL_CTA_SLOTS);
    __shared__ uint32_t s_warp[32][SMALL_SUMS], s_warp_live[32], s_live, s_base;
    __shared__ ull s_cta[SMALL_SUMS], s_all[SMALL_SUMS], s_word[CONTROL_WORDS];
    __shared__ double dT[ATREX_MAX_PHASES];
    __shared__ bool zeroT[ATREX_MAX_PHASES];
    const uint32_t t = threadIdx.x, lane = t & 31u, w = t >> 5, rank = cluster_rank(), ctas = gridDim.x;
    Control* const ctl = p.ctl;
    for (uint32_t i = t; i < 32 * SMALL_SUMS; i += SMALL_THREADS) (&s_warp[0][0])[i] = 0;
    grid_dependency_wait();
    ull sk[SMALL_ILP];
    ulonglong2 x[SMALL_ILP];
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        const uint32_t i = (rank * SMALL_ILP + u) * SMALL_THREADS + t;
        sk[u] = i < p.n_slots ? p.t.keys[i] : 0ull;
        x[u] = i < p.n_slots ? p.t.vals[i] : make_ulonglong2(0, 0);
    }
    if (rank == 0 && t < CONTROL_WORDS) s_word[t] = ld_relaxed(reinterpret_cast<const ull*>(ctl) + t);   // for the host, who is told by the first CTA
    for (uint32_t i = rank * SMALL_THREADS + t; i < n_phases * TOPK_BINS / 4; i += ctas * SMALL_THREADS)
        reinterpret_cast<uint4*>(next_hist)[i] = make_uint4(0, 0, 0, 0);
    // The live slots side by side: a table is hardly ever fuller than a half and often emptier than an eighth, and what follows
    // is a few hundred instructions a warp.
    uint32_t live = 0, at[SMALL_ILP];
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        const uint32_t votes = __ballot_sync(0xFFFFFFFFu, sk[u] != 0);
        at[u] = live + __popc(votes & ((1u << lane) - 1u));
        live += __popc(votes);
    }
    if (lane == 0) s_warp_live[w] = live;
    __syncthreads();
    uint32_t incl = s_warp_live[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    const uint32_t n_live = __shfl_sync(0xFFFFFFFFu, incl, 31), mine = __shfl_sync(0xFFFFFFFFu, incl, w) - live;
    if (t == 0) s_live = n_live;
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        if (sk[u] == 0) continue;
        q_key[mine + at[u]] = ~sk[u];
        q_val[mine + at[u]] = x[u];
    }
    __syncthreads();
    double roofline[SMALL_ILP];
    if (w * 32 < n_live) {
        bool beyond = false;            // (a merged entry of a phase that records of this handle cannot have)
#pragma unroll
        for (uint32_t u = 0; u < SMALL_ILP; ++u) {
            const uint32_t j = u * SMALL_THREADS + t;
            if (j >= n_live) continue;
            const uint32_t q = (uint32_t)(q_key[j] >> 48) & (ATREX_MAX_PHASES - 1);
            if (q < n_phases) atomicAdd(&hist[q * TOPK_BINS + topk_first_digit(q_val[j].x, q_val[j].y >> HI_SHIFT)], 1u);
            else beyond = true;
        }
        const uint32_t phases = __any_sync(0xFFFFFFFFu, beyond) ? ATREX_MAX_PHASES : n_phases;
        for (uint32_t q = 0; q < phases; ++q) {
            uint32_t c[SMALL_PIECES] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll
            for (uint32_t u = 0; u < SMALL_ILP; ++u) {
                const uint32_t j = u * SMALL_THREADS + t;
                if (j >= n_live || ((uint32_t)(q_key[j] >> 48) & (ATREX_MAX_PHASES - 1)) != q) continue;
                const ull lo = q_val[j].x, hi = q_val[j].y >> HI_SHIFT, n = q_val[j].y & COUNT_MASK;
                c[0] += (uint32_t)lo & 0x3FFFFFu;
                c[1] += (uint32_t)(lo >> 22) & 0x3FFFFFu;
                c[2] += (uint32_t)(lo >> 44) | ((uint32_t)hi & 3u) << 20;
                c[3] += (uint32_t)(hi >> 2);
                c[4] += (uint32_t)n & 0xFFFFFu;
                c[5] += (uint32_t)(n >> 20);
                c[6] += 1;
            }
            __syncwarp();
#pragma unroll
            for (uint32_t j = 0; j < SMALL_PIECES; ++j) {
                const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, c[j]);       // (128 slots: below 2^29)
                if (lane == j) s_warp[w][q * SMALL_PIECES + j] = sum;
            }
        }
    }
    __syncthreads();
    for (uint32_t i = w; i < SMALL_SUMS; i += SMALL_THREADS / 32) {
        const ull sum = warp_sum(s_warp[lane][i]);
        if (lane == 0) s_cta[i] = sum;
    }
    __syncthreads();
    cluster_arrive();
    // (the roofline times need no totals: their look-ups overlap the barrier)
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        const uint32_t j = u * SMALL_THREADS + t;
        roofline[u] = j < n_live ? roofline_time(p.work, p.peaks, q_key[j]) : 0.0;
    }
    cluster_wait();
    for (uint32_t i = w; i <= SMALL_SUMS; i += SMALL_THREADS / 32) {
        if (i < SMALL_SUMS) {
            const ull sum = warp_sum(lane < ctas ? remote_u64(&s_cta[i], lane) : 0ull);
            if (lane == 0) s_all[i] = sum;
        } else {
            const uint32_t n = lane < ctas ? remote_u32(&s_live, lane) : 0u;
            const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < rank ? n : 0u), all = __reduce_add_sync(0xFFFFFFFFu, n);
            if (lane == 0) {
                s_base = before;
                if (rank == 0) s_word[offsetof(Control, n_out) / 8] = ctl->n_out = all;
            }
        }
    }
    __syncthreads();
    if (t < ATREX_MAX_PHASES) {
        const ull* c = s_all + t * SMALL_PIECES;
        ull lo = c[0], hi = c[3] << 2;
        const ull add[2] = {c[1] << 22, c[2] << 44};
        hi += (c[1] >> 42) + (c[2] >> 20);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            lo += add[j];
            hi += lo < add[j] ? 1ull : 0ull;
        }
        if (given.use) {
            lo = given.lo[t];
            hi = given.hi[t];
        }
        dT[t] = u128_to_f64_rn(hi, lo);
        zeroT[t] = (lo | hi) == 0;
        if (rank == 0) {
            s_word[offsetof(Control, total_lo) / 8 + t] = ctl->total_lo[t] = lo;
            s_word[offsetof(Control, total_hi) / 8 + t] = ctl->total_hi[t] = hi;
            s_word[offsetof(Control, count_per_phase) / 8 + t] = ctl->count_per_phase[t] = c[4] + (c[5] << 20);
            s_word[offsetof(Control, keys_per_phase) / 8 + t] = ctl->keys_per_phase[t] = c[6];
        }
    }
    __syncthreads();
    grid_dependents_launch();
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        const uint32_t j = u * SMALL_THREADS + t;
        const ull pos = s_base + j;
        if (j >= n_live || pos >= p.out_cap) continue;
        const ulonglong2 y = q_val[j];
        atrex_entry_t e;
        e.key = q_key[j];
        e.count = y.y & COUNT_MASK;
        e.wt_lo = y.x;
        e.wt_hi = y.y >> HI_SHIFT;
        const uint32_t q = (uint32_t)(e.key >> 48) & (ATREX_MAX_PHASES - 1);
        e.phase_weight = zeroT[q] ? 0.0 : __ddiv_rn(u128_to_f64_rn(e.wt_hi, e.wt_lo), dT[q]);
        e.roofline_s = roofline[u];
        store_entry(p.out + pos, e);
    }
    __syncthreads();
    if (t == 0) __threadfence();
    cluster_arrive();                   // (no CTA leaves while another reads its shared memory, and the host is told last)
    cluster_wait();
    if (rank == 0 && t < CONTROL_WORDS) tell(p.told + t, s_word[t], p.stamp);
}

// Top-k of every phase of a small table in one launch: every CTA finds the digits and lists its candidates in shared
// memory, CTA q gathers those of phase q and ranks them.
struct SmallPick {
    ull key[SMALL_CTA_SLOTS], lo[SMALL_CTA_SLOTS], cnthi[SMALL_CTA_SLOTS];            // this CTA's candidates
    ull g_key[TOPK_PICK_MAX], g_lo[TOPK_PICK_MAX], g_cnthi[TOPK_PICK_MAX];            // this phase's
};
__global__ void __launch_bounds__(SMALL_THREADS) topk_small_kernel(const __grid_constant__ PickParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallPick& s = *reinterpret_cast<SmallPick*>(smem_raw);
    __shared__ uint32_t s_bin[ATREX_MAX_PHASES], s_sum[4 * ATREX_MAX_PHASES], s_n, s_gathered;
    __shared__ double dT[ATREX_MAX_PHASES];
    __shared__ bool zeroT[ATREX_MAX_PHASES];
    const uint32_t t = threadIdx.x, lane = t & 31u, w = t >> 5, rank = cluster_rank(), ctas = gridDim.x;
    if (t == 0) s_n = s_gathered = 0;
    grid_dependency_wait();
    ull sk[SMALL_ILP];
    ulonglong2 x[SMALL_ILP];
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        const uint32_t i = (rank * SMALL_ILP + u) * SMALL_THREADS + t;
        sk[u] = i < p.fin.n_slots ? p.fin.t.keys[i] : 0ull;
        x[u] = i < p.fin.n_slots ? p.fin.t.vals[i] : make_ulonglong2(0, 0);
    }
    find_digits(p, s_bin, s_sum);
#pragma unroll
    for (uint32_t u = 0; u < SMALL_ILP; ++u) {
        if (sk[u] == 0) continue;
        const uint32_t q = (uint32_t)(~sk[u] >> 48) & (ATREX_MAX_PHASES - 1);
        if (topk_first_digit(x[u].x, x[u].y >> HI_SHIFT) < s_bin[q]) continue;      // (PICK_NONE: never)
        const uint32_t at = atomicAdd(&s_n, 1u);
        s.key[at] = ~sk[u];
        s.lo[at] = x[u].x;
        s.cnthi[at] = x[u].y;
    }
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    const bool ranks = rank < p.n_phases && s_bin[rank] != PICK_NONE;
    if (ranks) {
        for (uint32_t r = w; r < ctas; r += SMALL_THREADS / 32) {
            const uint32_t n = remote_u32(&s_n, r);
            for (uint32_t i = lane; i < n; i += 32) {
                const ull key = remote_u64(&s.key[i], r);
                if (((uint32_t)(key >> 48) & (ATREX_MAX_PHASES - 1)) != rank) continue;
                const uint32_t at = atomicAdd(&s_gathered, 1u);
                if (at >= TOPK_PICK_MAX) continue;                               // (cannot happen: the digits were chosen so)
                s.g_key[at] = key;
                s.g_lo[at] = remote_u64(&s.lo[i], r);
                s.g_cnthi[at] = remote_u64(&s.cnthi[i], r);
            }
        }
        load_phase_totals(p.fin.ctl, dT, zeroT);      // (a barrier of the CTA)
    }
    cluster_arrive();                 // nobody reads anybody's shared memory any more
    if (ranks) {
        const uint32_t n = min(s_gathered, TOPK_PICK_MAX);
        const auto before = [&](uint32_t a, uint32_t b) {
            const ull ha = s.g_cnthi[a] >> HI_SHIFT, hb = s.g_cnthi[b] >> HI_SHIFT;
            if (ha != hb) return ha > hb;
            if (s.g_lo[a] != s.g_lo[b]) return s.g_lo[a] > s.g_lo[b];
            return s.g_key[a] < s.g_key[b];
        };
        const auto swap = [&](uint32_t a, uint32_t b) {
            exchange(s.g_key[a], s.g_key[b]);
            exchange(s.g_lo[a], s.g_lo[b]);
            exchange(s.g_cnthi[a], s.g_cnthi[b]);
        };
        __shared__ RankBins s_bins;
        rank_candidates<SMALL_THREADS>(s_bins, n, p.k, [&](uint32_t a) { return fine_digit(s.g_lo[a], s.g_cnthi[a] >> HI_SHIFT); }, before, swap, [&](uint32_t row, uint32_t i) {
            SlotView v;
            v.key = s.g_key[i];
            v.live = true;
            v.lo = s.g_lo[i];
            v.count = s.g_cnthi[i] & COUNT_MASK;
            v.hi = s.g_cnthi[i] >> HI_SHIFT;
            tell_row(p, rank, row, make_entry(v, dT, zeroT, p.fin));
        });
    }
    __syncthreads();
    if (t == 0 && rank < p.n_phases) tell_count(p, rank, ranks ? min(min(s_gathered, TOPK_PICK_MAX), p.k) : PICK_NONE);
    cluster_wait();
}

uint32_t small_ctas(ull n_slots) { return n_slots <= 8 * SMALL_CTA_SLOTS ? 8u : 16u; }

// A launch of one cluster, set up while its predecessor on the stream is still running (see launch_chained).
struct ClusterLaunch {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t config = {};
    ClusterLaunch(uint32_t ctas, size_t smem, cudaStream_t stream) {
        config.gridDim = dim3(ctas);
        config.blockDim = dim3(SMALL_THREADS);
        config.dynamicSmemBytes = smem;
        config.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        config.attrs = attr;
        config.numAttrs = 2;
    }
    ClusterLaunch(const ClusterLaunch&) = delete;
    ClusterLaunch& operator=(const ClusterLaunch&) = delete;
};

template <typename... P, typename... A>
cudaError_t launch_cluster(void (*kernel)(P...), uint32_t ctas, size_t smem, cudaStream_t stream, const A&... args) {
    ClusterLaunch launch(ctas, smem, stream);
    return cudaLaunchKernelEx(&launch.config, kernel, P(args)...);
}
template <typename... P>
bool cluster_fits(void (*kernel)(P...), uint32_t ctas, size_t smem) {
    ClusterLaunch launch(ctas, smem, nullptr);
    int n = 0;
    const bool fits = cudaOccupancyMaxActiveClusters(&n, kernel, &launch.config) == cudaSuccess && n > 0;
    if (!fits) cudaGetLastError();
    return fits;
}

cudaError_t finalize_prepare() {
    cudaError_t e = cudaFuncSetAttribute(totals_kernel<TOT_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)totals_smem(TOT_WIDE_FROM - 1));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(totals_kernel<2 * TOT_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)totals_smem(ATREX_MAX_PHASES));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(topk_rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PICK_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(finalize_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FINALIZE_SMALL_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(finalize_small_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(topk_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallPick));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(topk_small_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(topk_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ATREX_MAX_PHASES * TOPK_BINS * 4);
    return e;
}

cudaError_t launch_totals(const TableRef& t, ull n_slots, uint32_t n_phases, const GivenTotals& given, uint32_t* hist, uint32_t* next_hist,
                          int n_sms, cudaStream_t stream) {
    const size_t smem = totals_smem(n_phases);
    const uint32_t threads = totals_threads(n_phases);
    uint32_t per_sm = (uint32_t)(233472 / (smem + 1024));
    if (per_sm > 4) per_sm = 4;
    auto* kernel = threads == TOT_THREADS ? totals_kernel<TOT_THREADS> : totals_kernel<2 * TOT_THREADS>;
    return launch_chained(kernel, grid_for_work(n_slots, threads * TOT_ILP, n_sms, per_sm), threads, smem, stream, t, n_slots,
                          n_phases, given, hist, next_hist);
}

cudaError_t launch_emit(const FinalizeParams& p, int n_sms, cudaStream_t stream) {
    static const uint32_t per_sm = resident_ctas(emit_kernel, FIN_THREADS, 0);
    return launch_chained(emit_kernel, grid_for_work(p.n_slots, FIN_THREADS * EMIT_ILP, n_sms, per_sm), FIN_THREADS, 0, stream, p);
}

cudaError_t launch_work_insert(const atrex_work_t* rows, ull n, const WorkRef& w, Control* ctl, int grid,
                               cudaStream_t stream) {
    work_insert_kernel<<<grid, 256, 0, stream>>>(rows, n, w, ctl);
    return cudaGetLastError();
}

#ifndef ATREX_SMALL_CLUSTERS
#define ATREX_SMALL_CLUSTERS 1
#endif
// Small tables go through one cluster where the process has the SMs for it in one place; a share of the GPU (some of its
// SMs only) may not, and 16 CTAs are more than every GPU promises.
bool finalize_in_one_cluster(ull n_slots) {
    if (!ATREX_SMALL_CLUSTERS || n_slots > (ull)SMALL_CTAS_MAX * SMALL_CTA_SLOTS) return false;
    return cluster_fits(finalize_small_kernel, small_ctas(n_slots), FINALIZE_SMALL_SMEM) && cluster_fits(topk_small_kernel, small_ctas(n_slots), sizeof(SmallPick));
}

cudaError_t launch_finalize_small(const FinalizeParams& p, uint32_t n_phases, const GivenTotals& given, uint32_t* hist, uint32_t* next_hist, cudaStream_t stream) {
    return launch_cluster(finalize_small_kernel, small_ctas(p.n_slots), FINALIZE_SMALL_SMEM, stream, p, n_phases, given, hist, next_hist);
}

cudaError_t launch_topk_pick(const PickParams& p, bool one_cluster, int n_sms, cudaStream_t stream) {
    if (one_cluster) return launch_cluster(topk_small_kernel, small_ctas(p.fin.n_slots), sizeof(SmallPick), stream, p);
    static const uint32_t per_sm = resident_ctas(topk_collect_kernel, FIN_THREADS, 0);
    cudaError_t e = launch_chained(topk_collect_kernel, grid_for_work(p.fin.n_slots, FIN_THREADS * 4, n_sms, per_sm), FIN_THREADS, 0, stream, p);
    if (e == cudaSuccess) e = launch_chained(topk_rank_kernel, p.n_phases, RANK_THREADS, PICK_SMEM, stream, p);
    return e;
}

cudaError_t launch_topk_collect_all(const TopkAllParams& p, int grid, cudaStream_t stream) {
    topk_collect_all_kernel<<<grid, FIN_THREADS, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_topk_hist(const TopkAllParams& p, int n_sms, cudaStream_t stream) {
    const uint32_t rows = (uint32_t)__builtin_popcount(p.active_mask), per_sm = rows <= 6 ? 2 : 1;
    topk_hist_kernel<<<grid_for_work(p.n_slots, TOPK_HIST_THREADS * 4, n_sms, per_sm), TOPK_HIST_THREADS, rows * TOPK_BINS * 4, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_topk_digit(const TopkDigitParams& p, uint32_t n_phases, cudaStream_t stream) {
    return launch_chained(topk_digit_kernel, n_phases, TOPK_BINS / 4, 0, stream, p);
}

cudaError_t launch_topk_sort(const TopkSortParams& p, uint32_t n_phases, cudaStream_t stream) {
    topk_sort_kernel<<<n_phases, 1024, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_topk_emit(const FinalizeParams& p, const ull* sel, uint32_t n, cudaStream_t stream) {
    int grid = (int)((n + FIN_THREADS - 1) / FIN_THREADS);
    if (grid < 1) grid = 1;
    topk_emit_kernel<<<grid, FIN_THREADS, 0, stream>>>(p, sel, n);
    return cudaGetLastError();
}

}  // namespace atrex
