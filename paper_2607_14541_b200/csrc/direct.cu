// Ingest of small calls (Eq. 2's group-by sum): records straight into the key table in one launch.
//
// The two-pass route (scatter.cu, ingest.cu) pays per call: a kernel that sets up 230 KB of shared memory
// per SM, a launch that asks whether the buffers need draining, a directory built from a sample, and at the
// end a pass over every partition of the table.  Below about a million records those fixed costs (8 us for
// the smallest call, 170 us for a first call of 2^20 records, 0.4 ms for draining a 16 M-key table) are
// larger than adding the records to the table with global atomics, 44 G records/s into a table that L2
// holds and about 7 G records/s into one that it does not.
//   direct_records_kernel  up to 8 192 records: a thread each; lanes that hold the key of the warp's first
//                          lane are combined.  Bound by the latency of one record's chain (record, slot,
//                          two atomics).
//   direct_shared_kernel   more: each CTA first sums its share of the records per key in a shared-memory
//                          table, so that a frequent key costs one global update per CTA; keys that find no
//                          slot there go to the table at once.  Bound by the L2's atomic rate and the probes'
//                          divergence (2^20 records over 4 096 keys: 35 us).
#include "atrex_dev.cuh"
#include "kernels.h"

namespace atrex {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int RECORDS_THREADS = 128;
constexpr int SHARED_THREADS = 1024;
constexpr uint32_t SHARED_SLOTS_MAX = 8192;   // 20 B each: one CTA per SM
constexpr uint32_t SHARED_PROBES = 8;

struct Record {
    ull key;
    uint32_t h;
    ull prod;
    bool valid;
};

__device__ __forceinline__ Record decode(const DirectParams& p, uint4 v, bool present) {
    Record r;
    const uint32_t khi = v.y & 0x00FFFFFFu;
    r.valid = present && v.x < p.n_apps && khi < p.phase_lim;
    const uint32_t wgt = __ldg(p.app_w + (r.valid ? v.x : 0u));
    r.prod = (ull)wgt * (ull)v.w;
    r.key = ((ull)khi << 32) | v.z;
    r.h = hash32(khi & 0xFFFFu, v.z);
    return r;
}

__device__ __forceinline__ void count_rejected(const DirectParams& p, bool rejected) {
    const uint32_t votes = __ballot_sync(FULL, rejected);
    if (votes != 0 && (threadIdx.x & 31u) == (uint32_t)(__ffs(votes) - 1)) atomicAdd(&p.t.ctl->n_rejected, (ull)__popc(votes));
}

// The lanes that hold the key of the first valid lane are combined into it (a frequent key would otherwise
// queue at one address); the others keep their record.  Sums: (count, lo, hi) of this lane, count 0 = nothing left to do.
__device__ __forceinline__ uint32_t combine_first(const Record& r, ull& lo, ull& hi) {
    lo = r.prod;
    hi = 0;
    const uint32_t valid = __ballot_sync(FULL, r.valid);
    if (valid == 0) return 0;
    const int lead = __ffs(valid) - 1;
    const ull first = __shfl_sync(FULL, r.key, lead);
    const uint32_t same = __ballot_sync(FULL, r.valid && r.key == first);
    if ((same & (same - 1)) == 0 || !((same >> (threadIdx.x & 31u)) & 1u)) return r.valid ? 1u : 0u;
    // 64-bit products in four 16-bit pieces, each sum below 2^21
    const ull s0 = __reduce_add_sync(same, (uint32_t)(r.prod & 0xFFFFu)), s1 = __reduce_add_sync(same, (uint32_t)(r.prod >> 16) & 0xFFFFu);
    const ull s2 = __reduce_add_sync(same, (uint32_t)(r.prod >> 32) & 0xFFFFu), s3 = __reduce_add_sync(same, (uint32_t)(r.prod >> 48));
    if ((threadIdx.x & 31u) != (uint32_t)lead) return 0;
    const ull low = s0 + (s1 << 16) + (s2 << 32), add = s3 << 48;    // low < 2^54
    lo = low + add;
    hi = (s3 >> 16) + (lo < low ? 1ull : 0ull);
    return (uint32_t)__popc(same);
}

__global__ void __launch_bounds__(RECORDS_THREADS) direct_records_kernel(DirectParams p) {
    const uint32_t i = blockIdx.x * RECORDS_THREADS + threadIdx.x;
    const bool present = i < p.n;
    // (a prefetch into L2, where every write arrives, may come before the predecessor's writes are waited for)
    if (present && (threadIdx.x & 7u) == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.recs + i));
    grid_dependents_launch();   // (its successor does the same before it waits)
    grid_dependency_wait();
    const uint4 v = present ? __ldcs(p.recs + i) : make_uint4(0, 0, 0, 0);
    const Record r = decode(p, v, present);
    count_rejected(p, present && !r.valid);
    ull lo, hi;
    const uint32_t count = combine_first(r, lo, hi);
    if (count) table_accumulate(p.t, r.key, r.h, lo, hi, count);
}

// Four slots of the shared table to the key table at once: their key look-ups, then their returning adds,
// are in flight together.  (The counts added without waiting for the low words' answers, the rare carries by adds of
// their own: 2^20 records over 4 096 keys 5 us slower.)
__device__ __forceinline__ void flush_slots(const TableRef& t, const ull (&key)[4], const uint32_t (&h)[4], const ull (&v)[4],
                                            const uint32_t (&count)[4]) {
    ull idx[4], found[4], old[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        idx[u] = (ull)part_of(h[u], t.lp) * t.C + first_pair(window_of(h[u], t.lp), (uint32_t)(key[u] >> 48), t.C);
        found[u] = count[u] ? ld_relaxed(t.keys + ATREX_INDEX(idx[u], (ull)t.C << t.lp, t.ctl)) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (count[u] == 0 || found[u] == ~key[u]) continue;
        idx[u] = find_or_claim(t, key[u], h[u]);
        if (idx[u] == NO_INDEX) {
            atomicOr(&t.ctl->status, ST_TABLE_FULL);
            atomicAdd(&t.ctl->n_dropped, (ull)count[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (count[u] && idx[u] != NO_INDEX) old[u] = atomicAdd(reinterpret_cast<ull*>(t.vals + ATREX_INDEX(idx[u], (ull)t.C << t.lp, t.ctl)), v[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (count[u] && idx[u] != NO_INDEX)
            atomicAdd(reinterpret_cast<ull*>(t.vals + ATREX_INDEX(idx[u], (ull)t.C << t.lp, t.ctl)) + 1,
                      (ull)count[u] + ((old[u] + v[u] < old[u] ? 1ull : 0ull) << HI_SHIFT));
}

__global__ void __launch_bounds__(SHARED_THREADS) direct_shared_kernel(DirectParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t S = p.slots;                                            // a power of two
    ull* s_key = reinterpret_cast<ull*>(smem_raw);                         // key with bit 63 set, 0 = empty
    uint32_t* s_lo = reinterpret_cast<uint32_t*>(s_key + S);
    uint32_t* s_hi = s_lo + S;
    uint32_t* s_cnt = s_hi + S;
    for (uint32_t i = threadIdx.x; i < S * 5u / 4u; i += SHARED_THREADS) reinterpret_cast<uint4*>(smem_raw)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    grid_dependency_wait();
    // CTA b takes records [b * share, (b + 1) * share): at most 2^15, so that the high limb (product < 2^48,
    // a carry per record) stays below 2^32
    const uint32_t first = blockIdx.x * p.share, end = min(p.n, first + p.share);
    const uint32_t rounds = (end - first + SHARED_THREADS - 1) / SHARED_THREADS;
    uint4 next = make_uint4(0, 0, 0, 0);
    if (first + threadIdx.x < end) next = __ldcs(p.recs + first + threadIdx.x);
    for (uint32_t k = 0; k < rounds; ++k) {
        const uint32_t i = first + k * SHARED_THREADS + threadIdx.x;
        const bool present = i < end;
        const uint4 v = next;
        if (i + SHARED_THREADS < end) next = __ldcs(p.recs + i + SHARED_THREADS);
        const Record r = decode(p, v, present);
        count_rejected(p, present && !r.valid);
        ull lo, hi;
        const uint32_t count = combine_first(r, lo, hi);
        if (count == 0) continue;
        bool done = false;
        if (hi == 0 && (lo >> 48) < count) {   // (every record below 2^48, or as good as)
            const ull skey = r.key | (1ull << 63);
            uint32_t s = ((r.h ^ ((uint32_t)(r.key >> 48) * 0x9E3779B9u)) * 0xC2B2AE35u) >> 16 & (S - 1);
            for (uint32_t probe = 0; probe < SHARED_PROBES; ++probe) {
                ull at = *reinterpret_cast<volatile ull*>(s_key + s);
                if (at == 0) at = atomicCAS(s_key + s, 0ull, skey);
                if (at == 0 || at == skey) {
                    const uint32_t v0 = (uint32_t)lo, o = atomicAdd(s_lo + s, v0);
                    const uint32_t x = (uint32_t)(lo >> 32) + (o + v0 < o ? 1u : 0u);
                    if (x) atomicAdd(s_hi + s, x);
                    atomicAdd(s_cnt + s, count);
                    done = true;
                    break;
                }
                s = (s + 1) & (S - 1);
            }
        }
        if (!done) table_accumulate(p.t, r.key, r.h, lo, hi, count);
    }
    grid_dependents_launch();
    __syncthreads();
    uint32_t held = 0;
    const uint32_t turn = (uint32_t)((ull)S * blockIdx.x / gridDim.x);   // (the CTAs hold the same keys at the same places: they start apart)
    for (uint32_t i0 = threadIdx.x; i0 < S; i0 += 4 * SHARED_THREADS) {
        ull key[4], v[4];
        uint32_t h[4], count[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = i0 + u * SHARED_THREADS < S;
            const uint32_t i = (i0 + u * SHARED_THREADS + turn) & (S - 1);
            key[u] = (in ? s_key[i] : 0ull) & ~(1ull << 63);
            count[u] = in ? s_cnt[i] : 0u;
            v[u] = in ? (ull)s_lo[i] | ((ull)s_hi[i] << 32) : 0ull;
            h[u] = hash32(key[u]);
            held += count[u] ? 1u : 0u;
        }
        flush_slots(p.t, key, h, v, count);
    }
    held = __reduce_add_sync(FULL, held);
    if ((threadIdx.x & 31u) == 0 && held) atomicMax(&p.t.ctl->hot_n, (ull)held);
}

}  // namespace

cudaError_t direct_prepare() {
    return cudaFuncSetAttribute(direct_shared_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(SHARED_SLOTS_MAX * 20u));
}

cudaError_t launch_direct(DirectParams p, int n_sms, cudaStream_t stream) {
    if (p.n <= DIRECT_RECORDS_MAX)
        return launch_chained(direct_records_kernel, (p.n + RECORDS_THREADS - 1) / RECORDS_THREADS, RECORDS_THREADS, 0, stream, p);
    // at least one round of records per CTA, at most one CTA per SM; a slot table twice the CTA's records
    uint32_t grid = (p.n + SHARED_THREADS - 1) / SHARED_THREADS;
    if (grid > (uint32_t)n_sms) grid = (uint32_t)n_sms;
    p.share = (p.n + grid - 1) / grid;
    grid = (p.n + p.share - 1) / p.share;
    p.slots = 1024;
    while (p.slots < 2 * p.share && p.slots < SHARED_SLOTS_MAX) p.slots <<= 1;
    return launch_chained(direct_shared_kernel, grid, SHARED_THREADS, p.slots * 20u, stream, p);
}

}  // namespace atrex
