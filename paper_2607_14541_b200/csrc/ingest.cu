// Ingest, everything but the scatter pass (scatter.cu): Eq. 2's group-by sum, streamed, as a
// two-pass radix-partitioned aggregation.
//
// Random read-modify-write into a table far larger than L2 is bound by DRAM latency and by
// the L2's atomic rate, not by bandwidth, so the hot path avoids global atomics altogether:
//
// Pass 1  SCATTER  (scatter.cu) accumulates the records of hot keys in a shared-memory directory
//   and appends every other record as an entry of 8 or 12 bytes to the CTA's private buffer of the key's
//   partition.
//
// Pass 2  PARTITION  (persistent CTAs, one partition at a time each).  Runs lazily: only when a
//   buffer is filling up, or when results are about to be read.  The CTA copies its
//   partition's keys from HBM into shared memory, streams the partition's entries from all
//   scatter CTAs, finds or claims each key's slot in shared memory and accumulates there, then
//   adds the per-slot deltas back to the HBM table with coalesced read-modify-writes.  The CTA
//   is the only writer of its partition, so no global atomics are involved.
//
// All sums are integers, so the result does not depend on which route a record took, on
// scheduling, or on chunking.  Entries that do not fit a spill buffer, directory wraps and
// merges fall back to exact atomic updates of the HBM table.
#include <type_traits>

#include "atrex_dev.cuh"
#include "kernels.h"

namespace atrex {

constexpr int INGEST_THREADS = 1024;
constexpr uint32_t NEW_KEY_FLAG = 0x80000000u;     // partition pass: slot claimed in this launch

__device__ __forceinline__ uint32_t dir_bucket_of_key(ull key, uint32_t mult, uint32_t n_buckets) {
    return dir_bucket(hash32(key), (uint32_t)(key >> 48), mult, n_buckets);
}
__constant__ uint32_t DIR_MULTS[4] = {0xC2B2AE35u, 0x27D4EB2Fu, 0x165667B1u, 0x9E3779B9u};

// Shared memory is addressed explicitly through 32-bit shared-window addresses in the hot
// loops: one integer add per access instead of generic 64-bit pointer arithmetic.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint2 lds_v2u32(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t atoms_add(uint32_t a, uint32_t v) {
    uint32_t o;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ void reds_add(uint32_t a, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void reds_or(uint32_t a, uint32_t v) {
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atoms_exch(uint32_t a, uint32_t v) {
    uint32_t o;
    asm volatile("atom.shared.exch.b32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ uint32_t atoms_cas32(uint32_t a, uint32_t expected, uint32_t desired) {
    uint32_t o;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(o) : "r"(a), "r"(expected), "r"(desired) : "memory");
    return o;
}
__device__ __forceinline__ ull atoms_cas64(uint32_t a, ull expected, ull desired) {
    ull o;
    asm volatile("atom.shared.cas.b64 %0, [%1], %2, %3;" : "=l"(o) : "r"(a), "l"(expected), "l"(desired) : "memory");
    return o;
}

// Shared-memory accumulation uses native 32-bit atomics only (64-bit shared atomics are
// compare-and-swap loops).  A slot's weighted time is kept in two limbs: the returning add on
// the low limb tells the adder whether it wrapped, and the adder then adds the carry, with the
// value's high word, to the high limb (part_accumulate).  One add raises the high limb by at most 2^16, or 2^23 for a
// warp's combined 128 entries of < 2^48 each, so the adder that takes it across 2^30 drains both
// limbs; the adds that can slip in before its exchange (one per thread of the CTA, at most one of them
// per warp combined) stay below 2^31, so the high limb never wraps.
constexpr uint32_t DRAIN_BIT = 0x40000000u;

__device__ __forceinline__ ull limbs_drain(uint32_t a0, uint32_t a1, ull* hi_out) {
    // the two exchanges need not be simultaneous: whatever lands between them stays in the
    // limbs for the next drain or the final flush
    const ull lo = atoms_exch(a0, 0u);
    const ull hi = atoms_exch(a1, 0u);
    const ull v = lo + (hi << 32);
    *hi_out = v < lo ? 1ull : 0ull;
    return v;
}

// Adds every CTA's directory image row into the table (the next launch starts the rows afresh).  A CTA handles 32
// directory slots: warp w sums rows w, w + 16, ... of those slots (exact: 128-bit sum, count), the
// sixteen partial sums meet in shared memory and warp 0 does one table update per slot.
constexpr int FOLD_WARPS = 16;

__global__ void __launch_bounds__(FOLD_WARPS * 32) hot_fold_kernel(const ull* hot_keys, const ulonglong2* hot_img,
                                                                   uint32_t n_groups, uint32_t hot_slots, TableRef t) {
    __shared__ ull s_lo[FOLD_WARPS][32], s_hi[FOLD_WARPS][32], s_cnt[FOLD_WARPS][32];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    const uint32_t i = blockIdx.x * 32u + lane;
    ull lo = 0, hi = 0, count = 0;
    if (i < hot_slots) {
        constexpr uint32_t ILP = 5;     // rows in flight per lane
        for (uint32_t g0 = w; g0 < n_groups; g0 += ILP * FOLD_WARPS) {
            ulonglong2 v[ILP];
#pragma unroll
            for (uint32_t u = 0; u < ILP; ++u) {
                const uint32_t g = g0 + u * FOLD_WARPS;
                v[u] = g < n_groups ? hot_img[(size_t)g * hot_slots + i] : make_ulonglong2(0, 0);
            }
#pragma unroll
            for (uint32_t u = 0; u < ILP; ++u) {
                if ((v[u].x | v[u].y) == 0) continue;
                const ull s = lo + v[u].x;
                hi += (v[u].y >> HI_SHIFT) + (s < lo ? 1ull : 0ull);
                lo = s;
                count += v[u].y & COUNT_MASK;
            }
        }
    }
    s_lo[w][lane] = lo;
    s_hi[w][lane] = hi;
    s_cnt[w][lane] = count;
    __syncthreads();
    if (w == 0 && i < hot_slots) {
#pragma unroll
        for (int k = 1; k < FOLD_WARPS; ++k) {
            const ull s = lo + s_lo[k][lane];
            hi += s_hi[k][lane] + (s < lo ? 1ull : 0ull);
            lo = s;
            count += s_cnt[k][lane];
        }
        if ((lo | hi | count) != 0) {
            const ull key = ~hot_keys[i];
            table_accumulate(t, key, hash32(key), lo, hi, count);
        }
    }
}

// --------------------------------------------------------------------------------------
// Pass 2: a CTA aggregates one partition at a time entirely in shared memory.  CTAs are
// persistent; each begins with partition blockIdx.x and draws its further ones from a counter, early enough that
// their keys and first entries are pulled into L2 during the write-back.  Per partition: copy the
// keys in, each in the form that the entries carry it in (FormKey below: 32 or 64 bits, unique inside a
// partition); stream the entries of all scatter CTAs, four per lane,
// and settle each with one look at the first pair of its probe sequence (hit, or a new key with room
// there); entries that need more than that wait in the warp's segment of a per-CTA queue in global
// memory and are settled, 32 per round, once the warp's share of the stream is through (or earlier,
// when the segment could not take another batch); then write the deltas back.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Shared-window addresses of the partition pass's arrays: keys[C] (in the form of the entries, 0 = empty; ull, or
// u32 where entries are tight), acc {u32 low limb, u32 count | NEW_KEY_FLAG}[C], a1 u32[C] (high limb).
struct PartSmem {
    uint32_t keys, acc, a1;
    uint32_t weights;          // short entries: u32[n_apps]
};

__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint4 lds_v4u32(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// FORM_TIGHT: short entries of whose identities none has a rest.
constexpr ull FORM_TIGHT = FORM_LONG_ONLY + 1;

// The keys as the pass holds them.  Long entries: ckey_of.  Short ones: the words of an entry without its payload, bit 63
// set; tight ones the high word alone.  Keys that such an entry cannot have (operators that do not fit) are in the table
// too: they take their slots as something that no entry's key equals.
template <ull FORM>
struct FormKey {
    uint32_t hi, lo;           // tight: lo = 0
};
template <ull FORM>
constexpr uint32_t KEY_BYTES = FORM == FORM_TIGHT ? 4 : 8;
template <ull FORM>
constexpr uint32_t ENTRY_BYTES = FORM == FORM_LONG ? SPILL_ENTRY_BYTES : SHORT_ENTRY_BYTES;
template <ull FORM>
__device__ __forceinline__ FormKey<FORM> form_key(const PartitionParams& q, ull key) {
    if (FORM == FORM_LONG) {
        const ull c = ckey_of_key(key);
        return {(uint32_t)(c >> 32), (uint32_t)c};
    }
    const uint32_t khi = (uint32_t)(key >> 32), op = khi & 0xFFFFu, phase = (khi >> 16) & 0xFFu, h = hash32(op, (uint32_t)key);
    if (op >= q.fmt.max_ops || phase >> q.fmt.phase_bits != 0 || (FORM == FORM_TIGHT && (op << q.fmt.phase_bits) >> (q.t.lp - 1u) != 0)) return {1u, FORM == FORM_TIGHT ? 0u : h};
    const uint32_t id = (op << q.fmt.phase_bits) | phase, in_high = (1u << (q.t.lp - 1u)) - 1u;
    return {SHORT_CONTINUATION | ((h << q.t.lp) >> 1) | (id & in_high), FORM == FORM_TIGHT ? 0u : (id >> (q.t.lp - 1u)) << q.fmt.rest_shift};
}
template <ull FORM>
__device__ __forceinline__ ull key_of_form(const PartitionParams& q, FormKey<FORM> k, uint32_t part) {
    if (FORM == FORM_LONG) return key_of_ckey(((ull)k.hi << 32) | k.lo);
    const uint32_t rest = FORM == FORM_TIGHT ? 0u : (k.lo & q.fmt.rest_mask) >> q.fmt.rest_shift;
    const uint32_t id = (k.hi & ((1u << (q.t.lp - 1u)) - 1u)) | (rest << (q.t.lp - 1u)), op = id >> q.fmt.phase_bits;
    const uint32_t h = (part << (32 - q.t.lp)) | ((k.hi << 1) >> q.t.lp);
    return pack_key(id & ((1u << q.fmt.phase_bits) - 1u), op, shape_of_hash(h, op));
}
template <ull FORM>
__device__ __forceinline__ uint32_t window_of_form(const PartitionParams& q, FormKey<FORM> k) {
    return FORM == FORM_LONG ? window_of(k.lo, q.t.lp) : (k.hi << 1) & WINDOW_MASK;
}
template <ull FORM>
__device__ __forceinline__ uint32_t phase_of_form(const PartitionParams& q, FormKey<FORM> k) {
    return FORM == FORM_LONG ? (k.hi >> 16) & 0xFFu : k.hi & ((1u << q.fmt.phase_bits) - 1u);
}

// What a look at a pair of slots (the even one at `slot`) sees.
struct PairLook {
    bool first, second;            // the key is there
    bool first_free, second_free;
};
template <ull FORM>
__device__ __forceinline__ PairLook look_at(const PartSmem& m, uint32_t slot, FormKey<FORM> k) {
    if (FORM == FORM_TIGHT) {
        const uint2 v = lds_v2u32(m.keys + slot * 4u);
        return {v.x == k.hi, v.y == k.hi, v.x == 0, v.y == 0};
    }
    const uint4 v = lds_v4u32(m.keys + slot * 8u);
    return {v.x == k.lo && v.y == k.hi, v.z == k.lo && v.w == k.hi, v.y == 0, v.w == 0};
}
// Claims a free slot.  True: the key is there now (its own claim, noted for the write-back, or another lane's).
template <ull FORM>
__device__ __forceinline__ bool claim(const PartSmem& m, uint32_t slot, FormKey<FORM> k) {
    bool mine, there;
    if (FORM == FORM_TIGHT) {
        const uint32_t old = atoms_cas32(m.keys + slot * 4u, 0u, k.hi);
        mine = old == 0;
        there = mine || old == k.hi;
    } else {
        const ull skey = ((ull)k.hi << 32) | k.lo, old = atoms_cas64(m.keys + slot * 8u, 0ull, skey);
        mine = old == 0;
        there = mine || old == skey;
    }
    if (mine) reds_or(m.acc + slot * 8u + 4u, NEW_KEY_FLAG);
    return there;
}

// General probe, one entry per lane (busy = this lane has one): walks the key's probe sequence from
// the pair at `slot`, claims the first free slot if the key is not there.  Warp-convergent.  Returns
// the key's slot, or PROBE_FAILED when the partition has no room.
constexpr uint32_t PROBE_FAILED = 0xFFFFFFFFu;

template <ull FORM>
__device__ __forceinline__ uint32_t probe_general(const PartSmem& m, FormKey<FORM> key, uint32_t slot, uint32_t advance, bool busy, uint32_t count,
                                                  uint32_t C, Control* ctl) {
    uint32_t steps = 0;
    while (__any_sync(0xFFFFFFFFu, busy)) {
        if (busy) {
            const PairLook look = look_at(m, ATREX_INDEX(slot, C - 1u, ctl), key);
            if (look.first || look.second) {
                slot += look.second ? 1u : 0u;
                busy = false;
            } else if (look.first_free || look.second_free) {
                // claim the first empty slot of the pair; a lost race re-reads the pair
                const uint32_t at = slot + (look.first_free ? 0u : 1u);
                if (claim(m, at, key)) {
                    slot = at;
                    busy = false;
                }
            } else {
                slot += advance;
                if (slot >= C) slot -= C;
            }
            if (busy && ++steps > 2 * C) {  // partition full (bounded; counts lost races too)
                busy = false;
                slot = PROBE_FAILED;
                atomicOr(&ctl->status, ST_TABLE_FULL);
                atomicAdd(&ctl->n_dropped, (ull)count);
            }
        }
    }
    return slot;
}

// A slot whose high limb filled up: its sums move to HBM (this CTA owns the slot, so those adds are
// exact; the write-back adds on top).  Rare, hence not inlined.
__device__ __noinline__ void part_drain_slot(uint32_t acc, uint32_t a1, ulonglong2* val) {
    ull hi, lo = limbs_drain(acc, a1, &hi);
    ull* vp = reinterpret_cast<ull*>(val);
    ull old = atomicAdd(vp, lo);
    hi += (old + lo < old) ? 1ull : 0ull;
    if (hi) atomicAdd(vp + 1, hi << HI_SHIFT);
}

// One entry's product (vlo + 2^32 vhi, vhi < 2^16; combined entries: 2^23) and count (0: a continuation) into its slot's limbs: a returning add on
// the low limb, whose wrap is the carry; the high limb is touched only when there is something to add.
__device__ __forceinline__ void part_accumulate(const PartSmem& m, uint32_t slot, uint32_t vlo, uint32_t vhi, uint32_t count,
                                                ulonglong2* vals_of_partition, uint32_t C, Control* ctl) {
    slot = ATREX_INDEX(slot, C, ctl);
    const uint32_t acc = m.acc + slot * 8;
    const uint32_t o0 = atoms_add(acc, vlo);
    reds_add(acc + 4, count);
    const uint32_t x = vhi + ((o0 + vlo < o0) ? 1u : 0u);
    if (x != 0) {
        const uint32_t o1 = atoms_add(m.a1 + slot * 4, x);
        if (((o1 + x) & ~o1 & DRAIN_BIT) != 0) part_drain_slot(acc, m.a1 + slot * 4, vals_of_partition + slot);
    }
}

// Where a sub-buffer's entries are.
__device__ __forceinline__ const unsigned char* entries_of(const PartitionParams& q, ull sb) {
    return q.spill + sb * q.cap * SPILL_ENTRY_BYTES;     // (a buffer of short entries takes as many bytes)
}
// The first 256 entries (24 or 16 lines) of sub-buffer `sb` towards L2, as far as it holds that many.
template <ull FORM>
__device__ __forceinline__ void prefetch_entries(const PartitionParams& q, ull sb, uint32_t lane) {
    const uint32_t bytes = q.spill_cnt[sb] * ENTRY_BYTES<FORM>;
    if (lane < 2u * ENTRY_BYTES<FORM> && lane * 128u < bytes) prefetch_l2(entries_of(q, sb) + lane * 128u);
}

// Settles a warp's queued entries, one per lane and round, by the general probe.  Other warps may
// still be streaming: the probe copes with keys that appear meanwhile.  Called once the warp's share of
// the partition's stream is through, and before a batch that might not fit the queue (a crowded
// partition of new keys).  Not inlined: it runs a few times per partition and warp.
template <ull FORM>
__device__ __noinline__ void settle_queue(const PartitionParams& q, const PartSmem m, const ulonglong2* my_queue, uint32_t qn_w, ull base, uint32_t lane);

// A queued entry: {key, product}; bit 63 of the product word says that the key's first pair was full
// of other keys when the entry was looked up, so its probe may start at the second pair; bit 62 that it is a continuation.
constexpr ull QUEUED_SKIP_FIRST = 1ull << 63, QUEUED_CONTINUATION = 1ull << 62;

// One batch of 128 entries of a sub-buffer, four consecutive ones (48 bytes; 32 if short) per lane.  FULL: the
// batch is complete (no masks).  Entry state is bit sets per lane -- `open` (present, slot not known yet), `hit`
// (slot known), `room` (the first pair of the probe sequence had a free slot when it was read).
template <ull FORM, bool CROWDED, bool FULL>
__device__ __forceinline__ void stream_batch(const PartitionParams& q, const PartSmem& m, const unsigned char* src,
                                             uint32_t part, uint32_t e0, uint32_t n_e, uint32_t C, ull base,
                                             ulonglong2* my_queue, uint32_t queue_cap_w, uint32_t& qn_w, uint32_t lane) {
    FormKey<FORM> key[4];
    uint32_t vlo[4], vhi[4], slot[4];
    uint32_t open = 0, extra = 0;    // extra: continuations
    if (FORM != FORM_LONG) {
        const ShortFormat& f = q.fmt;
        const uint32_t e = e0 + 4u * lane;
        uint32_t w[8];
        if (FULL || e < n_e) {       // (a buffer's capacity is a multiple of 16: a lane that holds any entry may read all 32 bytes)
            asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                         : "l"(src + (size_t)e * SHORT_ENTRY_BYTES));
            open = FULL ? 0xFu : (0xFu >> (4u - min(n_e - e, 4u)));
            // (what lies behind the last entry may be anything: no application is to be read from it)
#pragma unroll
            for (int u = 1; u < 4; ++u)
                if (!FULL && (open & (1u << u)) == 0) w[2 * u] = 0;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t lo = w[2 * u], hi = w[2 * u + 1];
            key[u].hi = hi | SHORT_CONTINUATION;
            key[u].lo = FORM == FORM_TIGHT ? 0u : lo & f.rest_mask;
            const uint32_t more = hi >> 31;
            const uint32_t dur = (lo & f.dur_mask()) << (more ? f.dur_bits : 0u);
            const uint32_t app = ATREX_INDEX((lo >> f.dur_bits) & f.app_mask(), q.n_apps, q.t.ctl);
            const ull v = (ull)lds_u32(m.weights + app * 4u) * dur;
            extra |= more << u;
            vlo[u] = (uint32_t)v;
            vhi[u] = (uint32_t)(v >> 32);
            slot[u] = first_pair(window_of_form(q, key[u]), phase_of_form(q, key[u]), C);
        }
    } else {
        // the lane's entries e, e + 1, e + 2, e + 3 (e a multiple of 4) as twelve words; in an even
        // entry the 8-byte word comes first, in an odd one last.  A buffer's capacity is a multiple
        // of 4, so a lane that holds any entry may read all 48 bytes.
        const uint32_t e = e0 + 4u * lane;
        uint4 w[3];
        if (FULL || e < n_e) {
            const uint4* at = reinterpret_cast<const uint4*>(src + (size_t)e * SPILL_ENTRY_BYTES);
#pragma unroll
            for (int j = 0; j < 3; ++j) w[j] = __ldcs(at + j);
            open = FULL ? 0xFu : (0xFu >> (4u - min(n_e - e, 4u)));
        } else {
#pragma unroll
            for (int j = 0; j < 3; ++j) w[j] = make_uint4(0, 0, 0, 0);
        }
        const uint32_t alo[4] = {w[0].x, w[1].x, w[1].z, w[2].z}, ahi[4] = {w[0].y, w[1].y, w[1].w, w[2].w};
        const uint32_t b[4] = {w[0].z, w[0].w, w[2].x, w[2].y};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            key[u].hi = 0x80000000u | ((b[u] >> 8) & 0x00FF0000u) | (ahi[u] >> 16);
            key[u].lo = (part << (32 - q.t.lp)) | (b[u] & (0xFFFFFFFFu >> q.t.lp));
            vlo[u] = alo[u];
            vhi[u] = ahi[u] & 0xFFFFu;
            slot[u] = first_pair(window_of_form(q, key[u]), b[u] >> 24, C);
        }
    }
    // First look, straight-line for all four entries: most keys sit in the first pair of slots of
    // their probe sequence.  (Pairs fill from the even slot, and slots never empty again.)
    uint32_t hit = 0, room = 0, even_taken = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const PairLook look = look_at(m, ATREX_INDEX(slot[u], C - 1u, q.t.ctl), key[u]);
        if (look.second) slot[u] |= 1u;
        if (look.first || look.second) hit |= 1u << u;
        if (look.second_free) room |= 1u << u;
        if (!look.first_free) even_taken |= 1u << u;
    }
    hit &= open;     // (an absent entry is a well-formed key too)
    open &= ~hit;
    // A new key whose first pair has room is inserted at once, so that its later occurrences find it
    // there; a slot lost to another key defers the entry.
    if (__any_sync(0xFFFFFFFFu, (open & room) != 0)) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (open & room & (1u << u)) {
                const uint32_t at = slot[u] + ((even_taken >> u) & 1u);
                if (claim(m, at, key[u])) {
                    slot[u] = at;
                    hit |= 1u << u;
                    open &= ~(1u << u);
                }
            }
        }
    }
    if (__any_sync(0xFFFFFFFFu, open != 0)) {
        // The rest (keys further down their probe sequence, lost races: a few per batch) is not settled
        // here, where the fixed cost of a general probe round would be paid for a handful of entries: it
        // goes to this warp's queue and is settled by settle_queue, 32 entries per warp round.
        uint32_t before[4], total = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t pend = __ballot_sync(0xFFFFFFFFu, (open >> u) & 1u);
            before[u] = total + __popc(pend & ((1u << lane) - 1u));
            total += __popc(pend);
        }
        // (the caller settles the queue before a batch that might not fit: there is room for all 128)
        const uint32_t qbase = qn_w;
        qn_w += total;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (open & (1u << u)) {
                const ull v = vlo[u] | ((ull)vhi[u] << 32) | ((room >> u) & 1u ? 0ull : QUEUED_SKIP_FIRST) |
                              (FORM != FORM_LONG && ((extra >> u) & 1u) ? QUEUED_CONTINUATION : 0ull);
                my_queue[ATREX_INDEX(qbase + before[u], queue_cap_w, q.t.ctl)] = make_ulonglong2(((ull)key[u].hi << 32) | key[u].lo, v);
            }
        }
    }
    // (a crowded partition: where a quarter of the lanes' first entries share a slot, the batch's entries of that slot are
    // summed first)
    for (int turn = 0; CROWDED && turn < 4; ++turn) {
        const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit & 1u);
        if (hits == 0) break;
        const int lead = __ffs(hits) - 1;
        const uint32_t shared_slot = __shfl_sync(0xFFFFFFFFu, slot[0], lead);
        if (__popc(__ballot_sync(0xFFFFFFFFu, (hit & 1u) != 0 && slot[0] == shared_slot)) < 8) break;
        ull sum = 0;         // < 2^50
        uint32_t count = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if ((hit & (1u << u)) != 0 && slot[u] == shared_slot) {
                sum += (ull)vlo[u] | ((ull)vhi[u] << 32);
                count += FORM != FORM_LONG ? ~(extra >> u) & 1u : 1u;
                hit &= ~(1u << u);
            }
        }
        const ull all = (ull)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)sum & 0x1FFFFFFu) + ((ull)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)(sum >> 25)) << 25);
        count = __reduce_add_sync(0xFFFFFFFFu, count);
        if (lane == (uint32_t)lead) part_accumulate(m, shared_slot, (uint32_t)all, (uint32_t)(all >> 32), count, q.t.vals + base, C, q.t.ctl);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (hit & (1u << u)) part_accumulate(m, slot[u], vlo[u], vhi[u], FORM != FORM_LONG ? ~(extra >> u) & 1u : 1u, q.t.vals + base, C, q.t.ctl);
}

template <ull FORM>
__device__ __noinline__ void settle_queue(const PartitionParams& q, const PartSmem m, const ulonglong2* my_queue, uint32_t qn_w, ull base, uint32_t lane) {
    const uint32_t C = q.t.C;
    __syncwarp();   // the queue was written by other lanes of this warp
    for (uint32_t i0 = 0; i0 < qn_w; i0 += 32u) {
        const bool serving = i0 + lane < qn_w;
        const ulonglong2 ent = serving ? __ldcg(my_queue + i0 + lane) : make_ulonglong2(0, 0);
        const FormKey<FORM> key = {(uint32_t)(ent.x >> 32), (uint32_t)ent.x};
        const uint32_t window = window_of_form(q, key), advance = pair_stride(q.t, window);
        uint32_t start = first_pair(window, phase_of_form(q, key), C);
        if (ent.y & QUEUED_SKIP_FIRST) {
            start += advance;
            if (start >= C) start -= C;
        }
        const uint32_t count = ent.y & QUEUED_CONTINUATION ? 0u : 1u;
        const uint32_t found = probe_general(m, key, start, advance, serving, count, C, q.t.ctl);
        if (serving && found != PROBE_FAILED)
            part_accumulate(m, found, (uint32_t)ent.y, (uint32_t)(ent.y >> 32) & 0xFFFFu, count, q.t.vals + base, C, q.t.ctl);
    }
    __syncwarp();   // the queue may be overwritten from here on
}

// A warp's share of a partition's entries: sub-buffers warp, warp + n_warps, ...  Returns how many wait in its queue.
template <ull FORM, bool CROWDED>
__device__ __forceinline__ uint32_t stream_share(const PartitionParams& q, const PartSmem& m, uint32_t part, ulonglong2* my_queue, uint32_t queue_cap_w,
                                                 uint32_t warp, uint32_t n_warps, uint32_t lane) {
    const uint32_t C = q.t.C;
    const ull base = (ull)part * C;
    uint32_t qn_w = 0;  // entries in this warp's queue segment (warp-uniform)
    for (uint32_t g = warp; g < q.n_groups; g += n_warps) {
        const ull sb = ((ull)g << q.t.lp) + part;
        const uint32_t n_e = q.spill_cnt[sb];
        const unsigned char* buf = entries_of(q, sb);
        // Short-distance L2 prefetch, a fixed window of 256 entries per warp (a longer reach gets
        // evicted before use: all warps of all CTAs together must stay well inside L2): the head of
        // this warp's next sub-buffer now, and inside the loop the lines two batches ahead.
        if (g + n_warps < q.n_groups) prefetch_entries<FORM>(q, ((ull)(g + n_warps) << q.t.lp) + part, lane);
        for (uint32_t e0 = 0; e0 < n_e; e0 += 128) {
            if (lane < ENTRY_BYTES<FORM> && (e0 + 256u) * ENTRY_BYTES<FORM> + lane * 128u < n_e * ENTRY_BYTES<FORM>)
                prefetch_l2(buf + (e0 + 256u) * ENTRY_BYTES<FORM> + lane * 128u);
            if (qn_w + 128u > queue_cap_w) {   // (warp-uniform) the next batch might not fit the queue
                settle_queue<FORM>(q, m, my_queue, qn_w, base, lane);
                qn_w = 0;
            }
            if (e0 + 128u <= n_e)
                stream_batch<FORM, CROWDED, true>(q, m, buf, part, e0, n_e, C, base, my_queue, queue_cap_w, qn_w, lane);
            else
                stream_batch<FORM, CROWDED, false>(q, m, buf, part, e0, n_e, C, base, my_queue, queue_cap_w, qn_w, lane);
        }
    }
    return qn_w;
}

// A frequent key that found no place in the scatter pass's directory fills its partition, and the lanes queue at its
// limbs.  Whether a quarter of a partition's entries are alike shows in the first ones of a warp's share (2^27 records over
// 1 024 keys, 4 of them in such partitions: drain 240 -> 55 us).
__device__ __forceinline__ bool looks_crowded(const PartitionParams& q, uint32_t part, uint32_t warp, uint32_t lane) {
    if (warp >= q.n_groups) return false;
    const ull sb = ((ull)warp << q.t.lp) + part;
    const uint32_t n = q.spill_cnt[sb];
    const uint32_t hi = lane < n ? *reinterpret_cast<const uint32_t*>(entries_of(q, sb) + lane * SHORT_ENTRY_BYTES + 4) & ~SHORT_CONTINUATION : ~lane;
    const uint32_t common = __shfl_sync(0xFFFFFFFFu, hi, 0), other = __shfl_sync(0xFFFFFFFFu, hi, 1);
    return __popc(__ballot_sync(0xFFFFFFFFu, hi == common)) >= 8 || __popc(__ballot_sync(0xFFFFFFFFu, hi == other)) >= 8;
}

// What a CTA of the partition pass does, for each form of the entries.
template <ull FORM>
__device__ __forceinline__ void partition_cta(const PartitionParams& q, unsigned char* smem_raw) {
    const uint32_t C = q.t.C;
    uint2* s_acc = reinterpret_cast<uint2*>(smem_raw + C * KEY_BYTES<FORM>);   // {low limb, count | NEW_KEY_FLAG}
    uint32_t* s_a1 = reinterpret_cast<uint32_t*>(s_acc + C);  // high limb
    PartSmem m;
    m.keys = smem_addr(smem_raw);
    m.acc = smem_addr(s_acc);
    m.a1 = smem_addr(s_a1);
    m.weights = smem_addr(s_a1 + C);
    __shared__ uint32_t s_total;
    // each warp owns a segment of the CTA's queue: no shared counter, and a warp can settle its own
    // leftovers as soon as its share of the stream is through
    const uint32_t queue_cap_w = q.queue_cap / (INGEST_THREADS / 32);
    ulonglong2* const my_queue = q.queue + (size_t)blockIdx.x * q.queue_cap + (size_t)(threadIdx.x >> 5) * queue_cap_w;
    const uint32_t n_parts = 1u << q.t.lp;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, n_warps = blockDim.x >> 5;
    if (FORM != FORM_LONG)
        for (uint32_t i = threadIdx.x; i < q.n_apps; i += blockDim.x) (s_a1 + C)[i] = q.app_w[i];
    // Partitions are handed out by a counter (their entry counts differ by a few per cent, and a static
    // split leaves the kernel waiting for its slowest CTA).  A CTA draws its next one when its entries are through, early
    // enough to pull that one's keys and entries towards L2 during the write-back; drawn any earlier, the CTAs that
    // start first hold two of what little is left of 256 partitions (53 M entries: 730 us, three partitions at most CTAs' ends).
    __shared__ uint32_t s_next;
    const auto draw = [&] {
        if (threadIdx.x == 0) s_next = gridDim.x + (uint32_t)atomicAdd(&q.t.ctl->part_cursor, 1ull);   // (the first round is the static one)
    };
    uint32_t part = blockIdx.x;
    while (part < n_parts) {
        __syncthreads();  // the previous partition's write-back has finished reading shared memory
        if (threadIdx.x == 0) s_total = 0;
        __syncthreads();
        uint32_t local_total = 0;
        for (uint32_t g = threadIdx.x; g < q.n_groups; g += blockDim.x) local_total += q.spill_cnt[((ull)g << q.t.lp) + part];
        local_total = __reduce_add_sync(0xFFFFFFFFu, local_total);
        if (lane == 0 && local_total) atomicAdd(&s_total, local_total);

        __syncthreads();
        if (s_total == 0) {  // nothing was spilled to this partition (uniform)
            draw();
            __syncthreads();
            part = s_next;
            continue;
        }

        const ull base = (ull)part * C;
        for (uint32_t i0 = threadIdx.x; i0 < C; i0 += 4 * blockDim.x) {  // four key loads per thread in flight
            ull k[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) k[u] = i0 + u * blockDim.x < C ? q.t.keys[base + i0 + u * blockDim.x] : 0ull;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * blockDim.x;
                if (i < C) {
                    const FormKey<FORM> f = k[u] == 0 ? FormKey<FORM>{0u, 0u} : form_key<FORM>(q, ~k[u]);   // the table stores complemented keys, 0 = empty
                    if (FORM == FORM_TIGHT) reinterpret_cast<uint32_t*>(smem_raw)[i] = f.hi;
                    else reinterpret_cast<uint2*>(smem_raw)[i] = make_uint2(f.lo, f.hi);
                    s_acc[i] = make_uint2(0, 0);
                    s_a1[i] = 0;
                }
            }
        }
        {   // the accumulators of this partition are read back at the end: start them towards L2 now
            const unsigned char* vb = reinterpret_cast<const unsigned char*>(q.t.vals + base);
            for (uint32_t off = threadIdx.x * 128u; off < C * 16u; off += blockDim.x * 128u) prefetch_l2(vb + off);
        }
        __syncthreads();

        const uint32_t qn_w = FORM != FORM_LONG && looks_crowded(q, part, warp, lane)
                                  ? stream_share<FORM, FORM != FORM_LONG>(q, m, part, my_queue, queue_cap_w, warp, n_warps, lane)
                                  : stream_share<FORM, false>(q, m, part, my_queue, queue_cap_w, warp, n_warps, lane);
        draw();
        settle_queue<FORM>(q, m, my_queue, qn_w, base, lane);
        __syncthreads();
        const uint32_t next = s_next;
        {   // while the deltas are written back, pull the next partition's keys and each warp's
            // first sub-buffer towards L2 (used within microseconds, so they are still there)
            if (next < n_parts) {
                const unsigned char* nk = reinterpret_cast<const unsigned char*>(q.t.keys + (ull)next * C);
                for (uint32_t off = threadIdx.x * 128u; off < C * 8u; off += blockDim.x * 128u) prefetch_l2(nk + off);
                if (warp < q.n_groups) prefetch_entries<FORM>(q, ((ull)warp << q.t.lp) + next, lane);
            }
        }
        // read-modify-write of the touched slots, four per thread in flight (the loads miss L1 by
        // design and mostly come from L2, where the prefetch at the start of the partition put them)
        for (uint32_t i0 = threadIdx.x; i0 < C; i0 += 4 * blockDim.x) {
            uint2 c[4];   // {low limb, count | NEW_KEY_FLAG}
            ulonglong2 old[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * blockDim.x;
                c[u] = i < C ? s_acc[i] : make_uint2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                old[u] = make_ulonglong2(0, 0);
                if (c[u].y) {
                    const ull* vp = reinterpret_cast<const ull*>(q.t.vals + base + i0 + u * blockDim.x);
                    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(old[u].x), "=l"(old[u].y) : "l"(vp));
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (c[u].y == 0) continue;
                const uint32_t i = i0 + u * blockDim.x;
                const ull nlo = old[u].x + ((ull)c[u].x | ((ull)s_a1[i] << 32));
                const ull cnthi = old[u].y + (ull)(c[u].y & ~NEW_KEY_FLAG) + ((nlo < old[u].x ? 1ull : 0ull) << HI_SHIFT);
                q.t.vals[base + i] = make_ulonglong2(nlo, cnthi);
                if (c[u].y & NEW_KEY_FLAG) {
                    FormKey<FORM> f = {0u, 0u};
                    if (FORM == FORM_TIGHT) f.hi = reinterpret_cast<const uint32_t*>(smem_raw)[i];
                    else f = {reinterpret_cast<const uint2*>(smem_raw)[i].y, reinterpret_cast<const uint2*>(smem_raw)[i].x};
                    q.t.keys[base + i] = ~key_of_form<FORM>(q, f, part);
                }
            }
        }
        // this partition's buffers are empty again
        for (uint32_t g = threadIdx.x; g < q.n_groups; g += blockDim.x) q.spill_cnt[((ull)g << q.t.lp) + part] = 0;
        part = next;
    }
}

__global__ void __launch_bounds__(INGEST_THREADS, 1) partition_kernel(const __grid_constant__ PartitionParams q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_dependency_wait();
    // The spill buffers are drained lazily: unless forced, only when the scatter launch just before this one found a buffer
    // filling up.  A warp asks for all that this hangs on at once: asked by every warp of 148 CTAs, one word after the other, a
    // launch that has nothing to do waited for thousands of reads of one L2 sector (4.6 us; four words by every warp 6.5; now 2.9).
    Control* const ctl = q.t.ctl;
    __shared__ ull s_asked[4];
    if (threadIdx.x < 4)
        s_asked[threadIdx.x] = ld_relaxed(threadIdx.x == 0 ? &ctl->n_misfit : threadIdx.x == 1 ? &ctl->drain_seq : threadIdx.x == 2 ? &ctl->form : &ctl->rests);
    __syncthreads();
    const bool misfits = s_asked[0] > q.misfit_max;
    if (!q.force && !misfits && s_asked[1] != q.seq) return;
    const ull form = s_asked[2], rests = s_asked[3];
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&ctl->n_drains, 1ull);
    if (form != FORM_SHORT)
        partition_cta<FORM_LONG>(q, smem_raw);
    else if (rests != 0)
        partition_cta<FORM_SHORT>(q, smem_raw);
    else
        partition_cta<FORM_TIGHT>(q, smem_raw);
    grid_dependents_launch();
    // The last CTA rewinds the hand-out counter for the next launch.  Where many records did not fit the form of the
    // entries, the next ones are long (the buffers are empty now); the directory stays empty until the host, which is told,
    // has another built.
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ctl->part_done, 1ull) == gridDim.x - 1) {
            ctl->part_cursor = ctl->part_done = ctl->rests = 0;
            if (misfits) {
                ctl->form = FORM_LONG_ONLY;
                ctl->n_misfit = ctl->hot_n = 0;
                ctl->max_fill = (ctl->max_fill * SHORT_ENTRY_BYTES + SPILL_ENTRY_BYTES - 1) / SPILL_ENTRY_BYTES;   // (in entries: as many bytes)
                *(volatile ull*)q.told_long = q.trace;
            }
        }
    }
}

// --------------------------------------------------------------------------------------
// Hot-directory construction, small kernels over a sample of the records: one out of every `stride`, at a place in
// its stretch that a hash chooses.  Traces have neighbours that are alike (a kernel launched in a loop) and patterns
// that repeat (services taking turns), so records sampled side by side, or at a fixed distance, would show a key far
// more or less often than it occurs.  (Sampled four neighbours at a time, a trace whose keys come four times in a
// row lost 40 % of the keys that hold an eighth of it to keys that come once; single records lose 1 %, and cost 5 us
// more for 2^18 samples, 15 for 2^20.)
//   1. count   every sampled key bumps one of 2^20 counters chosen by its hash; the keys are kept side by side;
//   2. admit   sampled keys whose counter reached ADMIT_MIN are inserted, with exact counts,
//              into a candidate table (colliding cold keys may slip in; harmless);
//   3. level   how many candidates have which count, and from that the count that fills the directory;
//   4. gather  the candidates above it side by side, and how much weight each of four bucket hashes would lose;
//   5. list    the candidates of each bucket (two slots or four, see scatter.cu) under the best of them;
//   6. pick    each bucket takes its most frequent ones.
// Which keys end up in the directory only affects speed, never results.  Bound by latency and launches: 90 us for
// 2^20 samples; 187 us when single records were read (twice) and one CTA did steps 3 to 6.
constexpr uint32_t SKETCH_BITS = 20;   // as many counters as samples, so that cold keys stay below ADMIT_MIN
constexpr uint32_t ADMIT_MIN = 3;
constexpr uint32_t CAND_PROBES = 16;
constexpr uint32_t SAMPLE_ILP = 4;     // samples in flight per thread

__device__ __forceinline__ ull sample_at(const HotBuildParams& p, uint32_t j) {
    uint32_t h = j * HASH_A;
    h = (h ^ (h >> 15)) * HASH_C;
    return (ull)j * p.stride + __umulhi(h, (uint32_t)p.stride);
}

// Counts for lanes of a warp that target the same counter are combined first, and those of a CTA in a small
// shared-memory cache, so that a trace dominated by one key does not queue at one address.
constexpr uint32_t CACHE = 256;
struct CountCache {
    uint32_t index[CACHE], count[CACHE];   // index + 1, 0 = free
    __device__ __forceinline__ void clear() {
        for (uint32_t i = threadIdx.x; i < CACHE; i += blockDim.x) index[i] = count[i] = 0;
        __syncthreads();
    }
    __device__ __forceinline__ void add(uint32_t* counters, uint32_t at, bool active) {
        const unsigned act = __ballot_sync(0xFFFFFFFFu, active);
        if (!active) return;
        const unsigned same = __match_any_sync(act, at);
        if ((threadIdx.x & 31u) != (unsigned)(__ffs(same) - 1)) return;
        const uint32_t n = (uint32_t)__popc(same), slot = (at * 0x9E3779B1u) >> 24;
        static_assert(CACHE == 256, "top eight bits");
        if (n > 1) {
            const uint32_t owner = atomicCAS(&index[slot], 0u, at + 1u);
            if (owner == 0 || owner == at + 1u) {
                atomicAdd(&count[slot], n);
                return;
            }
        }
        atomicAdd(&counters[at], n);
    }
    __device__ __forceinline__ void flush(uint32_t* counters) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < CACHE; i += blockDim.x)
            if (count[i]) atomicAdd(&counters[index[i] - 1u], count[i]);
    }
};

__global__ void __launch_bounds__(256) hot_count_kernel(HotBuildParams p) {
    __shared__ CountCache cache;
    cache.clear();
    grid_dependency_wait();
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t rounds = (p.n_sample + stride * SAMPLE_ILP - 1) / (stride * SAMPLE_ILP);  // uniform trip count: warp collectives inside
    uint32_t max_op = 0, n_long = 0;
    for (uint32_t r = 0; r < rounds; ++r) {
        uint4 v[SAMPLE_ILP];
#pragma unroll
        for (uint32_t u = 0; u < SAMPLE_ILP; ++u) {
            const uint32_t j = (r * SAMPLE_ILP + u) * stride + blockIdx.x * blockDim.x + threadIdx.x;
            v[u] = j < p.n_sample ? p.recs[sample_at(p, j)] : make_uint4(0xFFFFFFFFu, 0, 0, 0);
        }
#pragma unroll
        for (uint32_t u = 0; u < SAMPLE_ILP; ++u) {
            const uint32_t j = (r * SAMPLE_ILP + u) * stride + blockIdx.x * blockDim.x + threadIdx.x;
            const uint32_t khi = v[u].y & 0x00FFFFFFu;
            const bool ok = j < p.n_sample && v[u].x < p.n_apps && (khi >> 16) < p.n_phases;
            if (j < p.n_sample) p.sample[j] = ok ? ((ull)khi << 32) | v[u].z : ~0ull;
            if (ok) max_op = max(max_op, khi & 0xFFFFu);
            if (ok && v[u].w > p.dur_mask) ++n_long;
            cache.add(p.sketch, hash32(khi & 0xFFFFu, v[u].z) >> (32 - SKETCH_BITS), ok);
        }
    }
    max_op = __reduce_max_sync(0xFFFFFFFFu, max_op);
    if ((threadIdx.x & 31u) == 0 && max_op >= p.max_ops) atomicMax(&p.scratch->max_op, max_op);   // (only what does not fit is told)
    n_long = __reduce_add_sync(0xFFFFFFFFu, n_long);
    if ((threadIdx.x & 31u) == 0 && n_long > rounds * SAMPLE_ILP * 4u) atomicAdd(&p.scratch->n_long, n_long);   // (an eighth of the warp's or more)
    grid_dependents_launch();
    cache.flush(p.sketch);
}

__global__ void __launch_bounds__(256) hot_admit_kernel(HotBuildParams p) {
    __shared__ CountCache cache;
    cache.clear();
    grid_dependency_wait();
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t rounds = (p.n_sample + stride * SAMPLE_ILP - 1) / (stride * SAMPLE_ILP);
    for (uint32_t r = 0; r < rounds; ++r) {
        ull key[SAMPLE_ILP];
        uint32_t seen[SAMPLE_ILP];
#pragma unroll
        for (uint32_t u = 0; u < SAMPLE_ILP; ++u) {
            const uint32_t j = (r * SAMPLE_ILP + u) * stride + blockIdx.x * blockDim.x + threadIdx.x;
            key[u] = j < p.n_sample ? p.sample[j] : ~0ull;
        }
#pragma unroll
        for (uint32_t u = 0; u < SAMPLE_ILP; ++u) seen[u] = key[u] != ~0ull ? p.sketch[hash32(key[u]) >> (32 - SKETCH_BITS)] : 0u;
#pragma unroll
        for (uint32_t u = 0; u < SAMPLE_ILP; ++u) {
            const ull skey = ~key[u];
            uint32_t s = (hash32(key[u]) * 0x9E3779B1u) >> (32 - p.cand_bits);
            bool found = false;
            if (seen[u] >= ADMIT_MIN) {
                for (uint32_t probe = 0; probe < CAND_PROBES && !found; ++probe) {
                    ull k = ld_relaxed(&p.cand_keys[s]);
                    if (k == 0) {
                        k = atomicCAS(&p.cand_keys[s], 0ull, skey);
                        if (k == 0) k = skey;
                    }
                    if (k == skey)
                        found = true;
                    else
                        s = (s + 1) & ((1u << p.cand_bits) - 1);
                }
            }
            cache.add(p.cand_cnt, s, found);
        }
    }
    grid_dependents_launch();
    cache.flush(p.cand_cnt);
}

// The words form's two-way buckets lose 5 % of 4 096 equally frequent keys and 9 % of 6 144, the tags form's four-way ones
// 2 and 6 %.  Words are faster where some keys are more frequent than others, which the buckets keep (2^27 records,
// Zipf(1.1) over 6 144 keys: 791 us against 884), and where keys are equally frequent but fewer (2 048: 740 against 809,
// 4 096: 811 against 860) or more (12 288: 1 056 against 1 082, 32 768: 1 357 against 1 808).  Between, tags hold more
// (6 144: 909 against 940, 6 880: 933 against 966), and from TAGS_PART on where such keys hold only a part of the trace.
// (These lines were measured while the scatter kernel spilled registers; without, words take 898 us against 935 at 6 144 keys
// and 1 550 against 1 730 where they hold 45 %.)
constexpr uint32_t TAGS_PART = 3500, TAGS_FROM = 5500, TAGS_TO = 7500, EVEN = 4;
// A duration that takes two short entries makes 16 bytes of a record, a long entry has 12.  Whole builds of 2^27 records, long
// entries and then short ones at a share of such durations of 0, 0.2, 0.5 and 1:
//   4 M keys Zipf(0.8), 75 % spilled     1 970   1 793 1 982 2 298 2 741 us       (short ones are faster until 0.18)
//   8 M keys Zipf(1.1), 50 %             2 045   1 848 1 956 2 215 2 554          (0.30)
//   35 % on one key, the rest over 2 M   1 885   1 719 1 850 2 122 2 701          (0.25)
//   90 % on one key                        728     729   752   781   760          (0.05)
//   12 288 equally frequent keys         1 065   1 022 1 096 1 225 1 178          (0.15)
//   4 096 equally frequent keys            855     786   809   842   891          (0.75)
//   32 768 equally frequent keys         1 690   1 292 1 390 1 564 1 948          (0.65)
//   0.5 M equally frequent keys          2 390   1 786 2 014 2 384 3 114          (0.50)
//   0.5 M keys Zipf(1.2), 27 %           1 095     947 1 011 1 100 1 219          (0.46)
// So entries are long from a quarter on, and from 7/16 on where the keys that the directory may hold have five eighths of the
// sample and where keys are equally frequent.  A trace of 2^20 records takes as long either way (192 us and
// 196, 285 and 296; of 2^24: 437 and 536), and how it goes on cannot be told from it.
constexpr ull FORM_MATTERS = 1u << 20;
constexpr uint32_t LIST_MAX = 16;       // candidates a bucket chooses from (five on average)
constexpr uint32_t LEVEL_THREADS = 1024;

__global__ void __launch_bounds__(LEVEL_THREADS) hot_level_kernel(HotBuildParams p) {
    __shared__ uint32_t s_hist[1024], s_warp[32];
    __shared__ bool s_last;
    const uint32_t t = threadIdx.x, lane = t & 31u, w = t >> 5;
    s_hist[t] = 0;
    __syncthreads();
    grid_dependency_wait();
    HotBuildScratch& x = *p.scratch;
    const uint32_t n_cand = 1u << p.cand_bits;
    uint32_t most = 0;
    for (uint32_t i0 = blockIdx.x * LEVEL_THREADS; i0 < n_cand; i0 += gridDim.x * LEVEL_THREADS) {
        const uint32_t c = p.cand_cnt[i0 + t];
        most = max(most, c);
        // (most counts are small: a warp's are counted by votes instead of queueing at a few bins)
#pragma unroll
        for (uint32_t k = ADMIT_MIN; k < ADMIT_MIN + 4; ++k) {
            const uint32_t votes = __ballot_sync(0xFFFFFFFFu, c == k);
            if (lane == 0 && votes) atomicAdd(&s_hist[k], (uint32_t)__popc(votes));
        }
        if (c != 0 && (c < ADMIT_MIN || c >= ADMIT_MIN + 4)) atomicAdd(&s_hist[min(c, 1023u)], 1u);
    }
    most = __reduce_max_sync(0xFFFFFFFFu, most);
    if (lane == 0 && most) atomicMax(&x.most, most);
    __syncthreads();
    if (s_hist[t]) atomicAdd(&x.hist[t], s_hist[t]);
    __syncthreads();
    if (t == 0) {
        __threadfence();
        s_last = atomicAdd(&x.done, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    // smallest threshold >= 2 whose class fits the directory with some over-subscription (a bucket of two ways fills
    // less evenly than one of four): thread t looks at the count 1023 - t, behind a scan over the higher ones
    const ull most_seen = __ldcg(&x.most);
    const ull skew = most_seen * 8u >= p.n_sample * 3ull ? SKEW_DOMINATED : (most_seen * 32u >= p.n_sample ? SKEW_COMBINE : SKEW_NONE);
    const bool fits = p.max_ops != 0 && __ldcg(&x.max_op) == 0;     // short entries and words can hold what was sampled
    const uint32_t mine = __ldcg(&x.hist[1023 - t]);
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        uint32_t v = s_warp[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, v, d);
            if (lane >= (uint32_t)d) v += o;
        }
        s_warp[lane] = v;
    }
    __syncthreads();
    incl += w ? s_warp[w - 1] : 0u;
    auto selection = [&](bool words) {                                     // counts 1023, 1022, ... that fit
        const uint32_t slots = p.slots[words][skew == SKEW_DOMINATED];
        const uint32_t budget = min(words ? 2 * slots : slots + slots / 4, HOT_SELECT_MAX);
        return (uint32_t)__syncthreads_count(t <= 1021 && incl <= budget);
    };
    uint32_t above = selection(fits);
    __shared__ uint32_t s_weight, s_selected;                              // of the sample, in the selected candidates; how many they are
    if (t == 0) s_weight = s_selected = 0;
    __syncthreads();
    const uint32_t weight = __reduce_add_sync(0xFFFFFFFFu, t < above ? mine * (1023u - t) : 0u);
    if (lane == 0 && weight) atomicAdd(&s_weight, weight);
    if (t + 1u == above) s_selected = incl;
    __syncthreads();
    const bool even = most_seen * s_selected < (ull)EVEN * s_weight;
    const bool tags = even && s_selected > (s_weight < p.n_sample / 2 ? TAGS_PART : TAGS_FROM) && s_selected <= TAGS_TO;
    const bool often_hit = s_weight / 5 >= p.n_sample / 8;
    const ull long_from = skew != SKEW_DOMINATED && (often_hit || even) ? p.n_sample / 16 * 7 : p.n_sample / 4;
    const bool often_long = __ldcg(&x.n_long) >= long_from && (skew == SKEW_DOMINATED || p.n_sample * p.stride > FORM_MATTERS);
    const bool words = fits && !often_long && !tags;
    if (fits && often_long) above = selection(false);
    if (t == 0) {
        x.threshold = 1024u - above;
        p.ctl->hot_skew = skew;
        p.ctl->hot_n = p.ctl->prefetch = 0;     // (hot_pick_kernel adds up)
        p.ctl->form = words ? FORM_SHORT : FORM_LONG;
    }
}

struct Buckets {
    uint32_t n, ways;
};
__device__ __forceinline__ Buckets buckets_in_use(const HotBuildParams& p) {
    const bool words = p.ctl->form != FORM_LONG;
    const uint32_t ways = words ? WORD_WAYS : TAG_WAYS;
    return {p.slots[words][p.ctl->hot_skew == SKEW_DOMINATED] / ways, ways};
}

// A multiplier's loss is approximated by arrival order among the keys that matter: those that hold 1/4096 of the sample.
// (A key of that size that finds no slot fills its partition, and the partition pass waits for the CTA that has it.)
__global__ void __launch_bounds__(256) hot_gather_kernel(HotBuildParams p) {
    __shared__ uint32_t s_lost[4];
    if (threadIdx.x < 4) s_lost[threadIdx.x] = 0;
    __syncthreads();
    grid_dependency_wait();
    HotBuildScratch& x = *p.scratch;
    const Buckets buckets = buckets_in_use(p);
    const uint32_t thr = x.threshold, lane = threadIdx.x & 31u;
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;      // (grid: one thread per candidate)
    const uint32_t c = p.cand_cnt[i];
    const uint32_t votes = __ballot_sync(0xFFFFFFFFu, c >= thr);
    uint32_t base = 0;
    if (lane == 0 && votes) base = atomicAdd(&x.n, (uint32_t)__popc(votes));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (c >= thr) {
        const uint32_t at = base + __popc(votes & ((1u << lane) - 1u));
        const ull skey = p.cand_keys[i];
        if (at < HOT_SELECT_MAX) {
            x.key[at] = skey;
            x.count[at] = c;
        }
        if (c == x.most) p.ctl->top_key = ~skey;   // (of several equally frequent ones, any)
        if (c >= max(p.n_sample >> 12, 16u)) {
#pragma unroll
            for (uint32_t m = 0; m < 4; ++m)
                if (atomicAdd(&x.occupancy[m][dir_bucket_of_key(~skey, DIR_MULTS[m], buckets.n)], 1u) >= buckets.ways) atomicAdd(&s_lost[m], c);
        }
    }
    grid_dependents_launch();
    __syncthreads();
    if (threadIdx.x < 4 && s_lost[threadIdx.x]) atomicAdd(&x.lost[threadIdx.x], s_lost[threadIdx.x]);
}

__device__ __forceinline__ uint32_t best_multiplier(const HotBuildScratch& x) {
    uint32_t best = 0;
#pragma unroll
    for (uint32_t m = 1; m < 4; ++m)
        if (x.lost[m] < x.lost[best]) best = m;
    return DIR_MULTS[best];
}

__global__ void __launch_bounds__(256) hot_list_kernel(HotBuildParams p) {
    grid_dependency_wait();
    HotBuildScratch& x = *p.scratch;
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i < min(x.n, HOT_SELECT_MAX)) {
        const uint32_t b = dir_bucket_of_key(~x.key[i], best_multiplier(x), buckets_in_use(p).n);
        const uint32_t at = atomicAdd(&x.listed[b], 1u);
        if (at < LIST_MAX) x.list[b][at] = i;
    }
    grid_dependents_launch();
}

__global__ void __launch_bounds__(128) hot_pick_kernel(HotBuildParams p) {
    __shared__ uint32_t s_inserted, s_weight;
    if (threadIdx.x == 0) s_inserted = s_weight = 0;
    __syncthreads();
    grid_dependency_wait();
    HotBuildScratch& x = *p.scratch;
    const uint32_t b = blockIdx.x * 128 + threadIdx.x;
    const Buckets buckets = buckets_in_use(p);
    const uint32_t ways = buckets.ways, mult = best_multiplier(x);
    uint32_t inserted = 0, weight = 0;
    if (b < p.hot_slots / ways) {        // (the whole image: buckets that are not in use have nothing listed)
        const uint32_t n = min(x.listed[b], LIST_MAX);
        uint32_t top[TAG_WAYS] = {0, 0, 0, 0}, who[TAG_WAYS] = {0, 0, 0, 0};
        for (uint32_t k = 0; k < n; ++k) {
            uint32_t i = x.list[b][k], c = x.count[i];
#pragma unroll
            for (uint32_t way = 0; way < TAG_WAYS; ++way) {   // insertion into the four best
                if (c > top[way]) {
                    const uint32_t tc = top[way], ti = who[way];
                    top[way] = c;
                    who[way] = i;
                    c = tc;
                    i = ti;
                }
            }
        }
        ull keys[TAG_WAYS];
#pragma unroll
        for (uint32_t way = 0; way < TAG_WAYS; ++way) {
            const bool taken = way < ways && top[way] != 0;
            keys[way] = taken ? x.key[who[way]] : 0ull;
            inserted += taken ? 1u : 0u;
            weight += taken ? top[way] : 0u;
        }
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(p.hot_keys + b * ways);
        dst[0] = make_ulonglong2(keys[0], keys[1]);
        if (ways == TAG_WAYS) {
            dst[1] = make_ulonglong2(keys[2], keys[3]);
        } else {   // (worked out here once and not by every CTA of every scatter launch)
            uint32_t word[WORD_WAYS];
#pragma unroll
            for (uint32_t way = 0; way < WORD_WAYS; ++way) {
                const uint32_t khi = (uint32_t)(~keys[way] >> 32) & 0x00FFFFFFu;
                const uint32_t left = dir_mix(hash32(~keys[way]), khi >> 16, mult) * buckets.n;
                word[way] = keys[way] ? dir_word(left, khi, p.phase_bits) : DIR_ID_MASK;
            }
            reinterpret_cast<uint2*>(p.hot_words)[b] = make_uint2(word[0], word[1]);
        }
        if (b == 0) p.ctl->dir_mult = mult;
    }
    inserted = __reduce_add_sync(0xFFFFFFFFu, inserted);
    weight = __reduce_add_sync(0xFFFFFFFFu, weight);
    if ((threadIdx.x & 31u) == 0 && inserted) {
        atomicAdd(&s_inserted, inserted);
        atomicAdd(&s_weight, weight);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_inserted) {
        atomicAdd(&p.ctl->hot_n, (ull)s_inserted);
        const uint32_t before = atomicAdd(&x.weight, s_weight);
        if (before * 3ull < p.n_sample && (before + s_weight) * 3ull >= p.n_sample) p.ctl->prefetch = 1;
    }
}

// --------------------------------------------------------------------------------------
// Merge of already aggregated units into the table: one entry per thread, a CTA per 256 entries.  Bound by the
// misses of the two atomics into a table larger than L2 (4 lists of 1.3 M entries into 4 M keys: 318 us; 368
// with a grid of 8 CTAs per SM that strode through the list, whose tail idled; two or four entries per thread
// at once were slower still).
__global__ void __launch_bounds__(256) merge_kernel(const atrex_entry_t* in, ull n, TableRef t) {
    const ull i = (ull)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const ulonglong2* e = reinterpret_cast<const ulonglong2*>(in + i);
    const ulonglong2 kc = __ldg(e), v = __ldg(e + 1);   // {key, count}, weighted time
    table_accumulate(t, kc.x, hash32(kc.x), v.x, v.y, kc.y);
}

// --------------------------------------------------------------------------------------
// host launchers

cudaError_t ingest_prepare() {
    cudaError_t e = scatter_prepare();
    if (e == cudaSuccess) e = direct_prepare();
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(partition_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448 - 2048);
}

cudaError_t launch_partition(const PartitionParams& q, int n_sms, cudaStream_t stream) {
    int grid = (int)(1u << q.t.lp) < n_sms ? (int)(1u << q.t.lp) : n_sms;
    return launch_chained(partition_kernel, (uint32_t)grid, INGEST_THREADS, partition_smem_bytes(q.t.C, q.n_apps, q.fmt.dur_bits != 0), stream, q);
}

cudaError_t launch_hot_build(const HotBuildParams& p, int n_sms, cudaStream_t stream) {
    // the caller has zeroed the sketch and the candidate table on this stream
    int grid = (int)((p.n_sample + 256 * SAMPLE_ILP - 1) / (256 * SAMPLE_ILP));
    if (grid > n_sms * 8) grid = n_sms * 8;
    hot_count_kernel<<<grid, 256, 0, stream>>>(p);
    hot_admit_kernel<<<grid, 256, 0, stream>>>(p);
    cudaError_t e = cudaGetLastError();
    const uint32_t n_cand = 1u << p.cand_bits, n_buckets = p.hot_slots / WORD_WAYS;
    if (e == cudaSuccess) e = launch_chained(hot_level_kernel, n_cand / LEVEL_THREADS, LEVEL_THREADS, 0, stream, p);
    if (e == cudaSuccess) e = launch_chained(hot_gather_kernel, n_cand / 256, 256, 0, stream, p);
    if (e == cudaSuccess) e = launch_chained(hot_list_kernel, (HOT_SELECT_MAX + 255) / 256, 256, 0, stream, p);
    if (e == cudaSuccess) e = launch_chained(hot_pick_kernel, (n_buckets + 127) / 128, 128, 0, stream, p);
    return e;
}

cudaError_t launch_hot_fold(const ull* hot_keys, const ulonglong2* hot_img, uint32_t n_groups, uint32_t hot_slots,
                            const TableRef& t, cudaStream_t stream) {
    if (hot_slots == 0) return cudaSuccess;
    hot_fold_kernel<<<(hot_slots + 31) / 32, FOLD_WARPS * 32, 0, stream>>>(hot_keys, hot_img, n_groups, hot_slots, t);
    return cudaGetLastError();
}

cudaError_t launch_merge(const atrex_entry_t* in, ull n, const TableRef& t, cudaStream_t stream) {
    constexpr ull PIECE = 1ull << 38;   // entries per launch (grid limit)
    for (ull off = 0; off < n; off += PIECE) {
        const ull m = n - off < PIECE ? n - off : PIECE;
        merge_kernel<<<(unsigned)((m + 255) / 256), 256, 0, stream>>>(in + off, m, t);
    }
    return cudaGetLastError();
}

}  // namespace atrex
