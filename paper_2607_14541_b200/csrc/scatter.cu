// Pass 1 of the ingest (Eq. 2's group-by sum, streamed): SCATTER, one persistent CTA per SM.
//
// Each thread pulls records with 32-byte vector loads (two 16-byte records per load, two loads
// alternating per thread so that one is in flight while the other is consumed, streaming cache policy),
// validates, packs the key and multiplies the application's card-hour weight by the duration.
//   * Keys found in the shared-memory HOT DIRECTORY (the most frequent keys of a sample of the
//     trace, identical in every CTA, read-only during the pass) are accumulated on the spot with
//     32-bit shared-memory atomics in limbs with explicit carries.  It comes in two forms:
//       words  a key's phase and operator, if they fit 11 bits together, and what its bucket leaves over of the bucket
//              hash (a bijection of the shape) make one 32-bit word that identifies it inside the bucket: one 8-byte
//              load looks at both slots of a bucket and settles the look-up.  16 bytes a slot instead of 21 hold a third more
//              keys, and what is left of a record fits a short entry (2^27 records, 50 % spilled: 820 -> 655 us; 67 %
//              spilled 970 -> 700; 27 % 690 -> 560; 1 024 keys, none spilled: 690 -> 550).
//       tags   operators of any size: a tag byte per slot of a 4-way bucket, the slot whose tag matches confirmed
//              against its 8-byte key.  Chosen by the directory build where a sampled operator does not fit a word.
//   * Every other record becomes an entry appended to the CTA's private buffer of the key's partition: with the words
//     form a short one of 8 bytes {phase, operator, hash bits, application, duration} (short_append), with the tags form,
//     or without a directory, one of 12 bytes {product, operator, phase, hash bits} (spill_append).
// At the end the CTA adds its directory accumulators to its own row of a directory image
// ([CTA][slot], plain coalesced read-modify-writes; hot_fold_kernel adds the rows into the table
// before results are read) and stores its per-partition cursors: the buffers persist across launches
// until the partition pass drains them.
//
// The kernel runs out of issue slots, shared-memory pipe cycles and latency-hiding warps long before
// it runs out of DRAM bandwidth, so the hot loop is written for a low instruction count: the shared-memory layout is a compile-time function
// of the partition count (every array address is a register plus an immediate), rarely taken
// branches (products of 2^48 and more, a full buffer, a drain of a directory slot) are calls to functions that are not inlined, and the load buffers alternate by
// name instead of being copied.
#include "atrex_dev.cuh"
#include "kernels.h"

namespace atrex {

namespace {

#ifndef ATREX_SCATTER_THREADS
#define ATREX_SCATTER_THREADS 1024
#endif
constexpr int SCATTER_THREADS = ATREX_SCATTER_THREADS;
constexpr uint32_t NO_SLOT = 0xFFFFFFFFu;
// the directory's form
constexpr int DIR_NONE = 0, DIR_TAGS = 1, DIR_WORDS = 2;

// Shared-memory map of the scatter pass for 2^LP partitions (byte offsets into the dynamic shared memory).
template <uint32_t LP, int DIR>
struct Smem {
    static constexpr uint32_t P = 1u << LP;
    static constexpr bool W = DIR == DIR_WORDS;
    static constexpr uint32_t WAYS = W ? WORD_WAYS : TAG_WAYS;
    static constexpr uint32_t SLOTS = scatter_slots(LP, W);     // directory slots, whole buckets
    static constexpr uint32_t NB = SLOTS / WAYS;
    static constexpr uint32_t RING = 0;                         // record ring: SCATTER_RING_STAGES tiles
    static constexpr uint32_t CUR = RING + SCATTER_RING_STAGES * SCATTER_RING_TILE;   // u32[P]  entries appended to this CTA's buffer of each partition
    static constexpr uint32_t APPW = CUR + 4u * P;              // u32[APPW_SMEM_MAX]  card-hour weights
    static constexpr uint32_t LONG = APPW + 4u * APPW_SMEM_MAX;    // words: records that took two short entries
    static constexpr uint32_t RESTS = LONG + 4u;                // ... whether an entry's identity has a rest
    static constexpr uint32_t MISFITS = LONG + 8u;              // ... records whose operator does not fit
    static constexpr uint32_t WORDS = LONG + 16u;               // ... u32[SLOTS]
    static constexpr uint32_t TAG = LONG;                       // tags: u32[NB + 1]  four 8-bit tags per bucket (+ one pad bucket)
    static constexpr uint32_t KEYS = (TAG + 4u * (NB + 1u) + 7u) & ~7u;   // ull[SLOTS + 4]  key, all ones = empty
    static constexpr uint32_t PAD = W ? 0u : TAG_WAYS;          // (a look-up without a match reads the slot behind its bucket)
    static constexpr uint32_t ACC = W ? WORDS + 4u * SLOTS : KEYS + 8u * (SLOTS + PAD);   // {u32 lo, u32 hi, u32 count}[SLOTS + PAD]
    static constexpr uint32_t TOTAL = ACC + 12u * (SLOTS + PAD);
    // one key dominates: fewer slots in use, the warps' queues behind them
    static constexpr uint32_t SLOTS_DOM = scatter_dominated_slots(LP, W), NB_DOM = SLOTS_DOM / WAYS;
    static constexpr uint32_t QUEUE = (ACC + 12u * SLOTS_DOM + 15u) & ~15u;   // uint4[32 warps][SCATTER_QUEUE]
    static_assert(QUEUE + SCATTER_QUEUE_BYTES <= TOTAL, "queues");
    template <ull SKEW>
    static constexpr uint32_t NB_OF = SKEW == SKEW_DOMINATED ? NB_DOM : NB;
    static_assert(TOTAL <= SCATTER_SMEM_BYTES, "scatter pass shared memory");
    static_assert(SLOTS % 32 == 0, "whole buckets");
    // The products hash x buckets of a bucket's hashes differ by multiples of the number of buckets in their low words,
    // so with at least 2^DIR_ID_BITS buckets the bits that a word keeps of it tell them apart.
    static_assert(!W || SCATTER_RING_STAGES != 0 || NB_DOM >= 1u << DIR_ID_BITS, "words identify keys");
};
template <uint32_t LP>
constexpr uint32_t smem_total() { return Smem<LP, DIR_WORDS>::TOTAL > Smem<LP, DIR_TAGS>::TOTAL ? Smem<LP, DIR_WORDS>::TOTAL : Smem<LP, DIR_TAGS>::TOTAL; }

__device__ __forceinline__ void ld_stream_256(const void* p, uint32_t (&w)[8]) {
    asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(p));
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Loads of the directory's words, tags and keys and of the weights: these arrays are read-only during the
// pass, so the loads are not volatile and the compiler may overlap the look-ups of several records.
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds_v2u32(uint32_t a) {
    uint2 v;
    asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ ull lds_u64(uint32_t a) {
    ull v;
    asm("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a));
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
__device__ __forceinline__ uint32_t atoms_exch(uint32_t a, uint32_t v) {
    uint32_t o;
    asm volatile("atom.shared.exch.b32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
// What the hot loop keeps in registers (everything else is read from the kernel's parameter block,
// i.e. straight from the constant bank).
struct Ctx {
    uint32_t sb;              // shared-window address of the dynamic shared memory
    uint32_t mult;            // bucket-hash multiplier of this directory image
    unsigned char* my_spill;  // this CTA's buffers
    ull keep;                 // L2 cache policy of the spill stores: evict last
};

// (rare) counters of invalid records and of records that found their buffer full
__device__ __noinline__ void count_one(ull* counter) { atomicAdd(counter, 1ull); }

// Shared-memory accumulation uses native 32-bit atomics only (64-bit shared atomics are
// compare-and-swap loops).  A slot's weighted time is kept in two limbs: the returning add on the
// low limb tells the adder whether it wrapped, and the adder then adds the carry, with the value's
// high word, to the high limb.  One add raises the high limb by at most 2^21 (a warp's combined 32
// records of < 2^48 each), so the adder that takes it across 2^30 drains both limbs; the adds that
// can slip in before its exchange (one per thread of the CTA) stay below 2^31, so the high limb
// never wraps.
constexpr uint32_t DRAIN_BIT = 0x40000000u;

// (rare) Moves a directory slot's limbs to the table.  The two exchanges need not be simultaneous:
// whatever lands between them stays in the limbs for the next drain or the final flush.
__device__ __noinline__ void drain_slot(TableRef t, uint32_t acc, ull key, uint32_t h) {
    const ull lo = atoms_exch(acc, 0u);
    const ull hi = atoms_exch(acc + 4, 0u);
    const ull v = lo + (hi << 32);
    table_accumulate(t, key, h, v, v < lo ? 1ull : 0ull, 0);
}

// (rare) A record that cannot take the limb route: straight to the table with full 64-bit adds.
__device__ __noinline__ void table_route(TableRef t, ull key, uint32_t h, ull prod) { table_accumulate(t, key, h, prod, 0, 1); }
// (rare) An invalid record is counted; a valid one whose product has bits at or above 2^48, or whose operator does not
// fit, goes to the table.  Those are counted in shared memory: there may be many, and a counter of the whole GPU takes
// no more than one and a half in a nanosecond.
template <bool COUNT_MISFITS>
__device__ __noinline__ void rare_record(TableRef t, bool valid, ull key, uint32_t h, ull prod, uint32_t misfits) {
    if (valid) {
        table_accumulate(t, key, h, prod, 0, 1);
        if (COUNT_MISFITS && (uint32_t)(prod >> 32) < 0x10000u) reds_add(misfits, 1u);
    } else
        atomicAdd(&t.ctl->n_rejected, 1ull);
}

// Add (count, v) to a directory slot, v < 2^53, count <= 32.  Most products fit 32 bits and most
// low-limb adds do not wrap: the high limb is then left alone (one returning atomic and one reduction
// per hit instead of two and one).
template <uint32_t LP, int DIR>
__device__ __forceinline__ void dir_add(const IngestParams& p, const Ctx& c, uint32_t slot, ull v, uint32_t count, ull key,
                                        uint32_t h) {
    const uint32_t acc = c.sb + Smem<LP, DIR>::ACC + ATREX_INDEX(slot, (Smem<LP, DIR>::SLOTS), p.t.ctl) * 12u;
    const uint32_t v0 = (uint32_t)v;
    const uint32_t o0 = atoms_add(acc, v0);
    reds_add(acc + 8, count);
    const uint32_t x1 = (uint32_t)(v >> 32) + ((o0 + v0 < o0) ? 1u : 0u);
    if (x1 != 0) {
        const uint32_t o1 = atoms_add(acc + 4, x1);
        if ((o1 + x1) & ~o1 & DRAIN_BIT) drain_slot(p.t, acc, key, h);
    }
}

// (rare) The buffer is full: the ticket has been handed back, the record takes the exact slow path.
__device__ __noinline__ void count_overflow(TableRef t, ull key, ull prod, uint32_t h) {
    table_accumulate(t, key, h, prod, 0, 1);
    atomicAdd(&t.ctl->n_overflow, 1ull);
}

// Spill: the record becomes a 12-byte entry in this CTA's buffer of the key's partition -- an 8-byte
// word {product (48 bits), operator} and a 4-byte word {phase, the hash bits below the partition's}.
// Inside its partition (the hash's top bits) the triple (phase, operator, hash) identifies the key:
// for a given operator the hash is a bijection of the shape (shape_of_hash).
template <uint32_t LP>
__device__ __forceinline__ void spill_append(const IngestParams& p, Ctx& c, bool todo, uint32_t khi, uint32_t shape, ull prod,
                                             uint32_t h) {
    if (!todo) return;
    const uint32_t part = ATREX_INDEX(h >> (32 - LP), 1u << LP, p.t.ctl);
    const uint32_t cw = c.sb + Smem<LP, DIR_NONE>::CUR + part * 4u;     // (the same in either form)
    const uint32_t tk = atoms_add(cw, 1u);
    if (tk < p.cap) {
        // Entry tk occupies bytes [12 tk, 12 tk + 12) of the buffer; its 8-byte word sits at whichever
        // end is 8-byte aligned.  Two or three entries before the buffer reaches its next 128-byte
        // line, that line is pulled into L2 (a partial store into a line that is not cached stalls on a
        // fill), and the stores ask the L2 to evict their lines last: a buffer's current line is
        // written to some 20 times over ~40 K cycles while 16 GiB of records stream through the same cache.
        // (a CTA's buffers together stay below 4 GB: 2^12 partitions x 2^15 entries x 12 bytes)
        const uint32_t off = (part * p.cap + ATREX_INDEX(tk, p.cap, p.t.ctl)) * SPILL_ENTRY_BYTES;
        const uint32_t odd = tk & 1u;
        // word a = product | operator << 48, word b = phase << 24 | low hash bits, put together bytewise
        const uint32_t a_hi = __byte_perm((uint32_t)(prod >> 32), khi, 0x5410);
        const uint32_t b = __byte_perm(h & (0xFFFFFFFFu >> LP), khi, 0x6210);
        {   // one address: the entry's parity picks between two pairs of stores at immediate offsets (the
            // 8-byte word goes to the 8-byte aligned end), which is cheaper than computing two addresses
            unsigned char* at = c.my_spill + off;
            asm volatile(
                "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t"
                "@q  st.global.L2::cache_hint.u32 [%0], %3, %4;\n\t"
                "@q  st.global.L2::cache_hint.v2.u32 [%0+4], {%1, %2}, %4;\n\t"
                "@!q st.global.L2::cache_hint.v2.u32 [%0], {%1, %2}, %4;\n\t"
                "@!q st.global.L2::cache_hint.u32 [%0+8], %3, %4;\n\t}"
                ::"l"(at), "r"((uint32_t)prod), "r"(a_hi), "r"(b), "l"(c.keep), "r"(odd) : "memory");
            if ((off & 127u) - 96u < 12u) asm volatile("prefetch.global.L2 [%0+64];" ::"l"(at));
        }
    } else {
        reds_add(cw, 0xFFFFFFFFu);
        count_overflow(p.t, ((ull)khi << 32) | shape, prod, h);
    }
}

// The same as a short entry (ShortFormat), in one store; a duration that does not fit takes a second entry behind it.
template <uint32_t LP, int DIR>
__device__ __forceinline__ void short_append(const IngestParams& p, Ctx& c, bool todo, uint32_t khi, uint32_t app, uint32_t shape,
                                             uint32_t dur, ull prod, uint32_t h) {
    if (!todo) return;
    const uint32_t part = ATREX_INDEX(h >> (32 - LP), 1u << LP, p.t.ctl);
    const uint32_t cw = c.sb + Smem<LP, DIR>::CUR + part * 4u;
    const ShortFormat& f = p.fmt;
    const uint32_t rest = dur >> f.dur_bits, n = rest ? 2u : 1u;
    const uint32_t tk = atoms_add(cw, n);
    if (tk + n <= p.short_cap) {
        const uint32_t id = identity(khi, f.phase_bits);
        const uint32_t hi = ((h << (LP - 1u)) & 0x7FFFFFFFu) | (id & ((1u << (LP - 1u)) - 1u));
        const uint32_t id_rest = id >> (LP - 1u), lo = (id_rest << f.rest_shift) | (app << f.dur_bits);
        if (LP - 1u < DIR_ID_BITS - 1u && id_rest) asm volatile("st.shared.u32 [%0], 1;" ::"r"(c.sb + Smem<LP, DIR>::RESTS) : "memory");
        unsigned char* at = c.my_spill + (part * p.short_cap + ATREX_INDEX(tk, p.short_cap, p.t.ctl)) * SHORT_ENTRY_BYTES;
        asm volatile("st.global.L2::cache_hint.v2.u32 [%0], {%1, %2}, %3;" ::"l"(at), "r"(lo | (dur & f.dur_mask())), "r"(hi), "l"(c.keep) : "memory");
        // three entries before the buffer reaches its next line (four, where this one takes two places), as above
        if ((tk & 15u) - (14u - n) < n) asm volatile("prefetch.global.L2 [%0+64];" ::"l"(at));
        if (rest) {
            reds_add(c.sb + Smem<LP, DIR>::LONG, 1u);
            asm volatile("st.global.L2::cache_hint.v2.u32 [%0+8], {%1, %2}, %3;" ::"l"(at), "r"(lo | rest), "r"(hi | SHORT_CONTINUATION), "l"(c.keep) : "memory");
        }
    } else {
        reds_add(cw, 0u - n);
        count_overflow(p.t, ((ull)khi << 32) | shape, prod, h);
    }
}

// One record, start to finish (the register-staged loop has no registers to spare for working on
// two records at once).  Called by all lanes of a warp together (absent records masked by `present`).
template <uint32_t LP, int DIR, ull SKEW, bool FULL>
__device__ __forceinline__ void one_record(const IngestParams& p, Ctx& c, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                           bool present) {
    using L = Smem<LP, DIR>;
    const uint32_t khi = w1 & 0x00FFFFFFu;                  // phase << 16 | op_id: the key's high word
    bool ok = w0 < p.n_apps && khi < p.phase_lim;
    if (!FULL) ok = ok && present;
    // card-hour weight: from shared memory when the table fits there (an out-of-range index reads
    // some other weight, which is not used), else from global memory
    const uint32_t wgt = (p.appw_in_smem != 0) ? lds_u32(c.sb + L::APPW + (w0 & (APPW_SMEM_MAX - 1u)) * 4u) : __ldg(p.app_w + (ok ? w0 : 0u));
    const ull prod = (ull)wgt * (ull)w3;
    const uint32_t h = hash32(khi & 0xFFFFu, w2);
    const ull key = ((ull)khi << 32) | w2;
    // The limb arithmetic and the 12-byte spill entries assume products below 2^48 (e.g. weights
    // < 2^20, durations < 2^28).  Anything larger is still exact: straight to the table.  That and
    // the count of invalid records share one rarely taken branch (two separate ones cost the
    // configurations whose records mostly hit the directory 4-9 %).
    bool todo_in = ok && (uint32_t)(prod >> 32) < 0x10000u;
    // (words form: an operator that no sampled record had may not fit a word and a short entry)
    if (L::W) todo_in = todo_in && (khi & 0xFFFFu) < p.fmt.max_ops;
    bool todo = todo_in;
    if ((FULL || present) && !todo_in) rare_record<L::W>(p.t, ok, key, h, prod, c.sb + L::MISFITS);
    if (DIR != DIR_NONE) {
        const uint32_t x = dir_mix(h, khi >> 16, c.mult);
        uint32_t at;
        bool hit;
        if (L::W) {
            const ull product = (ull)x * L::template NB_OF<SKEW>;
            const uint32_t b = ATREX_INDEX((uint32_t)(product >> 32), L::template NB_OF<SKEW>, p.t.ctl);
            const uint32_t word = dir_word((uint32_t)product, khi, p.fmt.phase_bits);
            const uint2 w = lds_v2u32(c.sb + L::WORDS + b * 8u);
            const bool second = w.y == word;
            at = b * 2u + (second ? 1u : 0u);
            hit = todo && (w.x == word || second);
        } else {
            // One 32-bit word per 4-slot bucket holds an 8-bit tag per slot (hash bits the bucket choice does not
            // use); the lowest slot whose tag matches is confirmed against the 8-byte key.  A wrong tag match (1 in
            // 64 look-ups) fails the confirmation and the record takes the spill path: slower, still exact.
            const uint32_t b = ATREX_INDEX(__umulhi(x, L::template NB_OF<SKEW>), L::template NB_OF<SKEW>, p.t.ctl);
            const uint32_t t = lds_u32(c.sb + L::TAG + b * 4u) ^ __byte_perm(x, 0, 0);   // 0 in the bytes that match
            const uint32_t m = (t - 0x01010101u) & ~t & 0x80808080u;                      // lowest flagged byte is exact
            at = ATREX_INDEX(b * TAG_WAYS + ((uint32_t)__clz((int)__brev(m)) >> 3), L::SLOTS + TAG_WAYS, p.t.ctl);
            hit = todo && m != 0 && lds_u64(c.sb + L::KEYS + at * 8u) == key;
        }
        if (SKEW != SKEW_NONE) {
            // a key is frequent enough for collisions inside a warp: combine the lanes that share the first hitting lane's slot
            const unsigned hits = __ballot_sync(0xFFFFFFFFu, hit);
            if (hits != 0) {
                const int lead = __ffs(hits) - 1;
                const uint32_t slot = hit ? at : NO_SLOT;
                const uint32_t ls = __shfl_sync(0xFFFFFFFFu, slot, lead);
                const unsigned same = __ballot_sync(0xFFFFFFFFu, slot == ls);
                if (__popc(same) >= 2 && slot == ls) {
                    const uint32_t s_lo = __reduce_add_sync(same, (uint32_t)prod & 0xFFFFFFu);
                    const uint32_t s_hi = __reduce_add_sync(same, (uint32_t)(prod >> 24));
                    if ((threadIdx.x & 31u) == (unsigned)lead)
                        dir_add<LP, DIR>(p, c, ls, (ull)s_lo + ((ull)s_hi << 24), (uint32_t)__popc(same), key, h);
                    hit = false;
                    todo = false;
                }
            }
        }
        if (hit) {
            dir_add<LP, DIR>(p, c, at, prod, 1u, key, h);
            todo = false;
        }
    }
    if (L::W)
        short_append<LP, DIR>(p, c, todo, khi, w0, w2, w3, prod, h);
    else
        spill_append<LP>(p, c, todo, khi, w2, prod, h);
}

// The same for R records per lane at once (used with the shared-memory record ring, where the
// registers allow it; w[r] = the record's four words).  Called by all lanes of a
// warp together (absent records masked by `present`).  Written in stages over the R records so that
// their shared-memory round trips overlap: all look-ups are issued before the first result is used.
template <uint32_t LP, int DIR, ull SKEW, bool FULL, int R>
__device__ __forceinline__ void process(const IngestParams& p, Ctx& c, const uint32_t (&w)[R][4], bool present) {
    using L = Smem<LP, DIR>;
    uint32_t khi[R], h[R], wgt[R], x[R], tags[R];
    bool todo[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        khi[r] = w[r][1] & 0x00FFFFFFu;                  // phase << 16 | op_id: the key's high word
        bool ok = w[r][0] < p.n_apps && khi[r] < p.phase_lim;
        if (!FULL) ok = ok && present;
        if ((FULL || present) && !ok) count_one(&p.t.ctl->n_rejected);
        todo[r] = ok;
        // card-hour weight: from shared memory when the table fits there (an out-of-range index reads
        // some other weight, which is not used), else from global memory
        wgt[r] = (p.appw_in_smem != 0) ? lds_u32(c.sb + L::APPW + (w[r][0] & (APPW_SMEM_MAX - 1u)) * 4u) : __ldg(p.app_w + (ok ? w[r][0] : 0u));
        h[r] = hash32(khi[r] & 0xFFFFu, w[r][2]);
        if (DIR != DIR_NONE) {
            // Directory look-up: one 32-bit word per 4-slot bucket holds an 8-bit tag per slot (hash
            // bits the bucket choice does not use)
            x[r] = dir_mix(h[r], khi[r] >> 16, c.mult);
            tags[r] = lds_u32(c.sb + L::TAG + __umulhi(x[r], L::template NB_OF<SKEW>) * 4u);
        }
    }
    ull prod[R];
    uint32_t at[R];
    ull found[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        prod[r] = (ull)wgt[r] * (ull)w[r][3];
        if (DIR != DIR_NONE) {
            // the lowest slot whose tag matches is confirmed against the 8-byte key; a wrong tag match
            // (1 in 64 look-ups) fails the confirmation and the record takes the spill path: slower,
            // still exact
            const uint32_t t = tags[r] ^ __byte_perm(x[r], 0, 0);                     // 0 in the bytes that match
            const uint32_t m = (t - 0x01010101u) & ~t & 0x80808080u;                  // lowest flagged byte is exact
            at[r] = __umulhi(x[r], L::template NB_OF<SKEW>) * TAG_WAYS + ((uint32_t)__clz((int)__brev(m)) >> 3);
            found[r] = ~0ull;
            if (m != 0) found[r] = lds_u64(c.sb + L::KEYS + at[r] * 8u);
        }
    }
    bool hit[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const ull key = ((ull)khi[r] << 32) | w[r][2];
        // The limb arithmetic and the 12-byte spill entries assume products below 2^48 (e.g. weights
        // < 2^20, durations < 2^28).  Anything larger is still exact: straight to the table.
        if (todo[r] && (uint32_t)(prod[r] >> 32) >= 0x10000u) {
            table_route(p.t, key, h[r], prod[r]);
            todo[r] = false;
        }
        hit[r] = DIR != DIR_NONE && todo[r] && found[r] == key;
    }
    if (DIR != DIR_NONE && SKEW != SKEW_NONE) {
        // a key is frequent enough for collisions inside a warp: combine the lanes that share the first hitting lane's slot
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const unsigned hits = __ballot_sync(0xFFFFFFFFu, hit[r]);
            if (hits == 0) continue;
            const int lead = __ffs(hits) - 1;
            const uint32_t slot = hit[r] ? at[r] : NO_SLOT;
            const uint32_t ls = __shfl_sync(0xFFFFFFFFu, slot, lead);
            const unsigned same = __ballot_sync(0xFFFFFFFFu, slot == ls);
            if (__popc(same) >= 2 && slot == ls) {
                const uint32_t s_lo = __reduce_add_sync(same, (uint32_t)prod[r] & 0xFFFFFFu);
                const uint32_t s_hi = __reduce_add_sync(same, (uint32_t)(prod[r] >> 24));
                if ((threadIdx.x & 31u) == (unsigned)lead)
                    dir_add<LP, DIR>(p, c, ls, (ull)s_lo + ((ull)s_hi << 24), (uint32_t)__popc(same), ((ull)khi[r] << 32) | w[r][2], h[r]);
                hit[r] = false;
                todo[r] = false;
            }
        }
    }
    if (DIR != DIR_NONE) {
        // hits: the returning low-limb adds of all R records first, then the rest
        uint32_t o0[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (hit[r]) o0[r] = atoms_add(c.sb + L::ACC + at[r] * 12u, (uint32_t)prod[r]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (hit[r]) {
                const uint32_t acc = c.sb + L::ACC + at[r] * 12u;
                const uint32_t v0 = (uint32_t)prod[r];
                reds_add(acc + 8, 1u);
                const uint32_t x1 = (uint32_t)(prod[r] >> 32) + ((o0[r] + v0 < o0[r]) ? 1u : 0u);
                if (x1 != 0) {
                    const uint32_t o1 = atoms_add(acc + 4, x1);
                    if ((o1 + x1) & ~o1 & DRAIN_BIT) drain_slot(p.t, acc, ((ull)khi[r] << 32) | w[r][2], h[r]);
                }
                todo[r] = false;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) spill_append<LP>(p, c, todo[r], khi[r], w[r][2], prod[r], h[r]);
}

template <uint32_t LP, int DIR, ull SKEW>
__device__ __forceinline__ void scatter_body(const IngestParams& p, Ctx& c) {
    // CTA b handles record pairs (b + k * gridDim) * 1024 + tid, k = 0, 1, ...  Two 32-byte loads
    // alternate per thread: while one is consumed the next is in flight.  Rounds in which every
    // CTA's tile is complete need no bounds checks; the last (ragged) ones are predicated.
    const unsigned char* body = reinterpret_cast<const unsigned char*>(p.body);
    const uint32_t stride = gridDim.x * SCATTER_THREADS;                  // pairs per round
    const uint32_t full_rounds = (uint32_t)(p.n_pairs / stride);
    const uint32_t rounds = (uint32_t)((p.n_pairs + stride - 1) / stride);
    const uint32_t first = blockIdx.x * SCATTER_THREADS + threadIdx.x;
    uint32_t bufA[8], bufB[8];
    auto fetch = [&](uint32_t round, uint32_t (&raw)[8]) {                // any round, bounds checked
        const ull i = first + (ull)round * stride;
        if (round < rounds && i < p.n_pairs) {
            ld_stream_256(body + i * 32, raw);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) raw[j] = 0;
        }
    };
    auto consume_full = [&](const uint32_t (&raw)[8]) {
        one_record<LP, DIR, SKEW, true>(p, c, raw[0], raw[1], raw[2], raw[3], true);
        one_record<LP, DIR, SKEW, true>(p, c, raw[4], raw[5], raw[6], raw[7], true);
    };
    auto consume_tail = [&](uint32_t round, const uint32_t (&raw)[8]) {
        const bool present = round < rounds && first + (ull)round * stride < p.n_pairs;
        one_record<LP, DIR, SKEW, false>(p, c, raw[0], raw[1], raw[2], raw[3], present);
        one_record<LP, DIR, SKEW, false>(p, c, raw[4], raw[5], raw[6], raw[7], present);
    };
    fetch(0, bufA);
    uint32_t round = 0;
    {
        // main part: every round fetched here is complete for every CTA, so the loads need no checks
        const unsigned char* next = body + (first + (ull)stride) * 32;
        const uint32_t step = gridDim.x * (SCATTER_THREADS * 32u);
        // Each load goes out behind an L2 prefetch of the round after it -- where a third of the sample or more is in
        // the directory: the lines of a trace that mostly spills need the L2 more (52 % spilled: 856 -> 832 us
        // per 2^27 records with the prefetch, 75 %: 1 003 -> 1 026).
        const bool ahead = (threadIdx.x & 3u) == 0 && DIR != DIR_NONE && p.t.ctl->prefetch != 0;
        for (; round + 4 <= full_rounds; round += 2) {
            ld_stream_256(next, bufB);
            if (ahead) asm volatile("prefetch.global.L2 [%0];" ::"l"(next + step));
            next += step;
            consume_full(bufA);
            ld_stream_256(next, bufA);
            if (ahead) asm volatile("prefetch.global.L2 [%0];" ::"l"(next + step));
            next += step;
            consume_full(bufB);
        }
    }
    for (; round < rounds; round += 2) {
        fetch(round + 1, bufB);
        consume_tail(round, bufA);
        fetch(round + 2, bufA);
        consume_tail(round + 1, bufB);
    }
    // records that do not form an aligned pair (at most one before and one after the body)
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        uint4 v = make_uint4(0, 0, 0, 0);
        const bool present = threadIdx.x < p.n_single;
        if (present) v = *reinterpret_cast<const uint4*>(threadIdx.x == 0 ? p.single[0] : p.single[1]);
        one_record<LP, DIR, SKEW, false>(p, c, v.x, v.y, v.z, v.w, present);
    }
}

// ---- one key dominates the trace -----------------------------------------------------------------
// Its records are recognised before anything else is done with them and summed in registers; the others go to the
// warp's queue in shared memory and through one_record 32 at a time, so that what is left of a warp's 32
// records does not cost the price of 32.  Bound by DRAM once the key holds most records (90 %: 140 -> 57 warp
// instructions per 32 records, 0.66 -> 0.39 ms per 2^27 records); the queue pays from a share of 3/8 on.
// The lane's number and the mask of the lanes below it are read where they are needed: kept in registers they pushed
// the loop's own values out to memory, beside five other bodies in one kernel (tags form, 2^29 records of two-entry durations:
// ingest 1 801 -> 1 690 us; words form, whole build 2 431 -> 2 409; tables of 2^21 to 2^25 keys: 1 to 8 % in the tags form).
__device__ __forceinline__ uint32_t lane_id() {
    uint32_t v;
    asm("mov.u32 %0, %%laneid;" : "=r"(v));
    return v;
}
__device__ __forceinline__ uint32_t lanes_below() {
    uint32_t v;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(v));
    return v;
}
template <uint32_t LP, int DIR>
__device__ __forceinline__ void dominated_body(const IngestParams& p, Ctx& c) {
    using L = Smem<LP, DIR>;
    const uint32_t queue = c.sb + L::QUEUE + (threadIdx.x >> 5) * (SCATTER_QUEUE * 16u);
    const ull top = p.t.ctl->top_key;
    const uint32_t top_hi = (uint32_t)(top >> 32), top_lo = (uint32_t)top;
    ull sum = 0;                           // (products of 2^48 and more take the queue, so that it cannot wrap)
    uint32_t count = 0, q = 0;
    auto settle = [&](uint32_t n) {        // the last n records of the queue (n = 32 but for the last time)
        __syncwarp();
        uint4 v = make_uint4(0, 0, 0, 0);
        if (lane_id() < n)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(queue + (q - n + lane_id()) * 16u) : "memory");
        __syncwarp();
        q -= n;
        one_record<LP, DIR, SKEW_DOMINATED, false>(p, c, v.x, v.y, v.z, v.w, lane_id() < n);
    };
    auto take = [&](uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, bool present) {
        const bool match = (((w1 ^ top_hi) & 0x00FFFFFFu) | (w2 ^ top_lo)) == 0u && w0 < p.n_apps && present;
        const uint32_t wgt = (p.appw_in_smem != 0) ? lds_u32(c.sb + L::APPW + (w0 & (APPW_SMEM_MAX - 1u)) * 4u) : __ldg(p.app_w + (match ? w0 : 0u));
        const ull prod = (ull)wgt * (ull)w3;
        const bool dom = match && (uint32_t)(prod >> 32) < 0x10000u;
        if (dom) {
            sum += prod;
            ++count;
        }
        const uint32_t others = __ballot_sync(0xFFFFFFFFu, present && !dom);
        if (present && !dom)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(queue + (q + __popc(others & lanes_below())) * 16u), "r"(w0), "r"(w1), "r"(w2), "r"(w3) : "memory");
        q += __popc(others);
        if (q >= 32) settle(32);
    };
    const unsigned char* body = reinterpret_cast<const unsigned char*>(p.body);
    const uint32_t stride = gridDim.x * SCATTER_THREADS;                  // pairs per round
    const uint32_t full_rounds = (uint32_t)(p.n_pairs / stride);
    const uint32_t rounds = (uint32_t)((p.n_pairs + stride - 1) / stride);
    const uint32_t first = blockIdx.x * SCATTER_THREADS + threadIdx.x;
    uint32_t bufA[8], bufB[8];
    auto fetch = [&](uint32_t round, uint32_t (&raw)[8]) {                // any round, bounds checked
        const ull i = first + (ull)round * stride;
        if (round < rounds && i < p.n_pairs) {
            ld_stream_256(body + i * 32, raw);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) raw[j] = 0;
        }
    };
    auto consume_full = [&](const uint32_t (&raw)[8]) {
        take(raw[0], raw[1], raw[2], raw[3], true);
        take(raw[4], raw[5], raw[6], raw[7], true);
    };
    auto consume_tail = [&](uint32_t round, const uint32_t (&raw)[8]) {
        const bool present = round < rounds && first + (ull)round * stride < p.n_pairs;
        take(raw[0], raw[1], raw[2], raw[3], present);
        take(raw[4], raw[5], raw[6], raw[7], present);
    };
    fetch(0, bufA);
    uint32_t round = 0;
    {   // two loads alternate (a third would not fit the registers), each behind an L2 prefetch of the round after it
        // (1 812 -> 1 559 us per 2^29 records; two rounds ahead 1 679); complete rounds need no checks
        const unsigned char* next = body + (first + (ull)stride) * 32;
        const uint32_t step = gridDim.x * (SCATTER_THREADS * 32u);
        for (; round + 4 <= full_rounds; round += 2) {
            ld_stream_256(next, bufB);
            if ((threadIdx.x & 3u) == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(next + step));
            next += step;
            consume_full(bufA);
            ld_stream_256(next, bufA);
            if ((threadIdx.x & 3u) == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(next + step));
            next += step;
            consume_full(bufB);
        }
    }
    for (; round < rounds; round += 2) {
        fetch(round + 1, bufB);
        consume_tail(round, bufA);
        fetch(round + 2, bufA);
        consume_tail(round + 1, bufB);
    }
    // records that do not form an aligned pair (at most one before and one after the body)
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        uint4 v = make_uint4(0, 0, 0, 0);
        const bool present = threadIdx.x < p.n_single;
        if (present) v = *reinterpret_cast<const uint4*>(threadIdx.x == 0 ? p.single[0] : p.single[1]);
        take(v.x, v.y, v.z, v.w, present);
    }
    if (q) settle(q);
    // the key's sum: lanes, warps, then one table update per CTA
    __shared__ ull s_lo, s_hi, s_count;
    if (threadIdx.x == 0) s_lo = s_hi = s_count = 0;
    __syncthreads();
    ull hi = 0, n = count;
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const ull o = __shfl_xor_sync(0xFFFFFFFFu, sum, d), s = sum + o;
        hi += __shfl_xor_sync(0xFFFFFFFFu, hi, d) + (s < sum ? 1ull : 0ull);
        sum = s;
        n += __shfl_xor_sync(0xFFFFFFFFu, n, d);
    }
    if (lane_id() == 0 && n) {
        const ull old = atomicAdd(&s_lo, sum);
        atomicAdd(&s_hi, hi + (old + sum < old ? 1ull : 0ull));
        atomicAdd(&s_count, n);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_count) table_accumulate(p.t, top, hash32(top), s_lo, s_hi, s_count);
}

// ---- shared-memory record ring (ATREX_SCATTER_RING stages) ----------------------------------------
// One warp of the CTA is the producer: a single lane issues one bulk asynchronous copy per tile of
// 992 records (this GPU's memory only, no multicast) into the next free stage and names the stage's
// "full" barrier as the copy's completion.  The other 31 warps are consumers: each thread reads its own
// record of two consecutive tiles (conflict-free 16-byte shared loads), the warp then releases the two
// stages on their "empty" barriers.  What the ring buys is registers: the records in flight live in
// shared memory, so a consumer thread holds only the two records it is working on.  Every wait is
// bounded; one that runs out latches ST_TIMEOUT, raises the CTA's abort flag and everybody leaves.
__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t a, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t a) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t a, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(a), "r"(parity)
                 : "memory");
    return ok != 0;
}
constexpr uint32_t RING_WAIT_TRIES = 1u << 22;
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, const volatile uint32_t* abort_flag) {
    for (uint32_t i = 0; i < RING_WAIT_TRIES; ++i) {
        if (mbar_try_wait(a, parity)) return true;
        if ((i & 63u) == 63u && *abort_flag) return false;
    }
    return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar, ull policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ uint4 lds_record(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}

template <uint32_t LP, int DIR, ull SKEW>
__device__ __forceinline__ void ring_body(const IngestParams& p, Ctx& c, ull* full_bar, ull* empty_bar, volatile uint32_t* abort_flag) {
    constexpr uint32_t S = SCATTER_RING_STAGES > 0 ? SCATTER_RING_STAGES : 1;
    constexpr uint32_t TILE_RECS = SCATTER_CONSUMER_WARPS * 32;
    const unsigned char* recs = reinterpret_cast<const unsigned char*>(p.recs);
    // tile T covers records [T * 992, (T + 1) * 992); CTA b takes tiles b, b + G, b + 2 G, ...
    const ull n_tiles = (p.n_recs + TILE_RECS - 1) / TILE_RECS;
    const uint32_t mine = blockIdx.x < n_tiles ? (uint32_t)((n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0u;
    const uint32_t fb = smem_addr(full_bar), eb = smem_addr(empty_bar);
    if (threadIdx.x >= TILE_RECS) {
        // producer warp
        if (threadIdx.x == TILE_RECS) {
            ull policy;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
            uint32_t issued = 0;
            for (uint32_t k = 0; k < mine; ++k, ++issued) {
                const uint32_t s = k % S;
                if (k >= S && !mbar_wait(eb + s * 8, ((k / S) - 1u) & 1u, abort_flag)) {
                    if (!*abort_flag) atomicOr(&p.t.ctl->status, ST_TIMEOUT);
                    *abort_flag = 1;
                    break;
                }
                const ull T = (ull)k * gridDim.x + blockIdx.x;
                const ull first = T * TILE_RECS;
                const uint32_t n_here = (uint32_t)(p.n_recs - first < TILE_RECS ? p.n_recs - first : TILE_RECS);
                mbar_expect_tx(fb + s * 8, n_here * 16u);
                bulk_load(c.sb + Smem<LP, DIR>::RING + s * SCATTER_RING_TILE, recs + first * 16, n_here * 16u, fb + s * 8, policy);
            }
            if (*abort_flag) {
                // leaving early: give the copies still in flight a (bounded) chance to land first
                for (uint32_t k = issued > S ? issued - S : 0; k < issued; ++k) {
                    bool done = false;
                    for (uint32_t i = 0; i < 4096 && !done; ++i) done = mbar_try_wait(fb + (k % S) * 8, (k / S) & 1u);
                }
            }
        }
        return;
    }
    // consumers: two tiles (two records per thread) at a time
    const uint32_t lane_off = threadIdx.x * 16u;
    for (uint32_t k = 0; k < mine; k += 2) {
        const uint32_t s0 = k % S, s1 = (k + 1) % S;
        const bool second = k + 1 < mine;
        bool ok = mbar_wait(fb + s0 * 8, (k / S) & 1u, abort_flag);
        if (ok && second) ok = mbar_wait(fb + s1 * 8, ((k + 1) / S) & 1u, abort_flag);
        if (!ok) {
            if (!*abort_flag) atomicOr(&p.t.ctl->status, ST_TIMEOUT);
            *abort_flag = 1;
            return;
        }
        const ull first0 = ((ull)k * gridDim.x + blockIdx.x) * TILE_RECS, first1 = first0 + (ull)gridDim.x * TILE_RECS;
        const bool p0 = first0 + threadIdx.x < p.n_recs, p1 = second && first1 + threadIdx.x < p.n_recs;
        uint4 r0 = make_uint4(0, 0, 0, 0), r1 = make_uint4(0, 0, 0, 0);
        if (p0) r0 = lds_record(c.sb + Smem<LP, DIR>::RING + s0 * SCATTER_RING_TILE + lane_off);
        if (p1) r1 = lds_record(c.sb + Smem<LP, DIR>::RING + s1 * SCATTER_RING_TILE + lane_off);
        __syncwarp();
        if ((threadIdx.x & 31u) == 0) {   // the warp has its records in registers: hand the stages back
            mbar_arrive(eb + s0 * 8);
            if (second) mbar_arrive(eb + s1 * 8);
        }
        const uint32_t w[2][4] = {{r0.x, r0.y, r0.z, r0.w}, {r1.x, r1.y, r1.z, r1.w}};
        const bool full = second && first1 + TILE_RECS <= p.n_recs;     // both tiles complete (uniform)
        if (full) {
            process<LP, DIR, SKEW, true, 2>(p, c, w, true);
        } else {
            // ragged end: one record at a time, each with its own mask
            const uint32_t wa[1][4] = {{r0.x, r0.y, r0.z, r0.w}}, wb[1][4] = {{r1.x, r1.y, r1.z, r1.w}};
            process<LP, DIR, SKEW, false, 1>(p, c, wa, p0);
            process<LP, DIR, SKEW, false, 1>(p, c, wb, p1);
        }
    }
}

struct RingBars {
    ull *full, *empty;
    volatile uint32_t* abort_flag;
};

// What a CTA does with the directory in the form DIR (empty: nothing is in it): loads it, goes through its records, stores cursors and sums.
template <uint32_t LP, int DIR>
__device__ __forceinline__ void scatter_cta(const IngestParams& p, Ctx& c, unsigned char* smem_raw, const RingBars& ring, bool empty) {
    using L = Smem<LP, DIR>;
    uint32_t* g_cursor = reinterpret_cast<uint32_t*>(smem_raw + L::CUR);
    uint32_t* g_acc = reinterpret_cast<uint32_t*>(smem_raw + L::ACC);
    const ull skew = DIR != DIR_NONE ? p.t.ctl->hot_skew : SKEW_NONE;
    if (L::W && threadIdx.x < 3) reinterpret_cast<uint32_t*>(smem_raw + L::LONG)[threadIdx.x] = 0;
    if (L::W) {
        for (uint32_t i = threadIdx.x; i < L::SLOTS / 4; i += blockDim.x) reinterpret_cast<uint4*>(smem_raw + L::WORDS)[i] = p.hot_words[i];
        for (uint32_t i = threadIdx.x; i < L::SLOTS * 3 / 4; i += blockDim.x) reinterpret_cast<uint4*>(g_acc)[i] = make_uint4(0, 0, 0, 0);
    } else if (DIR != DIR_NONE) {
        for (uint32_t i = threadIdx.x; i < L::SLOTS + L::PAD; i += blockDim.x) {
            const ull image = i < L::SLOTS && !empty ? p.hot_keys[i] : 0ull;   // ~key, 0 = empty
            reinterpret_cast<ull*>(smem_raw + L::KEYS)[i] = ~image;
            (smem_raw + L::TAG)[i] = image ? (unsigned char)(dir_mix(hash32(~image), (uint32_t)(~image >> 48) & 0xFFu, c.mult) & 0xFFu) : 0;
            g_acc[3 * i] = 0;
            g_acc[3 * i + 1] = 0;
            g_acc[3 * i + 2] = 0;
        }
    }
    __syncthreads();

    if (SCATTER_RING_STAGES > 0) {
        if (DIR != DIR_NONE && skew == SKEW_DOMINATED)
            ring_body<LP, DIR, SKEW_DOMINATED>(p, c, ring.full, ring.empty, ring.abort_flag);
        else if (DIR != DIR_NONE && skew == SKEW_COMBINE)
            ring_body<LP, DIR, SKEW_COMBINE>(p, c, ring.full, ring.empty, ring.abort_flag);
        else
            ring_body<LP, DIR, SKEW_NONE>(p, c, ring.full, ring.empty, ring.abort_flag);
    } else {
        if (DIR != DIR_NONE && skew == SKEW_DOMINATED)
            dominated_body<LP, DIR>(p, c);
        else if (DIR != DIR_NONE && skew == SKEW_COMBINE)
            scatter_body<LP, DIR, SKEW_COMBINE>(p, c);
        else
            scatter_body<LP, DIR, SKEW_NONE>(p, c);
    }

    grid_dependents_launch();
    __syncthreads();
    const uint32_t cap = L::W ? p.short_cap : p.cap;
    uint32_t drain_above = L::W ? p.short_drain_above : p.drain_above;
    // (where three eighths of the launch's records took two entries, the next launch may bring two entries for each of its)
    if (L::W && (ull)*reinterpret_cast<const uint32_t*>(smem_raw + L::LONG) * gridDim.x >= p.n_pairs / 4 * 3) drain_above = p.long_drain_above;
    uint32_t spilled = 0, fullest = 0;
    bool crowded = false;
    if (L::W && threadIdx.x == 0) {
        spilled = 0u - *reinterpret_cast<const uint32_t*>(smem_raw + L::LONG);      // (records, not entries)
        if (*reinterpret_cast<const uint32_t*>(smem_raw + L::RESTS)) p.t.ctl->rests = 1;
        const uint32_t misfits = *reinterpret_cast<const uint32_t*>(smem_raw + L::MISFITS);
        if (misfits) atomicAdd(&p.t.ctl->n_misfit, (ull)misfits);
    }
    for (uint32_t i = threadIdx.x; i < L::P; i += blockDim.x) {
        const size_t at = ((size_t)blockIdx.x << LP) + i;
        const uint32_t before = p.spill_cnt[at], n = min(g_cursor[i], cap);
        p.spill_cnt[at] = n;
        spilled += n - before;
        crowded |= n > drain_above;
        fullest = max(fullest, n);
    }
    fullest = __reduce_max_sync(0xFFFFFFFFu, fullest);
    spilled = __reduce_add_sync(0xFFFFFFFFu, spilled);
    crowded = __any_sync(0xFFFFFFFFu, crowded);
    if ((threadIdx.x & 31u) == 0) {
        if (spilled) atomicAdd(&p.t.ctl->n_spilled, (ull)(long long)(int32_t)spilled);   // (the first warp's may be negative)
        // a buffer is filling up: have the partition pass that follows this launch drain them
        if (crowded) atomicMax(&p.t.ctl->drain_seq, p.seq);
        atomicMax(&p.t.ctl->max_fill, (ull)fullest);
    }
    if (DIR != DIR_NONE) {
        // This launch's directory sums go to the CTA's own row of the directory image: plain coalesced
        // read-modify-writes, no atomics (148 CTAs adding the same few thousand keys into the table at
        // the end of every launch cost 59 us per launch).  hot_fold_kernel adds the rows into the table
        // before results are read.
        ulonglong2* img = p.hot_img + (size_t)blockIdx.x * p.hot_slots;
        const bool held = blockIdx.x < p.img_rows;   // the row holds earlier launches' sums
        const uint32_t in_use = skew == SKEW_DOMINATED ? L::SLOTS_DOM : L::SLOTS;
        for (uint32_t i0 = threadIdx.x; i0 < p.hot_slots; i0 += 4 * blockDim.x) {  // four slots per thread in flight
            uint32_t cn[4], lo[4], hi[4];
            ulonglong2 o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * blockDim.x;
                const bool in = i < in_use;
                lo[u] = in ? g_acc[3 * i] : 0u;
                hi[u] = in ? g_acc[3 * i + 1] : 0u;
                cn[u] = in ? g_acc[3 * i + 2] : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) o[u] = held && (cn[u] | lo[u] | hi[u]) ? img[i0 + u * blockDim.x] : make_ulonglong2(0, 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (i0 + u * blockDim.x >= p.hot_slots || (held && (cn[u] | lo[u] | hi[u]) == 0)) continue;
                const ull nlo = o[u].x + ((ull)lo[u] | ((ull)hi[u] << 32));
                img[i0 + u * blockDim.x] = make_ulonglong2(nlo, o[u].y + (ull)cn[u] + ((nlo < o[u].x ? 1ull : 0ull) << HI_SHIFT));
            }
        }
    }
}

template <uint32_t LP, bool HOT>
__global__ void __launch_bounds__(SCATTER_THREADS, 1) scatter_kernel(IngestParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using L = Smem<LP, DIR_NONE>;                  // (what is used of it here is the same in every form)
    uint32_t* g_cursor = reinterpret_cast<uint32_t*>(smem_raw + L::CUR);
    uint32_t* g_appw = reinterpret_cast<uint32_t*>(smem_raw + L::APPW);

    __shared__ __align__(8) ull s_full[SCATTER_RING_STAGES ? SCATTER_RING_STAGES : 1], s_empty[SCATTER_RING_STAGES ? SCATTER_RING_STAGES : 1];
    __shared__ uint32_t s_abort;
    if (SCATTER_RING_STAGES > 0 && threadIdx.x == 0) {
        for (uint32_t i = 0; i < SCATTER_RING_STAGES; ++i) {
            mbar_init(smem_addr(&s_full[i]), 1);                          // the producer's arrive + the copy's bytes
            mbar_init(smem_addr(&s_empty[i]), SCATTER_CONSUMER_WARPS);    // one arrive per consumer warp
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }

    grid_dependency_wait();
    Ctx c;
    c.sb = smem_addr(smem_raw);
    c.mult = HOT ? (uint32_t)p.t.ctl->dir_mult : 1u;
    c.my_spill = p.spill + ((size_t)blockIdx.x << LP) * p.cap * SPILL_ENTRY_BYTES;   // (as many bytes as short_cap short entries)
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(c.keep));

    // The buffers persist across launches until the partition pass drains them: resume the cursors.
    for (uint32_t i = threadIdx.x; i < L::P; i += blockDim.x) g_cursor[i] = p.spill_cnt[((size_t)blockIdx.x << LP) + i];
    if (p.appw_in_smem != 0)
        for (uint32_t i = threadIdx.x; i < p.n_apps; i += blockDim.x) g_appw[i] = p.app_w[i];
    const RingBars ring = {s_full, s_empty, &s_abort};
    const ull form = HOT ? p.t.ctl->form : FORM_LONG_ONLY;
    if (!HOT)
        scatter_cta<LP, DIR_NONE>(p, c, smem_raw, ring, true);
    else if (SCATTER_RING_STAGES == 0 && form == FORM_SHORT)
        scatter_cta<LP, DIR_WORDS>(p, c, smem_raw, ring, false);
    else
        scatter_cta<LP, DIR_TAGS>(p, c, smem_raw, ring, form == FORM_LONG_ONLY);
}

template <uint32_t LP>
cudaError_t prepare_lp() {
    cudaError_t e = cudaFuncSetAttribute(scatter_kernel<LP, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)SCATTER_SMEM_BYTES);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(scatter_kernel<LP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)SCATTER_SMEM_BYTES);
}

template <uint32_t LP>
cudaError_t launch_lp(const IngestParams& p, bool hot, int grid, cudaStream_t stream) {
    return launch_chained(hot ? scatter_kernel<LP, true> : scatter_kernel<LP, false>, (uint32_t)grid, SCATTER_THREADS, smem_total<LP>(), stream, p);
}

}  // namespace

cudaError_t scatter_prepare() {
    cudaError_t e = prepare_lp<8>();
    if (e == cudaSuccess) e = prepare_lp<9>();
    if (e == cudaSuccess) e = prepare_lp<10>();
    if (e == cudaSuccess) e = prepare_lp<11>();
    if (e == cudaSuccess) e = prepare_lp<12>();
    return e;
}

cudaError_t launch_scatter(const IngestParams& p, bool hot, int grid, cudaStream_t stream) {
    if (hot && p.hot_slots != scatter_hot_slots(p.t.lp)) return cudaErrorInvalidValue;
    switch (p.t.lp) {
        case 8: return launch_lp<8>(p, hot, grid, stream);
        case 9: return launch_lp<9>(p, hot, grid, stream);
        case 10: return launch_lp<10>(p, hot, grid, stream);
        case 11: return launch_lp<11>(p, hot, grid, stream);
        case 12: return launch_lp<12>(p, hot, grid, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace atrex
