// Roofline score aggregation (Eq. 4-6), batched over candidates.
//
//   Eq. 4  S_j = T_roofline,j / T_cand,j for units that passed correctness (a value above 1, or a
//          candidate time that is not a finite positive number, is counted as an evaluation
//          error; values above 1 are not clipped, unusable times are left out)
//   Eq. 5  S_i = median over operator i's correct shapes (even count: mean of the middle two),
//          0 when there is none
//   Eq. 6  S_agg = sum_i w_i S_i, accumulated in operator order
//
// Every floating-point step of a result is one explicit round-to-nearest operation in a fixed order, so
// the result has one bit pattern.
//
// Where a unit goes when units are grouped by operator is the same for every candidate, so a CTA works
// that out once and then goes through its candidates.  Three kernels:
//   score_warp_kernel  one candidate per warp, no barriers: many candidates of few units
//   score_cta_kernel   one candidate per CTA: few candidates, or more units than a warp should hold
//   score_bins_kernel  one candidate per CTA, no grouping: operators of 64 units and more, but for many candidates of up to 500 units
// The kernel before these (one candidate per CTA, grouping redone for every candidate, exact scores ranked
// against each other) was bound by its barriers and shared-memory atomics: 65 536 candidates x 440 units x
// 30 operators in 594 us, 1 000 x 12 001 units x 7 operators in 1 179 us.
//
// Ranking does not need exact quotients.  A unit's approximate score is formed in binary32 -- two
// conversions, a reciprocal and a product, within six units in the last place of the exact quotient -- and
// its bit pattern is the key; only the one or two middle units of an operator are divided in binary64.
// That is right as long as no other key of the operator is close to a middle one: then the middle units by
// key are the middle units by score.  Where one is (ties among them), or an operand is outside the range
// the approximation is good for, the operator's candidates for the middle are ranked by exact quotients.
#include <cmath>
#include <mutex>
#include <utility>

#include "kernels.h"

using namespace atrex;

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t SELECT_BINS = 128;

// Order-preserving key of an exact score: a double's bit pattern with the sign bit flipped for positive values
// and all bits flipped for negative ones.  Any NaN (a unit without a roofline) gets one pattern, above +inf.
__device__ __forceinline__ ull key_of_score(double x) {
    if (x != x) return 0xFFF8000000000000ull;
    const ull b = (ull)__double_as_longlong(x);
    return b ^ ((b >> 63) ? ~0ull : (1ull << 63));
}
__device__ __forceinline__ double score_of_key(ull k) { return __longlong_as_double((long long)(k ^ ((k >> 63) ? (1ull << 63) : ~0ull))); }
__device__ __forceinline__ double median_of_keys(ull lo, ull hi, bool odd) {
    const double h = score_of_key(hi);
    return odd ? h : __dmul_rn(__dadd_rn(score_of_key(lo), h), 0.5);
}
// Eq. 4 for one unit: its exact key, or all ones where it has no usable score.
__device__ __forceinline__ ull exact_key(double roofline, double t, bool ok) {
    return ok && t > 0.0 && !isinf(t) ? key_of_score(__ddiv_rn(roofline, t)) : ~0ull;
}

constexpr uint32_t K_ABSENT = 0x7FFFFFFFu;       // no usable score: sorts last
constexpr uint32_t K_UNKNOWN = 0x7FFFFFC0u;      // usable, but outside the approximation's range (above every approximation)
constexpr uint32_t K_APART = 16;                 // keys further apart than this are in the order of the exact scores
// Operands between 2^-60 and 2^60 keep every step of the approximation a normal number.
constexpr uint32_t SAFE_LOW = (1023u - 60u) << 20, SAFE_SPAN = 120u << 20;
__device__ __forceinline__ bool in_safe_range(double x) { return (uint32_t)__double2hiint(x) - SAFE_LOW < SAFE_SPAN; }
__device__ __forceinline__ float approx_roofline(double r) { return in_safe_range(r) ? (float)r : __int_as_float(0x7FFFFFFF); }

// Key of one unit and its evaluation errors; `r` = approx_roofline(*roofline), no branch on the usual way.
__device__ __forceinline__ uint32_t approx_key(float r, const double* roofline, double t, bool use, uint32_t& errors) {
    uint32_t key = (uint32_t)__float_as_int(__fdividef(r, (float)t));
    // fl(roofline / t) > 1 exactly when roofline > t; the approximation settles it away from 1
    const bool special = !in_safe_range(t) | (key > 0x3F800000u - K_APART);   // (a NaN is far above)
    key = use ? key : K_ABSENT;
    if (use & special) {
        if (!(t > 0.0) || isinf(t)) {
            key = K_ABSENT;
            ++errors;
        } else {
            if (!in_safe_range(t) || r != r) key = K_UNKNOWN;
            errors += __ldg(roofline) > t ? 1u : 0u;
        }
    }
    return key;
}

// The k-th and (k+1)-th smallest (from 0) of the usable keys among the g keys key_at(0 .. g - 1), by one warp:
// the range that holds the k-th is cut into up to 128 equal bins, counted, and narrowed to one bin until
// that bin's keys fit the lanes (two rounds for a thousand spread-out values), where they are ranked.
// A range of one value ends the search as well, so ties cost nothing; each round narrows the range at
// least 64-fold, so there are at most eleven.  K: 32- or 64-bit keys, all ones = no usable score.
// `bins`: SELECT_BINS words of this warp's.  (In place, or as a call.)
template <typename K, typename KeyAt>
__device__ __forceinline__ void warp_select_here(KeyAt key_at, uint32_t g, uint32_t k, uint32_t* bins, K* out_k, K* out_next) {
    constexpr K NONE = ~(K)0;
    const uint32_t lane = threadIdx.x & 31u;
    K lo = NONE, hi = 0;
#pragma unroll 4
    for (uint32_t a = lane; a < g; a += 32) {
        const K x = key_at(a);
        if (x == NONE) continue;
        lo = min(lo, x);
        hi = max(hi, x);
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        lo = min(lo, __shfl_xor_sync(FULL, lo, d));
        hi = max(hi, __shfl_xor_sync(FULL, hi, d));
    }
    K next_above = NONE;         // smallest key above the current range
    while (lo != hi) {
        const int len = 64 - __clzll((long long)(ull)(hi - lo));
        const int shift = len > 7 ? len - 7 : 0;
        reinterpret_cast<uint4*>(bins)[lane] = make_uint4(0, 0, 0, 0);
        __syncwarp();
#pragma unroll 4
        for (uint32_t a = lane; a < g; a += 32) {
            const K x = key_at(a);
            if (x >= lo && x <= hi) atomicAdd(&bins[(uint32_t)((x - lo) >> shift)], 1u);
        }
        __syncwarp();
        const uint4 c = reinterpret_cast<const uint4*>(bins)[lane];
        const uint32_t own = c.x + c.y + c.z + c.w;
        uint32_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(FULL, incl, d);
            if (lane >= (uint32_t)d) incl += o;
        }
        const uint32_t src = __ffs(__ballot_sync(FULL, incl > k)) - 1;   // the lane whose four bins hold the k-th
        uint32_t before = incl - own, bin = lane * 4, n = c.x;
        if (k >= before + n) { before += n; ++bin; n = c.y; if (k >= before + n) { before += n; ++bin; n = c.z; if (k >= before + n) { before += n; ++bin; n = c.w; } } }
        bin = __shfl_sync(FULL, bin, src);
        k -= __shfl_sync(FULL, before, src);
        n = __shfl_sync(FULL, n, src);
        __syncwarp();   // the bins are reused
        lo += (K)bin << shift;
        hi = min(hi, lo + (((K)1 << shift) - 1));
        if (n <= 32) break;
    }
    // keys in [lo, hi] to the lanes (at most 32 unless the range is one value), and the smallest key above it
    uint32_t n = 0;
    K* list = reinterpret_cast<K*>(bins);
#pragma unroll 4
    for (uint32_t a0 = 0; a0 < g; a0 += 32) {
        const K x = a0 + lane < g ? key_at(a0 + lane) : NONE;
        const bool in = x >= lo && x <= hi;
        if (x > hi) next_above = min(next_above, x);
        const uint32_t votes = __ballot_sync(FULL, in);
        const uint32_t pos = n + __popc(votes & ((1u << lane) - 1u));
        if (in && pos < 32) list[pos] = x;
        n += __popc(votes);
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) next_above = min(next_above, __shfl_xor_sync(FULL, next_above, d));
    __syncwarp();
    if (lo == hi) {
        *out_k = lo;
        *out_next = k + 1 < n ? lo : next_above;
    } else {
        const K x = lane < n ? list[lane] : NONE;
        uint32_t less = 0, leq = 0;
        for (uint32_t b = 0; b < n; ++b) {
            const K y = list[b];
            less += y < x ? 1u : 0u;
            leq += y <= x ? 1u : 0u;
        }
        const uint32_t at_k = __ffs(__ballot_sync(FULL, lane < n && less <= k && k < leq)) - 1;
        *out_k = __shfl_sync(FULL, x, at_k);
        const uint32_t at_next = __ballot_sync(FULL, lane < n && less <= k + 1 && k + 1 < leq);
        const K in_list = __shfl_sync(FULL, x, at_next ? __ffs(at_next) - 1 : 0);
        *out_next = k + 1 < n ? in_list : next_above;
    }
    __syncwarp();   // `bins` may be overwritten from here on
}

template <typename K, typename KeyAt>
__device__ __noinline__ void warp_select(KeyAt key_at, uint32_t g, uint32_t k, uint32_t* bins, K* out_k, K* out_next) {
    warp_select_here<K>(key_at, g, k, bins, out_k, out_next);
}

// The middle of one operator's keys, by one warp: number of usable units, the lower and upper middle keys (no
// key lies between them), how many keys are within K_APART of them, how many are below those.
struct Middle {
    uint32_t m, v_lo, v_up, close, below;
    bool unknown;                                       // a key outside the approximation's range: nothing else is valid
    __device__ __forceinline__ uint32_t from() const { return v_lo - K_APART; }
    __device__ __forceinline__ uint32_t span() const { return v_up - v_lo + 2 * K_APART; }
    __device__ __forceinline__ bool clear() const { return close == 2 - (m & 1u) && ((m & 1u) || v_up - v_lo > K_APART); }
};

// Up to 32 R keys held in registers.  Up to 32 keys, each lane counts how many are below its own (the k-th is the
// largest that has at most k below it); above, where that would take more instructions, the range of the wanted
// key is halved (a count over the warp each time) until one key is left in it.
template <int R>
__device__ __forceinline__ Middle middle_in_registers(const uint32_t* keys, uint32_t g) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t x[R], least = ~0u, most = 0, usable = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t a = lane + 32 * r;
        x[r] = a < g ? keys[a] : K_ABSENT;
        least = min(least, x[r]);
        most = max(most, x[r] == K_ABSENT ? 0u : x[r]);
        usable += x[r] != K_ABSENT ? 1u : 0u;
    }
    Middle d;
    d.m = __reduce_add_sync(FULL, usable);
    uint32_t lo = __reduce_min_sync(FULL, least), hi = __reduce_max_sync(FULL, most);
    d.unknown = hi == K_UNKNOWN;
    d.v_lo = d.v_up = d.close = d.below = 0;
    if (d.m == 0 || d.unknown) return d;
    const uint32_t k = (d.m - 1) / 2;
    if constexpr (R == 1) {
        uint32_t less[R] = {}, at_lo = 0, at_up = 0;
#pragma unroll 8
        for (uint32_t b = 0; b < g; ++b) {
            const uint32_t y = keys[b];
#pragma unroll
            for (int r = 0; r < R; ++r) less[r] += y < x[r] ? 1u : 0u;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (x[r] == K_ABSENT) continue;
            at_lo = max(at_lo, less[r] <= k ? x[r] : 0u);
            at_up = max(at_up, less[r] <= d.m / 2 ? x[r] : 0u);
        }
        d.v_lo = __reduce_max_sync(FULL, at_lo);
        d.v_up = __reduce_max_sync(FULL, at_up);
    } else {
        uint32_t before = 0, through = d.m;    // keys below lo, keys up to hi
        while (through - before > 1 && lo < hi) {
            const uint32_t half = lo + (hi - lo) / 2 + 1;
            uint32_t c = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) c += x[r] < half ? 1u : 0u;
            c = __reduce_add_sync(FULL, c);
            if (k < c) {
                hi = half - 1;
                through = c;
            } else {
                lo = half;
                before = c;
            }
        }
        uint32_t v = ~0u;
#pragma unroll
        for (int r = 0; r < R; ++r) v = min(v, x[r] >= lo ? x[r] : ~0u);
        d.v_lo = d.v_up = __reduce_min_sync(FULL, v);
        if (!(d.m & 1u)) {
            uint32_t leq = 0, up = ~0u;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                leq += x[r] <= d.v_lo ? 1u : 0u;
                up = min(up, x[r] > d.v_lo ? x[r] : ~0u);
            }
            up = __reduce_min_sync(FULL, up);
            if (__reduce_add_sync(FULL, leq) == k + 1) d.v_up = up;
        }
    }
    uint32_t close = 0, below = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        close += x[r] - d.from() <= d.span() ? 1u : 0u;
        below += x[r] < d.from() ? 1u : 0u;
    }
    d.close = __reduce_add_sync(FULL, close);
    d.below = __reduce_add_sync(FULL, below);
    return d;
}

__device__ __noinline__ Middle group_middle(const uint32_t* keys, uint32_t g, uint32_t* bins) {
    if (g <= 32) return middle_in_registers<1>(keys, g);
    if (g <= 64) return middle_in_registers<2>(keys, g);
    if (g <= 128) return middle_in_registers<4>(keys, g);
    if (g <= 256) return middle_in_registers<8>(keys, g);
    const uint32_t lane = threadIdx.x & 31u;
    Middle d;
    uint32_t m = 0, unknown = 0;
#pragma unroll 4
    for (uint32_t a = lane; a < g; a += 32) {
        const uint32_t x = keys[a];
        m += x != K_ABSENT ? 1u : 0u;
        unknown |= x == K_UNKNOWN ? 1u : 0u;
    }
    d.m = __reduce_add_sync(FULL, m);
    d.unknown = __any_sync(FULL, unknown);
    d.v_lo = d.v_up = d.close = d.below = 0;
    if (d.m == 0 || d.unknown) return d;
    uint32_t next;
    warp_select<uint32_t>([=](uint32_t a) { const uint32_t k = keys[a]; return k == K_ABSENT ? ~0u : k; }, g, (d.m - 1) / 2, bins, &d.v_lo, &next);
    d.v_up = (d.m & 1u) ? d.v_lo : next;
    uint32_t close = 0, below = 0;
#pragma unroll 4
    for (uint32_t a = lane; a < g; a += 32) {
        const uint32_t x = keys[a];
        close += x - d.from() <= d.span() ? 1u : 0u;
        below += x < d.from() ? 1u : 0u;
    }
    d.close = __reduce_add_sync(FULL, close);
    d.below = __reduce_add_sync(FULL, below);
    return d;
}

// Sizes of the operators' groups (whole CTA).
__device__ __forceinline__ void count_groups(const uint32_t* __restrict__ unit_op, uint32_t n_units, uint32_t n_ops, uint32_t* size) {
    for (uint32_t i = threadIdx.x; i < n_ops; i += blockDim.x) size[i] = 0;
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < n_units; j += blockDim.x) {
        const uint32_t op = unit_op[j];
        if (op < n_ops) atomicAdd(&size[op], 1u);
    }
    __syncthreads();
}

// ---- one candidate per warp ---------------------------------------------------------------------
// Bound by the integer pipe.  A lane sorts its operator's keys in registers (up to 32, a pruned odd-even
// merge network: two instructions per comparator, no divergence; each key carries its slot in its low five
// bits).  Groups above 32 are searched by the whole warp, operators whose keys cannot decide on exact
// quotients.  65 536 candidates x 440 units x 30 operators: 145 us (1 410 warp instructions per candidate,
// half of the issue slots; the inputs alone take 42 us); ranking exact keys by counting took 4 050
// instructions and 319 us.
constexpr uint32_t NET_MAX = 32;                 // largest group that a lane sorts
constexpr uint32_t K_SLOT = 31u;                 // low bits of a lane's keys: their slots
constexpr uint32_t NET_APART = 64;               // keys with slots: further apart than this is the order of the exact scores

// Ascending sort of v[0 .. N - 1]: Batcher's odd-even merge network for 32 with the comparators beyond N left
// out, spelled out at compile time (an index that is not a constant would put v in local memory).
template <int N>
struct Network {
    int n = 0, a[191] = {}, b[191] = {};
    constexpr Network() {
        for (int p = 1; p < 32; p *= 2)
            for (int k = p; k >= 1; k /= 2)
                for (int j = k % p; j + k < 32; j += 2 * k)
                    for (int i = 0; i < k; ++i)
                        if ((i + j) / (2 * p) == (i + j + k) / (2 * p) && i + j + k < N) {
                            a[n] = i + j;
                            b[n++] = i + j + k;
                        }
    }
};
template <int A, int B, int N>
__device__ __forceinline__ void compare_exchange(uint32_t (&v)[N]) {
    const uint32_t x = v[A], y = v[B];
    v[A] = min(x, y);
    v[B] = max(x, y);
}
template <int N, int... I>
__device__ __forceinline__ void sort_steps(uint32_t (&v)[N], std::integer_sequence<int, I...>) {
    constexpr Network<N> net;
    (compare_exchange<net.a[I], net.b[I]>(v), ...);
}
template <int N>
__device__ __forceinline__ void sort_network(uint32_t (&v)[N]) {
    constexpr Network<N> net;
    sort_steps(v, std::make_integer_sequence<int, net.n>());
}

// One lane's operator: N keys at col[0], col[32], ..., the unused ones absent (sorted in place).  Returns the number of usable units; the slots of the lower and upper middle in `low` and `up`; `search`
// where the keys cannot decide.
template <int N>
__device__ __forceinline__ uint32_t middle_slots(uint32_t* col, uint32_t& low, uint32_t& up, bool& search) {
    uint32_t v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = (col[32 * i] & ~K_SLOT) | (uint32_t)i;
    sort_network<N>(v);
#pragma unroll
    for (int i = 0; i < N; ++i) col[32 * i] = v[i];
    // (an absent unit's key has a slot in its low bits too: absent means at or above K_ABSENT without them)
    uint32_t m = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1)
        if (m + step <= N) m += col[32 * (m + step - 1)] < (K_ABSENT & ~K_SLOT) ? step : 0;
    if (N == 32 && m == 31 && col[32 * 31] < (K_ABSENT & ~K_SLOT)) m = 32;
    low = up = 0;
    search = false;
    if (m == 0) return 0;
    const uint32_t kl = (m - 1) / 2, ku = m / 2;
    const uint32_t vl = col[32 * kl], vu = col[32 * ku];
    const uint32_t below = kl > 0 ? col[32 * (kl - 1)] : 0u, above = ku + 1 < m ? col[32 * (ku + 1)] : K_ABSENT;
    search = col[32 * (m - 1)] >= K_UNKNOWN || (kl > 0 && vl - below <= NET_APART) || (kl != ku && vu - vl <= NET_APART) ||
             above - vu <= NET_APART;
    low = vl & K_SLOT;
    up = vu & K_SLOT;
    return m;
}

// Two lanes' operator: each of the pair sorts its own column of N keys, then both walk the two columns from the
// place where the middle begins (a binary search: `below` keys of the union lie before it).  `low` and `up`
// are slots counted from the pair's first column, in steps of one column and 32 per row.
template <int N>
__device__ __forceinline__ uint32_t middle_slots_of_pair(uint32_t* col, uint32_t& low, uint32_t& up, bool& search) {
    {
        uint32_t v[N];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = (col[32 * i] & ~K_SLOT) | (uint32_t)i;
        sort_network<N>(v);
#pragma unroll
        for (int i = 0; i < N; ++i) col[32 * i] = v[i];
    }
    uint32_t own = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1)
        if (own + step <= N) own += col[32 * (own + step - 1)] < (K_ABSENT & ~K_SLOT) ? step : 0;
    if (N == 32 && own == 31 && col[32 * 31] < (K_ABSENT & ~K_SLOT)) own = 32;
    const uint32_t most = own ? col[32 * (own - 1)] : 0u;
    __syncwarp();
    const bool odd = threadIdx.x & 1u;
    const uint32_t other = __shfl_xor_sync(FULL, own, 1), ma = odd ? other : own, mb = odd ? own : other, m = ma + mb;
    const uint32_t highest = max(most, __shfl_xor_sync(FULL, most, 1));
    low = up = 0;
    search = false;
    if (m == 0) return 0;
    const uint32_t *a = odd ? col - 1 : col, *b = a + 1;
    const uint32_t kl = (m - 1) / 2, t = kl > 0 ? kl - 1 : 0u;
    uint32_t i = t > mb ? t - mb : 0u, end = min(t, ma);    // how many of the first t come from column a
    while (i < end) {
        const uint32_t half = (i + end) / 2;
        if (a[32 * half] < b[32 * (t - half - 1)]) i = half + 1;
        else end = half;
    }
    uint32_t j = t - i;
    uint32_t x = i < ma ? a[32 * i] : K_ABSENT, y = j < mb ? b[32 * j] : K_ABSENT;
    uint32_t slot = 0;
    auto next = [&] {                                        // the next key of the union; K_ABSENT behind the last one
        const bool from_a = x <= y;
        const uint32_t k = from_a ? x : y;
        slot = 32 * (k & K_SLOT) + (from_a ? 0u : 1u);
        if (from_a) {
            ++i;
            x = i < ma ? a[32 * i] : K_ABSENT;
        } else {
            ++j;
            y = j < mb ? b[32 * j] : K_ABSENT;
        }
        return k;
    };
    uint32_t before = 0;
    if (kl > 0) before = next();
    const uint32_t vl = next();
    low = up = slot;
    uint32_t vu = vl;
    if (!(m & 1u)) {
        vu = next();
        up = slot;
    }
    const uint32_t above = m / 2 + 1 < m ? next() : K_ABSENT;
    search = highest >= K_UNKNOWN || (kl > 0 && vl - before <= NET_APART) || (!(m & 1u) && vu - vl <= NET_APART) || above - vu <= NET_APART;
    return m;
}

template <bool PAIRS, int N>
__device__ __forceinline__ uint32_t middle_of(uint32_t* col, uint32_t& low, uint32_t& up, bool& search) {
    if constexpr (PAIRS) return middle_slots_of_pair<N>(col, low, up, search);
    else return middle_slots<N>(col, low, up, search);
}

constexpr uint32_t WARP_ILP = 4;           // units per lane in flight
__host__ __device__ __forceinline__ uint32_t padded_units(uint32_t n) { return (n + 32u * WARP_ILP - 1u) / (32u * WARP_ILP) * (32u * WARP_ILP); }

struct WarpLayout {   // byte offsets; from `prod` on relative to the warp's own block (which starts with its keys)
    uint32_t roof, place, group, chunk, unit_at, warps, prod, bins, warp_bytes;
    __host__ __device__ WarpLayout(uint32_t n, uint32_t n_ops, uint32_t slots) {
        uint32_t o = 0;
        roof = o;    o += 4u * padded_units(n);            // f32 rooflines, NaN outside the safe range
        group = o;   o += 8u * n_ops;                      // {first list entry (large groups), size | large << 31}
        chunk = o;   o += 4u * ((n_ops + 15u) / 16u + 1u); // first slot of each chunk of 32 (pairs: 16) operators
        place = o;   o += 2u * padded_units(n);            // slot of each unit, NO_GROUP flag
        unit_at = o; o += 2u * (slots + n);                // unit of each slot; behind the columns, the large groups' units
        warps = (o + 15u) & ~15u;
        o = 4u * (slots + n + 1u);
        bins = o = (o + 15u) & ~15u;  o += 4u * SELECT_BINS;
        prod = o;    o += 8u * n_ops;
        warp_bytes = (o + 15u) & ~15u;
    }
};
// Columns come in the lengths of the networks.
__host__ __device__ __forceinline__ uint32_t column_length(uint32_t g) { return g <= 8 ? 8u : (g <= 16 ? 16u : (g + 3u) & ~3u); }
// Slots to provide: the group sizes are in device memory, so every chunk of operators gets room for groups
// three standard deviations above the mean (units falling to operators at random); what does not fit is
// treated as a large group.
inline uint32_t warp_slots(uint32_t n, uint32_t n_ops, bool pairs) {
    const double mean = (double)n / n_ops;
    double width = std::ceil(mean + 3.0 * std::sqrt(mean)) + 2.0;
    if (pairs) width = std::ceil(mean * 0.5 + 1.5 * std::sqrt(mean)) + 1.0;
    if (mean > (pairs ? 2 * NET_MAX : NET_MAX)) width = 8;         // (hardly any group is small enough)
    if (width > NET_MAX) width = NET_MAX;
    const uint32_t per_chunk = pairs ? 16u : 32u;
    return (n_ops + per_chunk - 1u) / per_chunk * 32u * column_length((uint32_t)width);
}

constexpr uint32_t NO_GROUP = 0x8000u;     // flag of a unit of an operator outside [0, n_ops)
constexpr uint32_t SLOT_MASK = 0x7FFFu;    // (units without a group write to a slot behind all others)
constexpr uint32_t WARP_KERNEL_THREADS = 256, WARP_KERNEL_CTAS = 3;   // per SM (80 registers a thread; four CTAs of 64 were 3 % slower)

template <bool PAIRS>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS, WARP_KERNEL_CTAS)
    score_warp_kernel(const double* __restrict__ roofline_s, const uint32_t* __restrict__ unit_op, uint32_t n_units,
                      const double* __restrict__ t_cand, const uint8_t* __restrict__ correct, uint32_t n_cand,
                      const double* __restrict__ w, uint32_t n_ops, uint32_t max_slots, double* s_agg, double* s_op_out, ull* errors_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr uint32_t PER_CHUNK = PAIRS ? 16 : 32, LANES = PAIRS ? 2 : 1;
    const WarpLayout L(n_units, n_ops, max_slots);
    float* roof = reinterpret_cast<float*>(smem_raw + L.roof);
    uint16_t* place = reinterpret_cast<uint16_t*>(smem_raw + L.place);
    uint2* group = reinterpret_cast<uint2*>(smem_raw + L.group);
    uint32_t* chunk = reinterpret_cast<uint32_t*>(smem_raw + L.chunk);
    uint16_t* unit_at = reinterpret_cast<uint16_t*>(smem_raw + L.unit_at);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, n_warps = blockDim.x >> 5;
    unsigned char* mine = smem_raw + L.warps + warp * L.warp_bytes;
    uint32_t* keys = reinterpret_cast<uint32_t*>(mine);
    uint32_t* bins = reinterpret_cast<uint32_t*>(mine + L.bins);
    double* prod = reinterpret_cast<double*>(mine + L.prod);

    // where each unit goes: operators in chunks of 32, one lane's column each
    uint32_t* size = reinterpret_cast<uint32_t*>(smem_raw + L.warps + L.prod);   // [n_ops], in the first warp's block for now
    for (uint32_t j = threadIdx.x; j < padded_units(n_units); j += blockDim.x) {
        roof[j] = approx_roofline(j < n_units ? roofline_s[j] : 0.0);
        if (j >= n_units) place[j] = (uint16_t)((max_slots + n_units) | NO_GROUP);
    }
    count_groups(unit_op, n_units, n_ops, size);
    if (threadIdx.x < 32) {
        uint32_t slot = 0, large = 0;
        for (uint32_t op0 = 0; op0 < n_ops; op0 += PER_CHUNK) {
            const uint32_t op = op0 + lane;
            const bool mine = lane < PER_CHUNK && op < n_ops;
            const uint32_t g = mine ? size[op] : 0u, rows = (g + LANES - 1) / LANES;
            const bool is_large = rows > NET_MAX || slot + 32 * column_length(rows) > max_slots;
            const uint32_t widest = __reduce_max_sync(FULL, is_large ? 0u : rows);
            uint32_t incl = is_large ? g : 0u;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(FULL, incl, d);
                if (lane >= (uint32_t)d) incl += o;
            }
            if (mine) {
                group[op] = is_large ? make_uint2(max_slots + large + incl - g, g | 0x80000000u) : make_uint2(0u, g);
                size[op] = 0;
            }
            if (lane == 0) chunk[op0 / PER_CHUNK] = slot;
            slot += widest ? 32 * column_length(widest) : 0u;
            large += __shfl_sync(FULL, incl, 31);
        }
        if (lane == 0) chunk[(n_ops + PER_CHUNK - 1) / PER_CHUNK] = slot;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < n_units; j += blockDim.x) {
        const uint32_t op = unit_op[j];
        uint32_t to = (max_slots + n_units) | NO_GROUP;
        if (op < n_ops) {
            const uint2 g = group[op];
            const uint32_t i = atomicAdd(&size[op], 1u);
            if (g.y >> 31) {
                to = g.x + i;
            } else {
                to = chunk[op / PER_CHUNK] + (op & (PER_CHUNK - 1)) * LANES + i % LANES + 32 * (i / LANES);
            }
            unit_at[to] = (uint16_t)j;
        }
        place[j] = (uint16_t)to;
    }
    __syncthreads();   // (the sizes lie in the first warp's block)
    for (uint32_t i = lane; i < chunk[(n_ops + PER_CHUNK - 1) / PER_CHUNK]; i += 32) keys[i] = K_ABSENT;   // unused slots stay absent
    __syncwarp();

    for (uint32_t cand = blockIdx.x * n_warps + warp; cand < n_cand; cand += gridDim.x * n_warps) {
        const double* t = t_cand + (size_t)cand * n_units;
        const uint8_t* ok = correct + (size_t)cand * n_units;
        if (cand + gridDim.x * n_warps < n_cand) {   // the warp's next candidate starts towards L2
            const size_t ahead = (size_t)gridDim.x * n_warps * n_units;
            for (uint32_t o = lane * 16u; o < n_units; o += 512u) asm volatile("prefetch.global.L2 [%0];" ::"l"(t + ahead + o));
            for (uint32_t o = lane * 128u; o < n_units; o += 4096u) asm volatile("prefetch.global.L2 [%0];" ::"l"(ok + ahead + o));
        }
        uint32_t errors = 0;
        for (uint32_t j0 = lane; j0 < n_units; j0 += 32 * WARP_ILP) {
            double tj[WARP_ILP];
            uint32_t okj[WARP_ILP];
#pragma unroll
            for (uint32_t u = 0; u < WARP_ILP; ++u) {
                const uint32_t j = min(j0 + 32 * u, n_units - 1);
                tj[u] = __ldg(t + j);
                okj[u] = __ldg(ok + j);
            }
#pragma unroll
            for (uint32_t u = 0; u < WARP_ILP; ++u) {
                const uint32_t j = j0 + 32 * u, to = place[j];          // (padded with units that do not count)
                const bool use = (okj[u] != 0) & ((to & NO_GROUP) == 0);
                const uint32_t key = approx_key(roof[j], roofline_s + j, tj[u], use, errors);
                keys[to & SLOT_MASK] = key;
            }
        }
        __syncwarp();
        for (uint32_t op0 = 0; op0 < n_ops; op0 += PER_CHUNK) {
            const uint32_t op = op0 + lane / LANES;
            const uint2 g = op < n_ops ? group[op] : make_uint2(0, 0);
            const bool is_large = g.y >> 31;
            const uint32_t at = chunk[op0 / PER_CHUNK], first_slot = at + lane / LANES * LANES, length = (chunk[op0 / PER_CHUNK + 1] - at) / 32;
            uint32_t* col = keys + at + lane;
            uint32_t low = 0, up = 0, m = 0;
            bool search = false;
            if (length == 8) m = middle_of<PAIRS, 8>(col, low, up, search);
            else if (length == 16) m = middle_of<PAIRS, 16>(col, low, up, search);
            else if (length == 20) m = middle_of<PAIRS, 20>(col, low, up, search);
            else if (length == 24) m = middle_of<PAIRS, 24>(col, low, up, search);
            else if (length == 28) m = middle_of<PAIRS, 28>(col, low, up, search);
            else if (length == 32) m = middle_of<PAIRS, 32>(col, low, up, search);
            double s = 0.0;
            if (m != 0 && !search) {
                const uint32_t ju = unit_at[first_slot + (PAIRS ? up : 32 * up)], jl = unit_at[first_slot + (PAIRS ? low : 32 * low)];
                s = __ddiv_rn(__ldg(roofline_s + ju), __ldg(t + ju));
                if (!(m & 1u)) s = __dmul_rn(__dadd_rn(__ddiv_rn(__ldg(roofline_s + jl), __ldg(t + jl)), s), 0.5);
            }
            for (uint32_t todo = __ballot_sync(FULL, (search || is_large) && lane % LANES == 0); todo; todo &= todo - 1) {
                const uint32_t src = __ffs(todo) - 1;
                const uint32_t first = __shfl_sync(FULL, is_large ? g.x : first_slot, src), packed = __shfl_sync(FULL, g.y, src);
                const uint32_t n = packed & 0x7FFFFFFFu, stride = packed >> 31 ? 1u : 32u;
                auto key_at = [=](uint32_t a) {
                    const uint32_t j = unit_at[first + (PAIRS && stride != 1 ? a % LANES + 32 * (a / LANES) : a * stride)];
                    return exact_key(__ldg(roofline_s + j), __ldg(t + j), __ldg(ok + j) != 0);
                };
                uint32_t usable = 0;
                ull k_lo, k_hi;
                bool found = false;
                if (stride == 1) {
                    const Middle d = group_middle(keys + first, n, bins);
                    usable = d.m;
                    if (!d.unknown && usable != 0 && d.close <= 32) {
                        // the exact scores of the units close to the middle, ranked
                        ull* list = reinterpret_cast<ull*>(bins);
                        uint32_t filled = 0;
                        for (uint32_t a0 = 0; a0 < n; a0 += 32) {
                            const bool in = a0 + lane < n && keys[first + a0 + lane] - d.from() <= d.span();
                            const uint32_t votes = __ballot_sync(FULL, in);
                            if (in) list[filled + __popc(votes & ((1u << lane) - 1u))] = key_at(a0 + lane);
                            filled += __popc(votes);
                        }
                        __syncwarp();
                        const ull x = lane < filled ? list[lane] : ~0ull;
                        uint32_t less = 0, leq = 0;
                        for (uint32_t i = 0; i < filled; ++i) {
                            less += list[i] < x ? 1u : 0u;
                            leq += list[i] <= x ? 1u : 0u;
                        }
                        const uint32_t kl = (usable - 1) / 2 - d.below, ku = usable / 2 - d.below;
                        k_lo = __shfl_sync(FULL, x, __ffs(__ballot_sync(FULL, lane < filled && less <= kl && kl < leq)) - 1);
                        k_hi = __shfl_sync(FULL, x, __ffs(__ballot_sync(FULL, lane < filled && less <= ku && ku < leq)) - 1);
                        __syncwarp();
                        found = true;
                    }
                }
                if (!found) {
                    usable = 0;
                    for (uint32_t a = lane; a < n; a += 32) usable += key_at(a) != ~0ull ? 1u : 0u;
                    usable = __reduce_add_sync(FULL, usable);
                    if (usable == 0) continue;
                    warp_select<ull>(key_at, n, (usable - 1) / 2, bins, &k_lo, &k_hi);
                }
                if (lane == src) s = median_of_keys(k_lo, (usable & 1u) ? k_lo : k_hi, usable & 1u);
            }
            if (op < n_ops && lane % LANES == 0) {
                prod[op] = __dmul_rn(w[op], s);
                if (s_op_out) s_op_out[(size_t)cand * n_ops + op] = s;
            }
        }
        errors = __reduce_add_sync(FULL, errors);
        __syncwarp();
        if (lane == 0) {
            double agg = 0.0;  // Eq. 6 in operator order
#pragma unroll 4
            for (uint32_t i = 0; i < n_ops; ++i) agg = __dadd_rn(agg, prod[i]);
            s_agg[cand] = agg;
            if (errors_out) errors_out[cand] = errors;
        }
        __syncwarp();
    }
}

// The same for g <= N keys in a row that stay where they are; the middle keys come with their slots.
template <int N>
__device__ __forceinline__ uint32_t middle_keys(const uint32_t* keys, uint32_t g, uint32_t& vl, uint32_t& vu, bool& search) {
    uint32_t v[N], m = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t k = (uint32_t)i < g ? keys[i] : K_ABSENT;
        m += k != K_ABSENT ? 1u : 0u;
        v[i] = (k & ~K_SLOT) | (uint32_t)i;
    }
    sort_network<N>(v);
    const int kl = ((int)m - 1) / 2, ku = (int)m / 2;
    uint32_t below = 0, above = K_ABSENT, last = 0;
    vl = vu = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        below = i == kl - 1 ? v[i] : below;
        vl = i == kl ? v[i] : vl;
        vu = i == ku ? v[i] : vu;
        above = i == ku + 1 && i < (int)m ? v[i] : above;
        last = i == (int)m - 1 ? v[i] : last;
    }
    search = m != 0 && (last >= K_UNKNOWN || (kl > 0 && vl - below <= NET_APART) || (kl != ku && vu - vl <= NET_APART) || above - vu <= NET_APART);
    return m;
}

// ---- one candidate per CTA ------------------------------------------------------------------------
// Bound by latency: the loads of Eq. 4, then the search rounds of the largest groups (one warp each).  Keys
// of four bytes and positions of two let two or three CTAs share an SM at ten thousand units, so that one's
// loads cover another's search: 1 000 candidates x 12 001 units x 7 operators in 142 us (with 64-bit exact
// keys, one CTA per SM: 166 us).
constexpr uint32_t MARK = 0x80000000u;        // top bit of a key: a middle unit of its operator, or close to one
// flags beside an operator's count of usable units: the marked units' exact scores are ranked / all are searched
constexpr uint32_t M_RANK = 0x40000000u, M_SEARCH = 0x80000000u, M_COUNT = 0x3FFFFFFFu;
constexpr uint32_t POOL_MAX = 128;            // exact scores kept for such ranking, per candidate

struct CtaLayout {
    uint32_t mid, bins, start, upper, count, place, total;
    __host__ __device__ CtaLayout(uint32_t n, uint32_t n_ops, uint32_t threads) {
        uint32_t o = (4u * n + 15u) & ~15u;          // (keys first)
        mid = o;    o += 16u * n_ops;                // exact scores of the lower and upper middle, then w * S in the first
        bins = o;   o += threads / 32u * 4u * SELECT_BINS;
        start = o;  o += 4u * (n_ops + 1u);
        upper = o;  o += 4u * n_ops;                 // key of the upper middle, or units below the marked ones (at first: group sizes)
        count = o;  o += 4u * n_ops;
        place = o;  o += 2u * n;
        total = o;
    }
};

__global__ void __launch_bounds__(1024)
    score_cta_kernel(const double* __restrict__ roofline_s, const uint32_t* __restrict__ unit_op, uint32_t n_units,
                     const double* __restrict__ t_cand, const uint8_t* __restrict__ correct, uint32_t n_cand,
                     const double* __restrict__ w, uint32_t n_ops, double* s_agg, double* s_op_out, ull* errors_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ ull s_pool[POOL_MAX];
    __shared__ uint16_t s_pool_op[POOL_MAX];
    __shared__ uint32_t s_errors, s_pooled;
    const CtaLayout L(n_units, n_ops, blockDim.x);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw);              // grouped by operator
    double* mid = reinterpret_cast<double*>(smem_raw + L.mid);
    uint32_t* start = reinterpret_cast<uint32_t*>(smem_raw + L.start);
    uint32_t* upper = reinterpret_cast<uint32_t*>(smem_raw + L.upper);
    uint32_t* count = reinterpret_cast<uint32_t*>(smem_raw + L.count);
    uint16_t* place = reinterpret_cast<uint16_t*>(smem_raw + L.place);   // position, 0xFFFF = none (positions stay below 2^14)
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, n_warps = blockDim.x >> 5;
    uint32_t* bins = reinterpret_cast<uint32_t*>(smem_raw + L.bins) + warp * SELECT_BINS;
    if (threadIdx.x == 0) s_errors = s_pooled = 0;
    {   // where each unit goes: segments of the operators one behind the other
        uint32_t* fill = upper;
        count_groups(unit_op, n_units, n_ops, fill);
        if (threadIdx.x < 32) {
            uint32_t run = 0;
            for (uint32_t i0 = 0; i0 < n_ops; i0 += 32) {
                const uint32_t i = i0 + lane, c = i < n_ops ? fill[i] : 0u;
                uint32_t incl = c;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(FULL, incl, d);
                    if (lane >= (uint32_t)d) incl += o;
                }
                if (i < n_ops) {
                    start[i] = run + incl - c;
                    fill[i] = 0;
                }
                run += __shfl_sync(FULL, incl, 31);
            }
            if (lane == 0) start[n_ops] = run;
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < n_units; j += blockDim.x) {
            const uint32_t op = unit_op[j];
            place[j] = op < n_ops ? (uint16_t)(start[op] + atomicAdd(&fill[op], 1u)) : (uint16_t)0xFFFFu;
        }
        __syncthreads();
    }

    // One operator's middle keys are marked, with whatever comes close to them (one warp).
    auto mark_middle = [&](uint32_t op) {
        const uint32_t b = start[op], g = start[op + 1] - b;
        const Middle d = group_middle(keys + b, g, bins);
        uint32_t flag = 0;
        if (d.unknown) {
            flag = M_SEARCH;
        } else if (d.m != 0) {
            if (!d.clear()) flag = d.close <= 32 ? M_RANK : M_SEARCH;
            for (uint32_t a = lane; a < g; a += 32) {
                const uint32_t k = keys[b + a];
                if (k - d.from() <= d.span()) keys[b + a] = k | MARK;
            }
        }
        if (lane == 0) {
            upper[op] = flag ? d.below : d.v_up;
            count[op] = d.m | flag;
        }
    };
    const bool lane_sorted = n_ops >= 4 * n_warps;   // (fewer operators: a warp for each is quicker than a lane for each)
    for (uint32_t cand = blockIdx.x; cand < n_cand; cand += gridDim.x) {
        const double* t = t_cand + (size_t)cand * n_units;
        const uint8_t* ok = correct + (size_t)cand * n_units;
        // 1. approximate keys
        uint32_t errors = 0;
        constexpr uint32_t U = 4;
        for (uint32_t j0 = threadIdx.x; j0 < n_units; j0 += blockDim.x * U) {
            double tj[U], rj[U];
            uint32_t okj[U];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                const uint32_t j = min(j0 + blockDim.x * u, n_units - 1);
                tj[u] = __ldg(t + j);
                okj[u] = __ldg(ok + j);
                rj[u] = __ldg(roofline_s + j);
            }
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                const uint32_t j = j0 + blockDim.x * u;
                const uint32_t pos = j < n_units ? place[j] : 0xFFFFu;
                if (pos != 0xFFFFu) keys[pos] = approx_key(approx_roofline(rj[u]), roofline_s + j, tj[u], okj[u] != 0, errors);
            }
        }
        errors = __reduce_add_sync(FULL, errors);
        if (lane == 0 && errors) atomicAdd(&s_errors, errors);
        __syncthreads();
        // 2. the middle keys of each operator are marked
        //    Groups of up to 32: one lane each, 32 operators to a warp, where that keeps the warps busy
        for (uint32_t op0 = warp * 32; lane_sorted && op0 < n_ops; op0 += n_warps * 32) {
            const uint32_t op = op0 + lane, b = op < n_ops ? start[op] : 0u, g = op < n_ops ? start[op + 1] - b : 0u;
            const bool small = g != 0 && g <= NET_MAX;
            const uint32_t widest = __reduce_max_sync(FULL, small ? g : 0u);
            uint32_t vl = 0, vu = 0, m = 0;
            bool search = false;
            if (widest == 0) {
            } else if (widest <= 8) m = middle_keys<8>(keys + b, small ? g : 0u, vl, vu, search);
            else if (widest <= 16) m = middle_keys<16>(keys + b, small ? g : 0u, vl, vu, search);
            else if (widest <= 24) m = middle_keys<24>(keys + b, small ? g : 0u, vl, vu, search);
            else m = middle_keys<32>(keys + b, small ? g : 0u, vl, vu, search);
            if (op < n_ops && g <= NET_MAX && !search) {
                if (m != 0) {
                    upper[op] = keys[b + (vu & K_SLOT)];
                    keys[b + (vu & K_SLOT)] |= MARK;
                    if (!(m & 1u)) keys[b + (vl & K_SLOT)] |= MARK;
                }
                count[op] = m;
            }
            for (uint32_t todo = __ballot_sync(FULL, search); todo; todo &= todo - 1) mark_middle(__ffs(todo) - 1 + op0);
        }
        for (uint32_t op = warp; op < n_ops; op += n_warps)
            if (!lane_sorted || start[op + 1] - start[op] > NET_MAX) mark_middle(op);
        __syncthreads();
        // 3. the marked units are divided exactly
        for (uint32_t j = threadIdx.x; j < n_units; j += blockDim.x) {
            const uint32_t pos = place[j];
            if (pos == 0xFFFFu) continue;
            const uint32_t k = keys[pos];
            if ((k & MARK) == 0) continue;
            const uint32_t op = __ldg(unit_op + j), m = count[op];
            const double s = __ddiv_rn(__ldg(roofline_s + j), __ldg(t + j));
            if (m & M_RANK) {
                const uint32_t at = atomicAdd(&s_pooled, 1u);
                if (at < POOL_MAX) {
                    s_pool[at] = key_of_score(s);
                    s_pool_op[at] = (uint16_t)op;
                }
            } else if (!(m & M_SEARCH)) {
                mid[2 * op + ((k & ~MARK) == upper[op] ? 1 : 0)] = s;
            }
        }
        __syncthreads();
        // 4. Eq. 5, and the products of Eq. 6
        for (uint32_t op0 = warp * 32; op0 < n_ops; op0 += n_warps * 32) {
            const uint32_t op = op0 + lane;
            const uint32_t m = op < n_ops ? count[op] : 0u;
            double s = 0.0;
            if (m != 0 && !(m & (M_RANK | M_SEARCH))) {
                s = mid[2 * op + 1];
                if (!(m & 1u)) s = __dmul_rn(__dadd_rn(mid[2 * op], s), 0.5);
            }
            for (uint32_t todo = __ballot_sync(FULL, m & (M_RANK | M_SEARCH)); todo; todo &= todo - 1) {
                const uint32_t src = __ffs(todo) - 1, o = op0 + src, flags = count[o], usable = flags & M_COUNT, k = (usable - 1) / 2;
                ull k_lo, k_hi;
                if ((flags & M_RANK) && s_pooled <= POOL_MAX) {
                    auto key_at = [=](uint32_t i) { return s_pool_op[i] == o ? s_pool[i] : ~0ull; };
                    warp_select<ull>(key_at, s_pooled, k - upper[o], bins, &k_lo, &k_hi);
                } else {
                    auto key_at = [=](uint32_t j) {   // (rare: every unit is asked whether it is the operator's)
                        return __ldg(unit_op + j) == o ? exact_key(__ldg(roofline_s + j), __ldg(t + j), __ldg(ok + j) != 0) : ~0ull;
                    };
                    warp_select<ull>(key_at, n_units, k, bins, &k_lo, &k_hi);
                }
                if (lane == src) s = median_of_keys(k_lo, (usable & 1u) ? k_lo : k_hi, usable & 1u);
            }
            __syncwarp();
            if (op < n_ops) {
                mid[2 * op] = __dmul_rn(w[op], s);
                if (s_op_out) s_op_out[(size_t)cand * n_ops + op] = s;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double agg = 0.0;  // Eq. 6 in operator order
#pragma unroll 4
            for (uint32_t i = 0; i < n_ops; ++i) agg = __dadd_rn(agg, mid[2 * i]);
            s_agg[cand] = agg;
            if (errors_out) errors_out[cand] = s_errors;
            s_errors = s_pooled = 0;
        }
        __syncthreads();   // the keys, counts and s_errors are reused
    }
}

// ---- one candidate per CTA, large groups ------------------------------------------------------------
// No order is made of an operator's units: while their keys are formed, each bumps one of its operator's counters by
// the key's range, a warp finds the range that holds the middle, and the few units in it (or as close to it as
// keys may err) are ranked by their exact scores.  Every step but the finding is spread over the whole CTA, and units stay
// where they are, so that nothing is worked out about the grouping.  Where the middle's range holds too many units it is
// cut again; what stays too many (ties) is searched among them.  Bound by latency at 44 warps per SM (loads, shared-memory
// atomics, barriers: 51 % of the issue slots).  1 000 candidates x 12 001 units x 7 operators: 145 us by score_cta_kernel, 78;
// with the next loads issued before a thread's units are worked on 116 (spills); strides not known at compile time 86.
constexpr uint32_t NEAR_MAX = 32;             // units near an operator's middle that one warp ranks, a lane each
constexpr uint32_t BINS_LOW = (127u - 7u) << 23, BINS_LOG_SPAN = 26;   // first cut: scores from 2^-7 to 2, what lies outside in the end bins
constexpr uint32_t CUTS_MAX = 6;              // (each narrows the range sevenfold or more, 32-fold where the middles are in one range or two that touch)
constexpr uint32_t NOWHERE = 0xFFFFFFFFu;     // no key is as close above it

struct BinsLayout {
    uint32_t prod, window, state, bins, listed, list, spare, op, total;
    __host__ __device__ BinsLayout(uint32_t n, uint32_t n_ops, uint32_t log_bins, uint32_t threads) {
        uint32_t o = (4u * n + 15u) & ~15u;          // (keys first)
        state = o;   o += 16u * n_ops;               // {lowest key of the middle's range, usable units below it, usable units, how to go on}
        bins = o;    o += n_ops << (log_bins + 1u);  // two counters to a word
        window = o;  o += 8u * (n_ops + 1u);                // {from, span}: units whose keys are near the middle; or {from, shift} of the next cut
        prod = o;    o += 8u * n_ops;                // w * S
        listed = o;  o += 4u * n_ops;
        list = o;    o += 2u * NEAR_MAX * n_ops;     // units near the middle
        spare = o = (o + 15u) & ~15u;  o += threads / 32u * 4u * SELECT_BINS;
        op = o;      o += n;
        total = (o + 15u) & ~15u;
    }
};
// Counters per operator: a quarter of the mean group, so that the middle's range holds about ten units of an even distribution.
inline uint32_t log_bins_for(uint32_t n, uint32_t n_ops) {
    uint32_t b = 6;
    while (b < 10 && (4u * n_ops << b) < n) ++b;
    return b;
}
constexpr uint32_t GO_NONE = 0, GO_RANK = 1, GO_CUT = 2, GO_SEARCH = 3, GO_SEARCH_ALL = 4;

// The counter (of 2 W per lane, W words) that holds the k-th counted unit; `incl`, `own`: units up to and in this lane's counters.
struct Bin {
    uint32_t at, before, n;
};
__device__ __forceinline__ Bin find_bin(const uint32_t* words, uint32_t W, uint32_t incl, uint32_t own, uint32_t k) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t src = __ffs(__ballot_sync(FULL, incl > k)) - 1, base = __shfl_sync(FULL, incl - own, src);
    if (W == 1) {
        const uint32_t word = words[src], first = word & 0xFFFFu;
        return base + first > k ? Bin{2 * src, base, first} : Bin{2 * src + 1, base + first, word >> 16};
    }
    uint32_t c = 0;
    if (lane < 2 * W) {
        const uint32_t word = words[src * W + lane / 2];
        c = lane & 1u ? word >> 16 : word & 0xFFFFu;
    }
    uint32_t upto = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(FULL, upto, d);
        if (lane >= (uint32_t)d) upto += o;
    }
    const uint32_t in = __ffs(__ballot_sync(FULL, base + upto > k)) - 1;
    return {src * 2 * W + in, base + __shfl_sync(FULL, upto - c, in), __shfl_sync(FULL, c, in)};
}

struct BinsArgs {             // what the search of a candidate needs
    const double *roofline_s, *t_cand, *w;
    double* s_op_out;
    uint32_t n_units, n_ops, log_bins;
};

// An operator that is searched, in its part of the list of units near the middles: where its units start, how many are in place, how
// many of them lie below the middle's range.
struct Segment {
    uint32_t first, placed, below, pad;
};
// The operators whose middles their keys do not tell, by exact scores: of the units in their windows, or of all.  The units are brought
// together by operator first (their numbers, where the keys were), so that a warp goes over its operator's units only: 5 000 candidates x 700
// units x 10 operators, scores alike in their keys 614 -> 239 us, 1 000 x 12 001 x 7 of two values 4 840 -> 733, 1 500 x 16 320 x 255 14.8 -> 1.2 ms (every
// warp over all units before; in place, as a call in the loop over candidates costs 2 to 4 % where nothing is searched).
// (Whole CTA, behind a barrier and with one at its end.  searched: {any operator is, their units}, both 0 again at the end)
template <int THREADS>
__device__ __forceinline__ void search_operators(const BinsArgs& a, uint32_t cand, uint32_t* searched) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t n_units = a.n_units, n_ops = a.n_ops;
    const double *roofline_s = a.roofline_s, *t = a.t_cand + (size_t)cand * n_units;
    const BinsLayout L(n_units, n_ops, a.log_bins, THREADS);
    uint32_t *keys = reinterpret_cast<uint32_t*>(smem_raw), *flags = reinterpret_cast<uint32_t*>(smem_raw + L.bins);   // a bit per unit, in the
    // counters' place (all 0 here; they are n / 8 words at least, or 512)
    uint4* state = reinterpret_cast<uint4*>(smem_raw + L.state);
    const uint2* window = reinterpret_cast<const uint2*>(smem_raw + L.window);
    const uint8_t* ops = smem_raw + L.op;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, n_warps = THREADS / 32;
    auto segment = [&](uint32_t op) { return reinterpret_cast<Segment*>(smem_raw + L.list) + op * (2 * NEAR_MAX / sizeof(Segment)); };
    uint32_t* listed = reinterpret_cast<uint32_t*>(smem_raw + L.listed);
    for (uint32_t op = threadIdx.x; op < n_ops; op += THREADS)
        if (state[op].w >= GO_SEARCH) *segment(op) = Segment{atomicAdd(&searched[1], listed[op]), 0, 0, 0};
    __syncthreads();
    for (uint32_t j0 = warp * 32; j0 < n_units; j0 += THREADS) {
        const uint32_t j = j0 + lane, op = j < n_units ? ops[j] : n_ops;
        bool in = false;
        if (op < n_ops && state[op].w >= GO_SEARCH) {
            const uint32_t key = keys[j];
            const uint2 win = window[op];
            in = key - win.x <= win.y;
            if (in && state[op].w == GO_SEARCH && key < state[op].x) atomicAdd(&segment(op)->below, 1u);
        }
        const uint32_t votes = __ballot_sync(FULL, in);
        if (lane == 0) flags[j0 / 32] = votes;
    }
    __syncthreads();
    uint16_t* units = reinterpret_cast<uint16_t*>(keys);
    for (uint32_t j = threadIdx.x; j < n_units; j += THREADS) {
        if (!(flags[j / 32] >> (j % 32) & 1u)) continue;
        Segment* s = segment(ops[j]);
        units[s->first + atomicAdd(&s->placed, 1u)] = (uint16_t)j;
    }
    __syncthreads();
    if (threadIdx.x == 0) searched[0] = searched[1] = 0;
    for (uint32_t i = threadIdx.x; i < (n_units + 31) / 32; i += THREADS) flags[i] = 0;
    for (uint32_t op = warp; op < n_ops; op += n_warps) {
        const uint4 st = state[op];
        if (st.w < GO_SEARCH) continue;
        const Segment g = *segment(op);
        const uint32_t usable = st.w == GO_SEARCH_ALL ? g.placed : st.z, below = st.w == GO_SEARCH_ALL ? 0u : st.y - g.below;
        const uint16_t* own = units + g.first;
        auto key_at = [=](uint32_t i) {
            const uint32_t j = own[i];
            return exact_key(__ldg(roofline_s + j), __ldg(t + j), true);
        };
        ull k_lo, k_hi;
        warp_select_here<ull>(key_at, g.placed, (usable - 1) / 2 - below, reinterpret_cast<uint32_t*>(smem_raw + L.spare) + warp * SELECT_BINS, &k_lo, &k_hi);
        if (lane == 0) {
            const double s = median_of_keys(k_lo, (usable & 1u) ? k_lo : k_hi, usable & 1u);
            reinterpret_cast<double*>(smem_raw + L.prod)[op] = __dmul_rn(a.w[op], s);
            if (a.s_op_out) a.s_op_out[(size_t)cand * n_ops + op] = s;
            listed[op] = 0;
            state[op].w = GO_NONE;
        }
    }
    __syncthreads();
}

constexpr int bins_ctas(int threads) { return threads == 1024 ? 1 : 1536 / threads; }   // per SM, by registers
template <int THREADS>
__global__ void __launch_bounds__(THREADS, bins_ctas(THREADS))
    score_bins_kernel(const double* __restrict__ roofline_s, const uint32_t* __restrict__ unit_op, uint32_t n_units,
                      const double* __restrict__ t_cand, const uint8_t* __restrict__ correct, uint32_t n_cand,
                      const double* __restrict__ w, uint32_t n_ops, uint32_t log_bins, double* s_agg, double* s_op_out, ull* errors_out) {
    __shared__ BinsArgs s_args;                                          // (for the search: held in registers for it they cost 1 to 2 % where nothing is searched)
    if (threadIdx.x == 0) s_args = BinsArgs{roofline_s, t_cand, w, s_op_out, n_units, n_ops, log_bins};
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_errors[2];
    constexpr uint32_t U = 4;                                            // units of a thread in flight
    __shared__ uint32_t s_cut;                                           // round of cuts that is still wanted
    __shared__ uint32_t s_searched[2];                                   // (see search_operators)
    const BinsLayout L(n_units, n_ops, log_bins, THREADS);
    uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw);
    uint4* state = reinterpret_cast<uint4*>(smem_raw + L.state);
    uint32_t* bins = reinterpret_cast<uint32_t*>(smem_raw + L.bins);
    uint2* window = reinterpret_cast<uint2*>(smem_raw + L.window);
    double* prod = reinterpret_cast<double*>(smem_raw + L.prod);
    uint32_t* listed = reinterpret_cast<uint32_t*>(smem_raw + L.listed);
    uint16_t* list = reinterpret_cast<uint16_t*>(smem_raw + L.list);
    uint8_t* ops = smem_raw + L.op;                                      // n_ops: none
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u, n_warps = THREADS / 32;
    const uint32_t n_bins = 1u << log_bins, op_words = n_bins / 2, W = op_words / 32, first_shift = BINS_LOG_SPAN - log_bins;
    for (uint32_t j = threadIdx.x; j < n_units; j += THREADS) {
        const uint32_t op = unit_op[j];
        ops[j] = (uint8_t)min(op, n_ops);
    }
    for (uint32_t i = threadIdx.x; i < n_ops * op_words; i += THREADS) bins[i] = 0;
    for (uint32_t i = threadIdx.x; i < n_ops; i += THREADS) {
        listed[i] = 0;
        state[i].w = GO_NONE;
    }
    if (threadIdx.x == 0) {
        s_errors[0] = s_errors[1] = s_cut = s_searched[0] = s_searched[1] = 0;
        window[n_ops] = make_uint2(NOWHERE, 0);                          // (units without an operator)
    }
    __syncthreads();
    auto count_in = [&](uint32_t op, uint32_t bin) { atomicAdd(&bins[op * op_words + bin / 2], 1u << (bin % 2 * 16)); };

    uint32_t turn = 0;
    for (uint32_t cand = blockIdx.x; cand < n_cand; cand += gridDim.x, turn ^= 1u) {
        const double* t = t_cand + (size_t)cand * n_units;
        const uint8_t* ok = correct + (size_t)cand * n_units;
        if (cand + gridDim.x < n_cand) {   // the CTA's next candidate starts towards L2
            const size_t ahead = (size_t)gridDim.x * n_units;
            for (uint32_t o = threadIdx.x * 16u; o < n_units; o += THREADS * 16u) asm volatile("prefetch.global.L2 [%0];" ::"l"(t + ahead + o));
            for (uint32_t o = threadIdx.x * 128u; o < n_units; o += THREADS * 128u) asm volatile("prefetch.global.L2 [%0];" ::"l"(ok + ahead + o));
        }
        // 1. approximate keys, counted by operator and range
        uint32_t errors = 0;
        auto some_units = [&](uint32_t j0, auto inside) {                // units j0, j0 + THREADS, ...
            double tj[U], rj[U];
            uint32_t okj[U];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                if (!inside(u)) continue;
                tj[u] = __ldg(t + j0 + u * THREADS);
                okj[u] = __ldg(ok + j0 + u * THREADS);
                rj[u] = __ldg(roofline_s + j0 + u * THREADS);
            }
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                if (!inside(u)) continue;
                const uint32_t op = ops[j0 + u * THREADS];
                const uint32_t key = approx_key(approx_roofline(rj[u]), roofline_s + j0 + u * THREADS, tj[u], (okj[u] != 0) & (op != n_ops), errors);
                keys[j0 + u * THREADS] = key;
                if (key < K_UNKNOWN)
                    count_in(op, min(n_bins - 1, (uint32_t)max((int)(key - BINS_LOW), 0) >> first_shift));
                else if (key == K_UNKNOWN)
                    state[op].w = GO_SEARCH_ALL;
            }
        };
        uint32_t j0 = threadIdx.x;
        for (; j0 + (U - 1) * THREADS < n_units; j0 += U * THREADS) some_units(j0, [](uint32_t) { return true; });
        some_units(j0, [&](uint32_t u) { return j0 + u * THREADS < n_units; });
        errors = __reduce_add_sync(FULL, errors);
        if (lane == 0 && errors) atomicAdd(&s_errors[turn], errors);
        __syncthreads();
        // 2. the range of each operator's middle; once more inside it where it holds too many
        for (uint32_t round = 1;; ++round) {
            for (uint32_t op = warp; op < n_ops; op += n_warps) {
                uint4 st = state[op];
                if (round > 1 && st.w != GO_CUT) continue;
                uint32_t* words = bins + op * op_words;
                uint32_t own = 0;
                for (uint32_t i = 0; i < W; ++i) own += (words[lane * W + i] & 0xFFFFu) + (words[lane * W + i] >> 16);
                uint32_t incl = own;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(FULL, incl, d);
                    if (lane >= (uint32_t)d) incl += o;
                }
                uint32_t base = BINS_LOW, shift = first_shift, below = 0, m = __shfl_sync(FULL, incl, 31);
                if (round > 1) {
                    const uint2 cut = window[op];
                    base = cut.x;
                    shift = cut.y;
                    below = st.y;
                    m = st.z;
                }
                uint2 win = make_uint2(NOWHERE, 0);
                if (st.w == GO_SEARCH_ALL) {
                    win = make_uint2(0, K_UNKNOWN);
                } else {
                    st = make_uint4(0, 0, m, GO_NONE);
                    if (m != 0) {
                        const Bin low = find_bin(words, W, incl, own, (m - 1) / 2 - below);
                        Bin up = low;
                        if (!(m & 1u) && m / 2 - below >= low.before + low.n) up = find_bin(words, W, incl, own, m / 2 - below);
                        uint32_t from = base + (low.at << shift), to = base + ((up.at + 1) << shift) - 1;
                        if (round == 1 && low.at == 0) from = 0;
                        if (round == 1 && up.at == n_bins - 1) to = K_UNKNOWN - 1;
                        to = min(to, K_UNKNOWN - 1);
                        st.x = from;
                        st.y = below + low.before;
                        const uint32_t in = up.before + up.n - low.before;
                        const bool far = (up.at - low.at) * 8 > n_bins;          // two middles that a cut would only trim the outsides of
                        st.w = in <= NEAR_MAX ? GO_RANK : (shift == 0 || round == CUTS_MAX || far ? GO_SEARCH : GO_CUT);
                        if (st.w == GO_CUT) {
                            const int len = 32 - __clz((int)(to - from));
                            win = make_uint2(from, len > (int)log_bins ? len - log_bins : 0u);
                        } else {
                            const uint32_t first = from > K_APART ? from - K_APART : 0u;
                            win = make_uint2(first, min(to + K_APART, K_UNKNOWN - 1) - first);
                        }
                    }
                }
                __syncwarp();
                for (uint32_t i = lane; i < op_words; i += 32) words[i] = 0;
                if (lane == 0) {
                    state[op] = st;
                    window[op] = win;
                    if (st.w == GO_CUT) s_cut = round;
                }
            }
            __syncthreads();
            if (s_cut != round) break;
            for (uint32_t j = threadIdx.x; j < n_units; j += THREADS) {
                const uint32_t key = keys[j];
                if (key >= K_UNKNOWN) continue;
                const uint32_t op = ops[j];
                if (state[op].w != GO_CUT) continue;
                const uint2 cut = window[op];
                const uint32_t bin = (key - cut.x) >> cut.y;
                if (key >= cut.x && bin < n_bins) count_in(op, bin);
            }
            __syncthreads();
        }
        // 3. the units near the middles
#pragma unroll 4
        for (uint32_t j = threadIdx.x; j < n_units; j += THREADS) {
            const uint32_t key = keys[j], op = ops[j];
            const uint2 win = window[op];
            if (key - win.x > win.y) continue;                           // (nothing is near K_UNKNOWN or above)
            const uint32_t at = atomicAdd(&listed[op], 1u);
            if (at < NEAR_MAX) list[op * NEAR_MAX + at] = (uint16_t)j;
        }
        __syncthreads();
        // 4. Eq. 5 by their exact scores, and the products of Eq. 6
        if (threadIdx.x == 0) s_cut = 0;
        for (uint32_t op = warp; op < n_ops; op += n_warps) {
            const uint4 st = state[op];
            const uint32_t n = listed[op], m = st.z;
            double s = 0.0;
            if (st.w == GO_RANK && n <= NEAR_MAX) {
                const uint32_t j = lane < n ? list[op * NEAR_MAX + lane] : 0u;
                const ull x = lane < n ? exact_key(__ldg(roofline_s + j), __ldg(t + j), true) : ~0ull;
                const uint32_t below = st.y - __popc(__ballot_sync(FULL, lane < n && keys[j] < st.x));   // units that are not listed
                uint32_t less = 0, leq = 0;
                for (uint32_t i = 0; i < n; ++i) {
                    const ull y = __shfl_sync(FULL, x, i);
                    less += y < x ? 1u : 0u;
                    leq += y <= x ? 1u : 0u;
                }
                const uint32_t kl = (m - 1) / 2 - below, ku = m / 2 - below;
                const ull k_lo = __shfl_sync(FULL, x, __ffs(__ballot_sync(FULL, lane < n && less <= kl && kl < leq)) - 1);
                const ull k_hi = __shfl_sync(FULL, x, __ffs(__ballot_sync(FULL, lane < n && less <= ku && ku < leq)) - 1);
                s = median_of_keys(k_lo, k_hi, m & 1u);
            } else if (st.w != GO_NONE) {            // too many units alike, or units whose keys say nothing
                __syncwarp();
                if (lane == 0) {
                    state[op].w = max(st.w, GO_SEARCH);
                    s_searched[0] = 1;
                }
                continue;
            }
            __syncwarp();
            if (lane == 0) {
                listed[op] = 0;
                state[op].w = GO_NONE;
                prod[op] = __dmul_rn(w[op], s);
                if (s_op_out) s_op_out[(size_t)cand * n_ops + op] = s;
            }
        }
        __syncthreads();
        if (s_searched[0] != 0) search_operators<THREADS>(s_args, cand, s_searched);
        if (threadIdx.x == 0) {   // (the others go on to the next candidate: nothing of this is touched before two more barriers)
            double agg = 0.0;     // Eq. 6 in operator order
#pragma unroll 4
            for (uint32_t i = 0; i < n_ops; ++i) agg = __dadd_rn(agg, prod[i]);
            s_agg[cand] = agg;
            if (errors_out) errors_out[cand] = s_errors[turn];
            s_errors[turn] = 0;
        }
    }
}

// One candidate per warp (true) or per CTA (false); `held`: candidates an SM holds at once by warps.  A CTA has the shorter
// chain, a warp the smaller sum of work, so the warps win once every SM has several candidates, and the sooner the better
// the operators fill a warp's lanes.  Device times in us, warps / CTAs, on both sides of each line:
//   up to 500 units     4 candidates per SM and one per unit (groups up to 48), 16 per SM beyond: 450 units in 16 operators, 660
//                       candidates 7.8 / 11.1; 300 in 12, 450 candidates 9.4 / 8.6
//   groups up to 30     8 per SM, and one per unit, 1.4 from 1 500 units on, where fewer warps fit an SM: 1 000 units in 35
//                       operators, 900 candidates 22.0 / 22.0, 2 000 25.0 / 37.2; 2 000 units in 83, 1 500 candidates 58 / 43
//   up to 50            5 per SM (8 from 44 on): two lanes an operator are full, and a CTA's warps search every group: 1 400 units
//                       in 35 operators, 600 candidates 27.5 / 27.9, 1 500 36.0 / 44.0
//   beyond (up to 64)   16 per SM, with fewer units the more groups are then too large for two lanes: 800 units
//                       in 15 operators, 2 400 candidates 18 / 34; 1 000 in 17, 2 400 candidates 48 / 39, 3 500 41 / 57
bool by_warps(uint32_t n, uint32_t n_ops, uint32_t b, uint32_t sms, uint32_t held) {
    if (held < (n <= 24 * n_ops ? 12u : 6u)) return false;
    if (n <= 500) return n <= 48 * n_ops ? b >= 4 * sms && b >= n : b >= 16 * sms;
    const bool enough = b * 10ull >= n * (n <= 1500 ? 10ull : 14ull);
    if (n <= 30 * n_ops) return b >= 8 * sms && enough;
    if (n <= 50 * n_ops) return b >= (n <= 44 * n_ops ? 5 : 8) * sms && (n <= 2200 || enough);
    if (n <= 700) return b >= 16 * sms;
    return b >= 16 * sms && (ull)n * (n - 44 * n_ops) <= (b < 20 * sms ? 14000ull : 19000ull) * n_ops;
}

// Threads of a CTA that holds one candidate.  Where there are more candidates than the SMs hold at 256 threads (four CTAs
// each, by registers), smaller CTAs take all of them at once (700 units in 28 operators: 600 candidates 16.6 us at 256 threads,
// 11.0 at 192, 900 18.9, 13.8 at 128).  Larger groups need the warps (19 operators of 36: 825 candidates 16.9, 18.2 at 128).
uint32_t cta_threads(uint32_t n, uint32_t n_ops, uint32_t b, uint32_t sms) {
    if (n > 4096) return n <= 13000 ? 512u : 1024u;
    if (n > 1400 || b <= 4 * sms) return 256u;
    if (b <= 5 * sms) return n <= 36 * n_ops ? 192u : 256u;
    return n <= 30 * n_ops && (n <= 800 || b <= 8 * sms) ? 128u : 256u;
}

// One candidate per CTA by counting (score_bins_kernel), from groups of 64 units on in the mean (us, counting / the better of
// the other two: 6 000 units in 90 operators, 600 candidates 60 / 69, 5 000 387 / 421; 700 in 10, 1 500 22.5 / 26.6; 12 001 in 7, 1 000
// 78 / 145; but 1 000 in 15, 5 000 78 / 74); below, its two steps of a warp per operator
// outweigh what it saves (6 000 in 150, 500 candidates 73 / 78; 8 000 in 200, 3 000 487 / 438; 3 000 in 300, 5 000 950 / 226).
// Up to 500 units, a warp per candidate is quicker once it is by_warps' choice (100 in 1, 20 000 candidates 57 / 35, 100 000 268 / 141; 200 in 2,
// 13 000 49 / 39; 300 in 4, 45 000 209 / 196; 500 in 2, 13 000 69 / 55, in 7, 45 000 338 / 311, though 4 500 39 / 47; scores alike in their keys, 500 in
// 7, 13 000 482 / 234), and not above (550 in 2, 13 000 66 / 74, in 7 100 / 104; 600 in 4, 20 000 122 / 130).
constexpr uint32_t BINS_GROUP_MIN = 64, BINS_UNITS_FEW = 500;
constexpr uint32_t BINS_OPS_MAX = 255;        // (a unit's operator is kept in a byte, n_ops where it has none)

// Its threads.  A candidate's latency falls with the threads as long as SMs would idle; with several candidates per SM, CTAs
// that are large enough to cover the loads and no larger, as fewer warps wait while an operator's warp works (us at 128 / 256 /
// 512 / 1 024 threads: 700 units in 4 operators, 100 candidates 12.6 / 12.6 / 12.1 / 12.2, 5 000 37 / 41 / 61 / 121;
// 3 000 in 15, 300 candidates 30 / 21.5 / 17.7 / 22.8, 5 000 121 / 120 / 129 / 188; 6 000 in 4, 100 candidates 22.9 / 18.6 / 14.6
// / 13.2, 5 000 175 / 141 / 148 / 219).  Where shared memory holds one or two CTAs an SM, or the operators are many, the largest
// (16 000 in 80, 1 500 candidates 560 / 321 / 218 / 203; 12 000 in 181 741 / 412 / 267 / 254, in 4 179 / 119 / 98 / 108).
uint32_t bins_threads(uint32_t n, uint32_t n_ops, uint32_t b, uint32_t sms) {
    if (b <= sms) return n > 3000 ? 1024u : n > 1000 ? 512u : 256u;
    if (n > 14000 || (n > 9000 && n_ops > 100)) return 1024u;
    if (n > 4000 || (n > 2000 && b <= 3 * sms)) return 512u;
    return n > 1000 || b <= 4 * sms ? 256u : 128u;
}

constexpr int SCORE_MAX_DEVICES = 64;
std::mutex g_score_lock;
int g_score_sms[SCORE_MAX_DEVICES];   // per device: its SM count, once the kernels' shared-memory limit has been raised there
constexpr int SCORE_SMEM_MAX = 232448 - 1536;   // (the CTA kernel has 1.3 KB of its own beside the dynamic part)
constexpr size_t SM_SMEM = 233472;              // shared memory of one SM; a CTA takes 1 KB beside its own

struct ScoreDeviceGuard {
    int prev = -1;
    bool switched = false, ok = true;
    explicit ScoreDeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) {
            switched = cudaSetDevice(dev) == cudaSuccess;
            ok = switched;
        }
    }
    ~ScoreDeviceGuard() {
        if (switched && prev >= 0) cudaSetDevice(prev);
    }
};

}  // namespace

extern "C" int atrex_score_aggregate(const double* d_roofline_s, const uint32_t* d_unit_op, uint64_t n_units,
                                     const double* d_t_cand, const uint8_t* d_correct, uint64_t n_candidates,
                                     const double* d_w, uint32_t n_ops, double* d_s_agg, double* d_s_op,
                                     uint64_t* d_errors, void* stream) {
    if (n_candidates == 0) return ATREX_OK;
    if (!d_roofline_s || !d_unit_op || !d_t_cand || !d_correct || !d_w || !d_s_agg) return ATREX_ERR_INVALID;
    if (n_units == 0 || n_ops == 0) return ATREX_ERR_INVALID;
    if (n_units > ATREX_SCORE_MAX_UNITS || n_ops > ATREX_SCORE_MAX_OPS || n_candidates > 0x7FFFFFFFull)
        return ATREX_ERR_TOO_LARGE;
    // the inputs live on some device: run there, and raise that device's shared-memory limit once
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, d_t_cand) != cudaSuccess || attr.type != cudaMemoryTypeDevice || attr.device < 0 ||
        attr.device >= SCORE_MAX_DEVICES) {
        cudaGetLastError();
        return ATREX_ERR_INVALID;
    }
    ScoreDeviceGuard guard(attr.device);
    if (!guard.ok) {
        cudaGetLastError();
        return ATREX_ERR_CUDA;
    }
    int n_sms;
    {
        std::lock_guard<std::mutex> hold(g_score_lock);
        if (g_score_sms[attr.device] == 0) {
            int v = 0;
            if (cudaFuncSetAttribute(score_bins_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_bins_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_bins_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_bins_kernel<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_warp_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_warp_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaFuncSetAttribute(score_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_SMEM_MAX) != cudaSuccess ||
                cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, attr.device) != cudaSuccess) {
                cudaGetLastError();
                return ATREX_ERR_CUDA;
            }
            g_score_sms[attr.device] = v;
        }
        n_sms = g_score_sms[attr.device];
    }
    const uint32_t n = (uint32_t)n_units, b = (uint32_t)n_candidates;
    ull* errors = reinterpret_cast<ull*>(d_errors);
    // A lane to an operator up to a mean group of 24, two above (8 000 candidates: 440 units in 14 operators 70 -> 29 us,
    // 1 000 units in 25 operators 181 -> 62; 440 units in 27 operators 31, by pairs 42).
    const bool pairs = n > 24u * n_ops;
    const uint32_t slots = warp_slots(n, n_ops, pairs);
    const WarpLayout wl(n, n_ops, slots);
    uint32_t warps = 0, per_sm = 0;    // the split of an SM's shared memory that holds most warps
    for (uint32_t c = WARP_KERNEL_CTAS; c >= 1; --c) {
        const size_t room = SM_SMEM / c - 1024 < (size_t)SCORE_SMEM_MAX ? SM_SMEM / c - 1024 : (size_t)SCORE_SMEM_MAX;
        uint32_t k = room > wl.warps ? (uint32_t)((room - wl.warps) / wl.warp_bytes) : 0u;
        if (k > WARP_KERNEL_THREADS / 32) k = WARP_KERNEL_THREADS / 32;
        if (k * c > warps * per_sm) warps = k, per_sm = c;
    }
    const uint32_t sms = (uint32_t)n_sms, held = warps * per_sm;
    const bool warp_each = by_warps(n, n_ops, b, sms, held) && slots + n < SLOT_MASK;
    if (n >= BINS_GROUP_MIN * n_ops && n_ops <= BINS_OPS_MAX && !(warp_each && n <= BINS_UNITS_FEW)) {
        const uint32_t threads = bins_threads(n, n_ops, b, sms), log_bins = log_bins_for(n, n_ops);
        const size_t smem = BinsLayout(n, n_ops, log_bins, threads).total;
        auto* kernel = threads == 128 ? score_bins_kernel<128> : threads == 256 ? score_bins_kernel<256> : threads == 512 ? score_bins_kernel<512> : score_bins_kernel<1024>;
        per_sm = (uint32_t)(SM_SMEM / (smem + 1024 + 64));
        if (per_sm > (uint32_t)bins_ctas((int)threads)) per_sm = (uint32_t)bins_ctas((int)threads);
        if (per_sm < 1) per_sm = 1;
        kernel<<<b < sms * per_sm ? b : sms * per_sm, threads, smem, (cudaStream_t)stream>>>(
            d_roofline_s, d_unit_op, n, d_t_cand, d_correct, b, d_w, n_ops, log_bins, d_s_agg, d_s_op, errors);
    } else if (warp_each) {
        const uint32_t want = (b + warps - 1) / warps, most = (uint32_t)n_sms * per_sm;
        const size_t warp_smem = wl.warps + (size_t)wl.warp_bytes * warps;
        auto* kernel = pairs ? score_warp_kernel<true> : score_warp_kernel<false>;
        kernel<<<want < most ? want : most, warps * 32, warp_smem, (cudaStream_t)stream>>>(
            d_roofline_s, d_unit_op, n, d_t_cand, d_correct, b, d_w, n_ops, slots, d_s_agg, d_s_op, errors);
    } else {
        const uint32_t threads = cta_threads(n, n_ops, b, sms);
        const size_t smem = CtaLayout(n, n_ops, threads).total;
        per_sm = (uint32_t)(SM_SMEM / (smem + 2560));
        if (per_sm > 1024u / threads) per_sm = 1024u / threads;   // (64 registers a thread)
        if (per_sm < 1) per_sm = 1;
        const uint32_t most = (uint32_t)n_sms * per_sm;
        score_cta_kernel<<<b < most ? b : most, threads, smem, (cudaStream_t)stream>>>(
            d_roofline_s, d_unit_op, n, d_t_cand, d_correct, b, d_w, n_ops, d_s_agg, d_s_op, errors);
    }
    return cudaGetLastError() == cudaSuccess ? ATREX_OK : ATREX_ERR_CUDA;
}
