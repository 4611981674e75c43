// Operator importance weights exactly as Eq. 2-3 state them.
//
//   Eq. 2  D[i][a][phi] = summed duration of operator i's invocations in application a, phase phi;
//          D_a[phi] = sum over all operators of D[.][a][phi]
//   Eq. 3  wtilde_i = sum_a p_a (1/|Phi_i|) sum_{phi in Phi_i} D[i][a][phi] / D_a[phi];
//          w_i = wtilde_i / sum over retained j of wtilde_j
//
// The group-by runs over (operator, application, phase) cells.  Two routes:
//   local   the cells fit a CTA's shared memory and there are records enough: every CTA sums its share there
//           and adds its cells to the global ones at the end (70 M records into 11 560 cells: 1 056 -> 197 us,
//           most of it DRAM time; the few hot cells of a small trace no longer queue at L2)
//   direct  one 64-bit reduction per record into L2.  (Binning the records by cell first, entries kept in L2, one
//           CTA summing each bin in shared memory, was measured for 10^6 cells: 2.0 ms per 2^28 records against
//           1.8 by reductions; the bin pass spends its time between barriers.)
// While fewer than 2^32 records have been ingested no cell can overflow 64 bits (durations are below 2^32), so
// reductions need not return a value; from then on every add does and wraps are counted in a second limb.
// The floating-point part sums in ascending phase, application and operator order with every operation
// rounded once, which gives one bit pattern.
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "kernels.h"

using namespace atrex;

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t LOCAL_CELLS_MAX = 28 * 1024; // 8 bytes each

}  // namespace

struct atrex_eq3 {
    uint32_t n_apps = 0, n_ops = 0, n_phases = 0;
    int device = 0, n_sms = 0;
    unsigned char* arena = nullptr;   // one allocation for everything below
    ull* d_lo = nullptr;          // [n_phases][n_ops][n_apps] low 64 bits of D
    ull* d_hi = nullptr;          //                           wraps of the low limb
    double* d_den = nullptr;      // [n_phases][n_apps] fl(D_a[phi])
    double* d_pa = nullptr;       // [n_apps] card-hour fractions
    double* d_wt = nullptr;       // [n_ops] wtilde
    uint32_t* d_present = nullptr;   // [n_ops] bit phi: operator i has time in phase phi (cleared by every finalize)
    ull* d_ctl = nullptr;         // [0] rejected, [1] finalize: operators done
    size_t h_bytes = 0;
    double* h_out = nullptr;      // pinned: w [n_ops], wtilde [n_ops], rejected, number of the finalize; then the retained flags [n_ops]
    ull n_finalized = 0;
    size_t cells = 0;
    double c_total = 0.0;
    bool hi_used = false;
    ull n_ingested = 0;           // records handed to ingest since create/reset (decides the carry handling)
};

namespace {

struct Guard {
    int prev = -1;
    bool switched = false;
    explicit Guard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) switched = cudaSetDevice(dev) == cudaSuccess;
    }
    ~Guard() {
        if (prev >= 0 && switched) cudaSetDevice(prev);
    }
};

struct Eq3Params {
    const uint4* recs;
    ull n;
    uint32_t n_apps, n_ops, n_phases, cells;
    ull *lo, *hi, *rejected;
};

__device__ __forceinline__ void red_add_u64(ull* p, ull v) {
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
template <bool CARRY>
__device__ __forceinline__ void add_cell(const Eq3Params& p, uint32_t cell, ull v) {
    if (CARRY) {
        const ull old = atomicAdd(&p.lo[cell], v);
        if (old + v < old) atomicAdd(&p.hi[cell], 1ull);
    } else {
        red_add_u64(&p.lo[cell], v);
    }
}
__device__ __forceinline__ bool cell_of(const Eq3Params& p, const uint4& r, uint32_t& cell) {
    const uint32_t op = r.y & 0xFFFFu, phase = (r.y >> 16) & 0xFFu;
    cell = (phase * p.n_ops + op) * p.n_apps + r.x;
    return r.x < p.n_apps && op < p.n_ops && phase < p.n_phases;
}
__device__ __forceinline__ void count_rejected(const Eq3Params& p, uint32_t bad) {
    bad = __reduce_add_sync(FULL, bad);
    if ((threadIdx.x & 31u) == 0 && bad) atomicAdd(p.rejected, (ull)bad);
}

// ---- direct: bound by the L2's reduction rate, ~150 G/s for random 8-byte targets
template <bool CARRY>
__global__ void __launch_bounds__(512) eq3_direct_kernel(const Eq3Params p) {
    grid_dependency_wait();
    uint32_t bad = 0;
    const ull stride = (ull)gridDim.x * 512;
    for (ull i0 = (ull)blockIdx.x * 512 + threadIdx.x; i0 < p.n; i0 += 4 * stride) {
        uint4 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * stride < p.n) r[u] = __ldcs(p.recs + i0 + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u * stride >= p.n) continue;
            uint32_t cell;
            if (cell_of(p, r[u], cell)) add_cell<CARRY>(p, cell, r[u].w);
            else ++bad;
        }
    }
    grid_dependents_launch();
    count_rejected(p, bad);
}

// ---- local: {u32 low, u32 wraps} per cell in shared memory; bound by the records' DRAM reads
__device__ __forceinline__ void smem_add(uint32_t* lo, uint32_t* hi, uint32_t at, uint32_t v) {
    const uint32_t o = atomicAdd(lo + at, v);
    if (o + v < o) atomicAdd(hi + at, 1u);
}
template <bool CARRY>
__global__ void __launch_bounds__(1024) eq3_local_kernel(const Eq3Params p) {
    extern __shared__ __align__(16) uint32_t s_cells[];
    uint32_t *s_lo = s_cells, *s_hi = s_cells + p.cells;
    for (uint32_t i = threadIdx.x; i < 2 * p.cells; i += blockDim.x) s_cells[i] = 0;
    __syncthreads();
    grid_dependency_wait();
    uint32_t bad = 0;
    const ull stride = (ull)gridDim.x * blockDim.x;
    for (ull i0 = (ull)blockIdx.x * blockDim.x + threadIdx.x; i0 < p.n; i0 += 4 * stride) {
        uint4 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * stride < p.n) r[u] = __ldcs(p.recs + i0 + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u * stride >= p.n) continue;
            uint32_t cell;
            if (cell_of(p, r[u], cell)) smem_add(s_lo, s_hi, cell, r[u].w);
            else ++bad;
        }
    }
    grid_dependents_launch();
    count_rejected(p, bad);
    __syncthreads();
    // the CTAs start at different cells, so that they do not queue at the same ones
    const uint32_t first = (uint32_t)((ull)p.cells * blockIdx.x / gridDim.x);
    for (uint32_t i = threadIdx.x; i < p.cells; i += blockDim.x) {
        uint32_t cell = first + i;
        if (cell >= p.cells) cell -= p.cells;
        const ull v = (ull)s_lo[cell] | ((ull)s_hi[cell] << 32);
        if (v != 0) add_cell<CARRY>(p, cell, v);
    }
}

// ---- D_a[phi] and Phi_i: a CTA per 32 applications and phase, its warps share the operators
constexpr int TOTAL_WARPS = 16;
__global__ void __launch_bounds__(TOTAL_WARPS * 32) eq3_app_totals_kernel(const ull* lo, const ull* hi, uint32_t n_apps, uint32_t n_ops, double* den,
                                                                          uint32_t* present) {
    __shared__ ull s_lo[TOTAL_WARPS][32], s_hi[TOTAL_WARPS][32];
    grid_dependency_wait();
    const uint32_t per_phase = (n_apps + 31) / 32, phase = blockIdx.x / per_phase;
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, app = blockIdx.x % per_phase * 32 + lane;
    ull t_lo = 0, t_hi = 0;
    for (uint32_t i0 = w; i0 < n_ops; i0 += 4 * TOTAL_WARPS) {
        ull x[4], y[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t i = i0 + u * TOTAL_WARPS;
            const bool in = i < n_ops && app < n_apps;
            const size_t cell = ((size_t)phase * n_ops + i) * n_apps + app;
            x[u] = in ? lo[cell] : 0ull;
            y[u] = in && hi ? hi[cell] : 0ull;
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            const ull s = t_lo + x[u];
            t_hi += y[u] + (s < t_lo ? 1ull : 0ull);
            t_lo = s;
            if (__any_sync(FULL, (x[u] | y[u]) != 0) && lane == 0) atomicOr(&present[i0 + u * TOTAL_WARPS], 1u << phase);
        }
    }
    grid_dependents_launch();
    s_lo[w][lane] = t_lo;
    s_hi[w][lane] = t_hi;
    __syncthreads();
    if (w != 0 || app >= n_apps) return;
    for (int k = 1; k < TOTAL_WARPS; ++k) {
        const ull s = t_lo + s_lo[k][lane];
        t_hi += s_hi[k][lane] + (s < t_lo ? 1ull : 0ull);
        t_lo = s;
    }
    den[(size_t)phase * n_apps + app] = u128_to_f64_rn(t_hi, t_lo);   // (+0.0: no time, nothing to divide)
}

// ---- wtilde_i: one CTA per operator.  The terms p_a * (1/|Phi_i|) * sum_phi D[i][a][phi] / D_a[phi] (each a fixed
// sequence of rounded operations, independent of the others) are worked out by all warps but the first, in
// chunks; the running sum over the applications, whose order is part of the result, by one thread of the
// first warp, a chunk behind.  Bound by that chain: 4 096 additions.  The last CTA forms w.
constexpr int WT_THREADS = 512;
constexpr uint32_t WT_CHUNK = 960;    // two terms per computing thread

__global__ void __launch_bounds__(WT_THREADS) eq3_wtilde_kernel(const ull* lo, const ull* hi, const double* den, const double* pa, uint32_t* present,
                                                                uint32_t n_apps, uint32_t n_ops, uint32_t n_phases, bool any_weight, double* wt,
                                                                const uint8_t* retained, ull* ctl, double* h_out, ull seq) {
    __shared__ __align__(16) double s_term[2][WT_CHUNK];
    __shared__ double s_total;
    __shared__ bool s_last;
    grid_dependency_wait();
    const uint32_t i = blockIdx.x, mask = present[i];
    const int n_phi = __popc(mask);
    double acc = 0.0;   // thread 0's
    if (n_phi != 0 && any_weight) {
        const double d_phi = (double)n_phi;
        const uint32_t chunks = (n_apps + WT_CHUNK - 1) / WT_CHUNK;
        for (uint32_t c = 0; c <= chunks; ++c) {
            if (threadIdx.x >= 32) {
                if (c < chunks) {
                    for (uint32_t k = threadIdx.x - 32; k < WT_CHUNK; k += WT_THREADS - 32) {
                        const uint32_t a = c * WT_CHUNK + k;
                        double term = 0.0;
                        if (a < n_apps) {
                            double inner = 0.0;
                            for (uint32_t p = 0; p < n_phases; ++p) {
                                if (!(mask & (1u << p))) continue;
                                const double d = den[(size_t)p * n_apps + a];
                                if (d == 0.0) continue;
                                const size_t cell = ((size_t)p * n_ops + i) * n_apps + a;
                                inner = __dadd_rn(inner, __ddiv_rn(u128_to_f64_rn(hi ? hi[cell] : 0ull, lo[cell]), d));
                            }
                            term = __dmul_rn(pa[a], __ddiv_rn(inner, d_phi));
                        }
                        s_term[c & 1][k] = term;
                    }
                }
            } else if (threadIdx.x == 0 && c > 0) {
                // (terms behind the last application are +0.0, which leaves a sum of non-negative terms as it is)
                const double2* v = reinterpret_cast<const double2*>(s_term[(c - 1) & 1]);
                const uint32_t n = min(WT_CHUNK, n_apps - (c - 1) * WT_CHUNK);
                for (uint32_t k = 0; k < (n + 15) / 16 * 8; k += 8) {
                    double2 t[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) t[u] = v[k + u];
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc = __dadd_rn(__dadd_rn(acc, t[u].x), t[u].y);
                }
            }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) {
        wt[i] = acc;
        present[i] = 0;
        __threadfence();
        s_last = atomicAdd(&ctl[1], 1ull) == n_ops - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    double total = 0.0;
    for (uint32_t i0 = 0; i0 < n_ops; i0 += WT_CHUNK) {
        for (uint32_t k = threadIdx.x; k < WT_CHUNK; k += WT_THREADS)
            s_term[0][k] = i0 + k < n_ops && retained[i0 + k] ? __ldcg(wt + i0 + k) : 0.0;
        __syncthreads();
        if (threadIdx.x == 0)
            for (uint32_t k = 0; k < min(WT_CHUNK, n_ops - i0); ++k) total = __dadd_rn(total, s_term[0][k]);
        __syncthreads();
    }
    if (threadIdx.x == 0) s_total = total;
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < n_ops; k += WT_THREADS) {
        const double v = __ldcg(wt + k);
        h_out[k] = retained[k] && s_total > 0.0 ? __ddiv_rn(v, s_total) : 0.0;
        h_out[n_ops + k] = v;
    }
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) {
        reinterpret_cast<ull*>(h_out)[2 * (size_t)n_ops] = ctl[0];
        ctl[1] = 0;
        __threadfence_system();
        reinterpret_cast<volatile ull*>(h_out)[2 * (size_t)n_ops + 1] = seq;   // the host waits for this word
    }
}

// ---- launches
cudaError_t prepare_kernels() {
    const cudaError_t e = cudaFuncSetAttribute(eq3_local_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LOCAL_CELLS_MAX * 8);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(eq3_local_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, LOCAL_CELLS_MAX * 8);
}

template <bool CARRY>
cudaError_t launch_ingest(const atrex_eq3* h, const atrex_record_t* recs, ull n, cudaStream_t s) {
    Eq3Params p;
    p.recs = (const uint4*)recs;
    p.n = n;
    p.n_apps = h->n_apps; p.n_ops = h->n_ops; p.n_phases = h->n_phases;
    p.cells = (uint32_t)h->cells;
    p.lo = h->d_lo; p.hi = h->d_hi;
    p.rejected = h->d_ctl;
    const size_t cell_bytes = h->cells * 8;
    // local: as long as every SM gets twice as many records as it has cells to add up at the end
    if (h->cells <= LOCAL_CELLS_MAX && n >= 2ull * h->cells * h->n_sms && n >= 65536) {
        const uint32_t threads = cell_bytes > 72 * 1024 ? 1024 : 512;
        uint32_t per_sm = (uint32_t)(232448 / (cell_bytes + 1024));
        if (per_sm > 2048 / threads) per_sm = 2048 / threads;
        ull grid = n / (2 * h->cells);
        if (grid > n / (4 * threads)) grid = n / (4 * threads);
        if (grid > (ull)h->n_sms * per_sm) grid = (ull)h->n_sms * per_sm;
        if (grid < 1) grid = 1;
        return launch_chained(eq3_local_kernel<CARRY>, (uint32_t)grid, threads, cell_bytes, s, p);
    }
    return launch_chained(eq3_direct_kernel<CARRY>, grid_for_work(n, 512, h->n_sms, 4), 512, 0, s, p);
}

}  // namespace

extern "C" {

int atrex_eq3_create(uint32_t n_apps, uint32_t n_ops, uint32_t n_phases, const uint32_t* app_weights, int32_t device,
                     atrex_eq3_t** out) {
    if (!out) return ATREX_ERR_INVALID;
    *out = nullptr;
    if (!app_weights || n_apps == 0 || n_ops == 0 || n_ops > 65536 || n_phases == 0 || n_phases > ATREX_MAX_PHASES)
        return ATREX_ERR_INVALID;
    const size_t cells = (size_t)n_apps * n_ops * n_phases;
    if (cells > ((size_t)1 << 28)) return ATREX_ERR_TOO_LARGE;
    atrex_eq3* h = new (std::nothrow) atrex_eq3;
    if (!h) return ATREX_ERR_NOMEM;
    h->n_apps = n_apps; h->n_ops = n_ops; h->n_phases = n_phases; h->device = device; h->cells = cells;
    // card-hour fractions: fl(c_a / fl(sum of all))
    ull c_sum = 0;
    for (uint32_t a = 0; a < n_apps; ++a) c_sum += app_weights[a];
    h->c_total = (double)c_sum;
    double* pa = (double*)malloc((size_t)n_apps * 8);
    if (!pa) {
        delete h;
        return ATREX_ERR_NOMEM;
    }
    for (uint32_t a = 0; a < n_apps; ++a) pa[a] = c_sum ? (double)app_weights[a] / h->c_total : 0.0;
    Guard g(device);
    cudaError_t e = cudaDeviceGetAttribute(&h->n_sms, cudaDevAttrMultiProcessorCount, device);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_ctl = take(16), o_present = take((size_t)n_ops * 4), o_lo = take(cells * 8), o_hi = take(cells * 8),
                 o_den = take((size_t)n_phases * n_apps * 8), o_pa = take((size_t)n_apps * 8), o_wt = take((size_t)n_ops * 8);
    if (e == cudaSuccess) e = cudaMalloc((void**)&h->arena, o);
    if (e == cudaSuccess) e = pinned_alloc((void**)&h->h_out, h->h_bytes = ((size_t)n_ops * 2 + 2) * 8 + n_ops);
    if (e == cudaSuccess) {
        h->d_ctl = (ull*)(h->arena + o_ctl);
        h->d_present = (uint32_t*)(h->arena + o_present);
        h->d_lo = (ull*)(h->arena + o_lo);
        h->d_hi = (ull*)(h->arena + o_hi);
        h->d_den = (double*)(h->arena + o_den);
        h->d_pa = (double*)(h->arena + o_pa);
        h->d_wt = (double*)(h->arena + o_wt);
        e = cudaMemset(h->arena, 0, o_den);   // control, Phi, cells
    }
    if (e == cudaSuccess) e = cudaMemcpy(h->d_pa, pa, (size_t)n_apps * 8, cudaMemcpyHostToDevice);
    free(pa);
    if (e == cudaSuccess) e = prepare_kernels();
    if (e != cudaSuccess) {
        cudaGetLastError();
        atrex_eq3_destroy(h);
        return e == cudaErrorMemoryAllocation ? ATREX_ERR_NOMEM : ATREX_ERR_CUDA;
    }
    *out = h;
    return ATREX_OK;
}

void atrex_eq3_destroy(atrex_eq3_t* h) {
    if (!h) return;
    Guard g(h->device);
    cudaDeviceSynchronize();
    cudaFree(h->arena);
    pinned_free(h->h_out, h->h_bytes);
    delete h;
}

int atrex_eq3_reset(atrex_eq3_t* h, void* stream) {
    if (!h) return ATREX_ERR_INVALID;
    Guard g(h->device);
    cudaStream_t s = (cudaStream_t)stream;
    // control, Phi, low limbs; the second limb only where wraps were counted
    const unsigned char* end = (const unsigned char*)(h->hi_used ? h->d_hi + h->cells : h->d_lo + h->cells);
    if (cudaMemsetAsync(h->arena, 0, end - h->arena, s) != cudaSuccess) return ATREX_ERR_CUDA;
    h->n_ingested = 0;
    h->hi_used = false;
    return ATREX_OK;
}

int atrex_eq3_ingest(atrex_eq3_t* h, const atrex_record_t* d_records, uint64_t n, void* stream) {
    if (!h) return ATREX_ERR_INVALID;
    if (n == 0) return ATREX_OK;
    if (!d_records || ((uintptr_t)d_records & 15u)) return ATREX_ERR_INVALID;
    Guard g(h->device);
    // below 2^32 records in total no cell's 64-bit sum can wrap: reductions that return nothing
    const bool carry = h->n_ingested + n >= (1ull << 32);
    h->n_ingested += n;
    h->hi_used |= carry;
    const cudaError_t e = carry ? launch_ingest<true>(h, d_records, n, (cudaStream_t)stream) : launch_ingest<false>(h, d_records, n, (cudaStream_t)stream);
    return e == cudaSuccess ? ATREX_OK : ATREX_ERR_CUDA;
}

int atrex_eq3_finalize(atrex_eq3_t* h, const uint8_t* h_retained, double* h_w, double* h_wtilde, uint64_t* h_rejected,
                       void* stream) {
    if (!h || !h_w) return ATREX_ERR_INVALID;
    Guard g(h->device);
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t n_ops = h->n_ops;
    // the flags are read and the results written by the kernels, in pinned memory
    uint8_t* retained = (uint8_t*)(h->h_out + 2 * (size_t)n_ops + 2);
    if (h_retained) memcpy(retained, h_retained, n_ops);
    else memset(retained, 1, n_ops);
    const ull* hi = h->hi_used ? h->d_hi : nullptr;
    const volatile ull* done = (const volatile ull*)h->h_out + 2 * (size_t)n_ops + 1;
    const ull seq = ++h->n_finalized;
    *(volatile ull*)done = 0;    // (a block from the pool holds whatever its last owner left)
    if (launch_chained(eq3_app_totals_kernel, (h->n_apps + 31) / 32 * h->n_phases, TOTAL_WARPS * 32, 0, s, h->d_lo, hi, h->n_apps, n_ops, h->d_den,
                       h->d_present) != cudaSuccess)
        return ATREX_ERR_CUDA;
    const bool any_weight = h->c_total != 0.0;
    if (launch_chained(eq3_wtilde_kernel, n_ops, WT_THREADS, 0, s, h->d_lo, hi, h->d_den, h->d_pa, h->d_present, h->n_apps, n_ops, h->n_phases,
                       any_weight, h->d_wt, retained, h->d_ctl, h->h_out, seq) != cudaSuccess)
        return ATREX_ERR_CUDA;
    if (wait_for_kernel([=] { return *done == seq; }, s) != cudaSuccess) return ATREX_ERR_CUDA;
    memcpy(h_w, h->h_out, (size_t)n_ops * 8);
    if (h_wtilde) memcpy(h_wtilde, h->h_out + n_ops, (size_t)n_ops * 8);
    if (h_rejected) memcpy(h_rejected, h->h_out + 2 * (size_t)n_ops, 8);
    return ATREX_OK;
}

}  // extern "C"
