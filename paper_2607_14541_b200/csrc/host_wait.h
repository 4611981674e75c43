// What the host does until a kernel has answered in pinned memory (host code only).
#pragma once
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <mutex>

#include <cuda_runtime_api.h>

namespace atrex {

typedef unsigned long long ull;

// Waits until `done()` sees what a kernel on `s` wrote to pinned memory as its last act, which the host notices
// several microseconds before the stream counts as idle; after a millisecond, or if the kernel cannot get there,
// by the stream itself.
template <typename Done>
inline cudaError_t wait_for_kernel(Done done, cudaStream_t s) {
    const auto limit = std::chrono::steady_clock::now() + std::chrono::milliseconds(1);
    for (uint32_t i = 1;; ++i) {
        if (done()) {
            std::atomic_thread_fence(std::memory_order_acquire);
            return cudaSuccess;
        }
        if ((i & 63u) == 0 && std::chrono::steady_clock::now() > limit) return cudaStreamSynchronize(s);
    }
}

constexpr int REPORT_SLOTS = 32;
struct BinReport {               // in pinned host memory, written by the kernels of a sort or ranking
    ull overflow, counter, total_lo, total_hi, n_keep, covered_lo, covered_hi, too_large;
    ull done;                    // the call's last kernel is through
    ull pad[7];
};

// Reports from the device: a few pinned slots for the whole process, handed out per call (a call that finds
// none free waits for one; calls are milliseconds at most).  A call that ends before its last kernel has said so --
// a launch in the middle of the chain failed -- waits for the stream before it gives the slot back: the kernels
// already launched may still write to it.
class ReportSlot {
public:
    explicit ReportSlot(cudaStream_t s) : stream_(s) {
        std::unique_lock<std::mutex> hold(lock());
        if (pool() == nullptr && cudaHostAlloc((void**)&pool(), SLOTS * sizeof(BinReport), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        freed().wait(hold, [] { return used() != 0xFFFFFFFFu; });
        slot_ = __builtin_ctz(~used());
        used() |= 1u << slot_;
        memset((void*)get(), 0, sizeof(BinReport));
    }
    ~ReportSlot() {
        if (slot_ < 0) return;
        if (*(const volatile ull*)&get()->done == 0) cudaStreamSynchronize(stream_);
        std::lock_guard<std::mutex> hold(lock());
        used() &= ~(1u << slot_);
        freed().notify_one();
    }
    ReportSlot(const ReportSlot&) = delete;
    ReportSlot& operator=(const ReportSlot&) = delete;
    BinReport* get() const { return slot_ < 0 ? nullptr : pool() + slot_; }
    uint32_t number() const { return (uint32_t)slot_; }
    // waits for the call's last kernel
    cudaError_t wait() const {
        const volatile ull* done = &get()->done;
        return wait_for_kernel([=] { return *done != 0; }, stream_);
    }

private:
    static constexpr int SLOTS = REPORT_SLOTS;
    static std::mutex& lock() { static std::mutex m; return m; }
    static std::condition_variable& freed() { static std::condition_variable c; return c; }
    static BinReport*& pool() { static BinReport* p = nullptr; return p; }
    static uint32_t& used() { static uint32_t u = 0; return u; }
    cudaStream_t stream_;
    int slot_ = -1;
};

}  // namespace atrex
