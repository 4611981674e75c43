// Pool of pinned host blocks (pinning one takes half a millisecond, longer than a build of a small trace).  One
// size for all, mapped and usable from every device; larger requests are pinned and released on the spot.
#include <mutex>

#include "kernels.h"

namespace atrex {

namespace {
constexpr size_t BLOCK_BYTES = 512 << 10;
constexpr int POOL_MAX = 8;
std::mutex g_lock;
void* g_free[POOL_MAX];
int g_n = 0;
}  // namespace

cudaError_t pinned_alloc(void** out, size_t bytes) {
    *out = nullptr;
    if (bytes <= BLOCK_BYTES) {
        std::lock_guard<std::mutex> hold(g_lock);
        if (g_n > 0) {
            *out = g_free[--g_n];
            return cudaSuccess;
        }
    }
    return cudaHostAlloc(out, bytes <= BLOCK_BYTES ? BLOCK_BYTES : bytes, cudaHostAllocMapped | cudaHostAllocPortable);
}

void pinned_free(void* block, size_t bytes) {
    if (!block) return;
    if (bytes <= BLOCK_BYTES) {
        std::lock_guard<std::mutex> hold(g_lock);
        if (g_n < POOL_MAX) {
            g_free[g_n++] = block;
            return;
        }
    }
    cudaFreeHost(block);
}

}  // namespace atrex
