// Report slots against a runtime whose calls are counted: argv[1] names the case, exit code 0 = as expected.
#include "host_wait.h"

#include <cstdio>
#include <cstdlib>
#include <string>

using namespace atrex;

static int g_syncs = 0;
static uint32_t g_held = ~0u, g_other = ~0u;
static cudaStream_t g_stream = nullptr;
static bool g_no_memory = false;

extern "C" cudaError_t cudaHostAlloc(void** out, size_t bytes, unsigned) {
    if (g_no_memory) return cudaErrorMemoryAllocation;
    *out = calloc(1, bytes);
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    ++g_syncs;
    g_stream = s;
    ReportSlot other(nullptr);     // another call that comes while kernels of the first one still run
    g_other = other.number();
    other.get()->done = 1;
    return cudaSuccess;
}

int main(int argc, char** argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    const cudaStream_t s = (cudaStream_t)0x1234;
    if (what == "cut_short") {     // the last kernel never ran
        {
            ReportSlot slot(s);
            g_held = slot.number();
        }
        ReportSlot next(s);
        next.get()->done = 1;
        return g_syncs == 1 && g_stream == s && g_other != g_held && next.number() == g_held ? 0 : 1;
    }
    if (what == "answered") {
        {
            ReportSlot slot(s);
            slot.get()->done = 1;
            if (slot.wait() != cudaSuccess) return 2;
        }
        return g_syncs == 0 ? 0 : 1;
    }
    if (what == "no_memory") {
        g_no_memory = true;
        {
            ReportSlot slot(s);
            if (slot.get() != nullptr) return 2;
        }
        return g_syncs == 0 ? 0 : 1;
    }
    return 3;
}
