// A CUDA runtime without a GPU: it keeps the library's launches instead of
// running them, so that the host side (which kernel, how many chunks, which
// limits) can be tested on a CPU. The library's objects are linked against it.
//
// A launch above its kernel's shared-memory limit is refused, as the runtime
// does, and the limit is held per kernel, whichever thread set it.
#include <chrono>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>

#include "prcr_internal.h"

namespace {

struct State {
    std::mutex mu;
    std::map<const void*, std::string> names;
    std::map<const void*, size_t> limits;
    std::string log;
    int lowered = 0;
};
State& st() {
    static State* s = new State;  // used by static initialisers of the objects
    return *s;
}

}  // namespace

extern "C" {

// launches since the last call, one per line: kernel, grid, block, dynamic
// shared memory, and of a decode its splits, chunk and team, of a rebind the
// CTAs that prefetch rows, of a cached selection whether keys are read from
// the cache (not the workspace)
__attribute__((visibility("default"))) size_t fake_log(char* out, size_t n) {
    std::lock_guard<std::mutex> g(st().mu);
    std::snprintf(out, n, "%s", st().log.c_str());
    const size_t len = st().log.size();
    st().log.clear();
    return len;
}
// times a kernel's shared-memory limit was lowered
__attribute__((visibility("default"))) int fake_lowered() { return st().lowered; }

void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    st().names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaErrorNotSupported; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaErrorNotSupported; }

cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;  // SMs
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = reinterpret_cast<void*>(uintptr_t(1) << 40);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    {
        std::lock_guard<std::mutex> g(st().mu);
        size_t& have = st().limits[f];
        st().lowered += have > size_t(v);
        have = size_t(v);
    }
    std::this_thread::sleep_for(std::chrono::microseconds(50));  // another thread's turn
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
    // as a GB300 answers for one CTA per SM: clusters do not fill every GPC
    static const int held[17] = {0, 152, 70, 46, 36, 28, 23, 15, 15, 15, 13, 8, 8, 7, 7, 7, 7};
    *n = held[c->gridDim.x];
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    std::lock_guard<std::mutex> g(st().mu);
    const auto it = st().limits.find(f);
    if (c->dynamicSmemBytes > (it == st().limits.end() ? size_t(48 * 1024) : it->second)) return cudaErrorInvalidValue;
    const std::string& name = st().names[f];
    char line[512];
    int n = std::snprintf(line, sizeof line, "%s %u %u %u %u %zu", name.c_str(), c->gridDim.x, c->gridDim.y,
                          c->gridDim.z, c->blockDim.x, c->dynamicSmemBytes);
    if (name.find("decode") != std::string::npos) {
        const auto* a = static_cast<const prcr::DecodeArgs*>(args[0]);
        std::snprintf(line + n, sizeof line - size_t(n), " %d %d %d", a->splits, a->chunk, a->team);
    } else if (name.find("rebind_kernel") != std::string::npos) {
        std::snprintf(line + n, sizeof line - size_t(n), " %d", static_cast<const prcr::RebindArgs*>(args[0])->early_ctas);
    } else if (name.find("select_fused") != std::string::npos || name.find("select_logits") != std::string::npos) {
        const auto* a = static_cast<const prcr::SelectArgs*>(args[0]);
        std::snprintf(line + n, sizeof line - size_t(n), " %d", a->cache_k && a->cache_k != reinterpret_cast<const uint16_t*>(a->logits));
    }
    st().log += std::string(line) + "\n";
    return cudaSuccess;
}

}  // extern "C"
