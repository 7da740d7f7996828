// csrc/memory.cu on a made-up driver (host memory addresses that nothing touches, a limited amount of them), for the unit
// test that needs no GPU.
#include <map>

#include "../paper_2607_21985_b200/csrc/memory.cu"

static size_t g_limit = 0, g_used = 0;
static std::map<void*, size_t> g_live;
static uintptr_t g_next = uintptr_t(1) << 40;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    if (g_used + n > g_limit) return cudaErrorMemoryAllocation;
    *p = reinterpret_cast<void*>(g_next);
    g_next += n + 4096;
    g_used += n;
    g_live[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = g_live.find(p);
    if (it == g_live.end()) return cudaErrorInvalidValue;
    g_used -= it->second;
    g_live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t*, const cudaMemPoolProps*) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaErrorNotSupported; }
cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t, cudaStream_t) { return cudaErrorNotSupported; }

void shim_limit(unsigned long long n) { g_limit = n; }
unsigned long long shim_used(void) { return g_used; }
int shim_alloc(unsigned long long n, spdp::DeviceBlock* out) { return spdp::handle_alloc(0, n, out); }
void shim_give(spdp::DeviceBlock* b, int idle) { spdp::handle_give(0, *b, idle != 0); }
void shim_give_back_all(void) { spdp::give_back_all(); }
}
namespace spdp {
void note_cuda_error(cudaError_t, const char*) {}
}
