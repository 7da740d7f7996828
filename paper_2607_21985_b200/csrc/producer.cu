// The operation in front of a dynamically pruned projection, fused with the pruning decision
// (Sec. 6: DP variants that materialise a mask feed the same column-selection interface; Sec. 4.2
// step (3): the decision is a magnitude test against a threshold calibrated offline).  For a gated
// MLP the down-projection's input is x = silu(gate) * up; this kernel writes x (fp16) and, in the
// same pass, the K-bit mask "NOT(|x_j| <= thr)" that spdp_spmspv takes with SPDP_DP_MASK, so the
// decode kernel's list phase reads one bit per column instead of testing activations again, and a
// caller with another selection rule can write the mask itself.
#include "spdp_internal.h"

namespace spdp {
namespace {

// gate and up are not __restrict__: the kernels that write them may still run when this one starts, and the read-only path that
// const __restrict__ allows is for data that nothing writes in the kernel's lifetime.
__global__ void swiglu_dp_kernel(const __half* gate, const __half* up, int64_t K, float thr,
                                 __half* __restrict__ x_out, uint32_t* __restrict__ mask_out, int* __restrict__ count) {
    // The kernel after this one (the decode call) may start its matrix-only prologue now; what the kernel before this one
    // wrote or still reads (gate, up, x_out, mask_out) is touched only after the wait.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    bool active = false;
    if (j < K) {
        const float g = __half2float(gate[j]), u = __half2float(up[j]);
        const __half x = __float2half_rn(g / (1.0f + expf(-g)) * u);        // silu(g) * u in fp32, rounded once
        x_out[j] = x;
        active = !(fabsf(__half2float(x)) <= thr);                          // the decision is taken on the stored fp16 value
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, active);
    if ((threadIdx.x & 31) == 0 && (j >> 5) < ((K + 31) >> 5)) {
        mask_out[j >> 5] = m;
        if (count != nullptr && m != 0u) atomicAdd(count, __popc(m));
    }
}

// Fetches the vectors of a host-vector call over the bus: one 16-byte load per thread where the address allows it.
__global__ void fetch_kernel(const __half* x, int K, __half* __restrict__ x_out, const uint32_t* mask, int mask_words,
                             uint32_t* __restrict__ mask_out) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");                  // the buffers may still be read by the call before
    const int t = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    const bool wide = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
    const int pieces = wide ? K / 8 : 0;
    for (int i = t; i < pieces; i += n) reinterpret_cast<uint4*>(x_out)[i] = reinterpret_cast<const uint4*>(x)[i];
    for (int i = 8 * pieces + t; i < K; i += n) x_out[i] = x[i];
    for (int i = t; i < mask_words; i += n) mask_out[i] = mask[i];
}

}  // namespace

constexpr int kFetchThreads = 128;

spdp_status set_fetch_node(cudaGraphExec_t exec, cudaGraphNode_t node, const __half* x, int64_t K, __half* x_out, const uint32_t* mask,
                           int mask_words, uint32_t* mask_out) {
    int k32 = static_cast<int>(K);
    void* args[6] = {&x, &k32, &x_out, &mask, &mask_words, &mask_out};
    cudaKernelNodeParams k = {};
    k.func = reinterpret_cast<void*>(fetch_kernel);
    k.gridDim = dim3(static_cast<unsigned>((K + 8 * kFetchThreads - 1) / (8 * kFetchThreads)));
    k.blockDim = dim3(kFetchThreads);
    k.kernelParams = args;
    SPDP_CUDA_TRY(cudaGraphExecKernelNodeSetParams(exec, node, &k));
    return SPDP_OK;
}

spdp_status launch_fetch(const __half* x, int64_t K, __half* x_out, const uint32_t* mask, int mask_words, uint32_t* mask_out, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((K + 8 * kFetchThreads - 1) / (8 * kFetchThreads)));
    cfg.blockDim = dim3(kFetchThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SPDP_CUDA_TRY(cudaLaunchKernelEx(&cfg, fetch_kernel, x, static_cast<int>(K), x_out, mask, mask_words, mask_out));
    return SPDP_OK;
}

spdp_status launch_swiglu_dp(const __half* gate, const __half* up, int64_t K, float thr, __half* x_out, uint32_t* mask_out,
                             int* count, cudaStream_t s) {
    if (count != nullptr) SPDP_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(int), s));
    const int threads = 256;
    const int64_t blocks = (((K + 31) / 32) * 32 + threads - 1) / threads;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SPDP_CUDA_TRY(cudaLaunchKernelEx(&cfg, swiglu_dp_kernel, gate, up, K, thr, x_out, mask_out, count));
    return SPDP_OK;
}

}  // namespace spdp
