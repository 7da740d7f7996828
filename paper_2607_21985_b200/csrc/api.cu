// C ABI of libspdp (declared in spdp.h): argument checks, handle life cycle, host-side layout
// of the split-K work partition.  Every numerical step runs in the kernels of pack.cu and
// spmspv.cu.
#include <cuda.h>

#include <cstdio>
#include <cstring>
#include <new>

#include "spdp_hostdev.h"
#include "spdp_internal.h"

namespace spdp {

static thread_local char g_cuda_error[256] = "";

void note_cuda_error(cudaError_t e, const char* what) {
    std::snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s (%s)", what, cudaGetErrorName(e),
                  cudaGetErrorString(e));
    cudaGetLastError();   // clear the sticky-free error state
}

namespace {

// Makes `device` current for a scope.
struct DeviceScope {
    int before = -1;
    explicit DeviceScope(int device) {
        if (cudaGetDevice(&before) != cudaSuccess || before == device || cudaSetDevice(device) != cudaSuccess) before = -1;
    }
    ~DeviceScope() {
        if (before >= 0) cudaSetDevice(before);
    }
};

void drop_host_graph(spdp_matrix* h) {
    if (h->host_exec != nullptr) cudaGraphExecDestroy(h->host_exec);
    if (h->host_graph != nullptr) cudaGraphDestroy(h->host_graph);
    h->host_exec = nullptr;
    h->host_graph = nullptr;
}

void release(spdp_matrix* h) {
    if (h == nullptr) return;
    {
        DeviceScope on(h->device);
        // the handle's memory may be in use on any stream (cudaFree would wait for them too)
        const bool idle = cudaDeviceSynchronize() == cudaSuccess;
        for (DeviceBlock* b : {&h->arrays, &h->values_block, &h->workspace_block, &h->packing}) handle_give(h->device, *b, idle);
        if (!idle) cudaGetLastError();
        cudaFree(h->probe_items);
        cudaFree(h->probe_count);
        drop_host_graph(h);
        if (h->capture_stream != nullptr) cudaStreamDestroy(h->capture_stream);
    }
    count_handle(h->device, -1);
    h->magic = 0;
    delete h;
}

spdp_status new_handle(int64_t M, int64_t K, int pad_elems, spdp_matrix** out) {
    if (M < 1 || K < 1 || M > (int64_t(1) << 30) || K > (int64_t(1) << 30)) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (pad_elems != 8 && pad_elems != 1 && pad_elems != 32) return SPDP_ERR_UNSUPPORTED_SHAPE;
    spdp_matrix* h = new (std::nothrow) spdp_matrix();
    if (h == nullptr) return SPDP_ERR_ALLOC;
    std::memset(h, 0, sizeof(*h));
    h->magic = kMagic;
    h->M = M;
    h->K = K;
    h->R = (M + kTileM - 1) / kTileM;
    h->C = (K + kTileK - 1) / kTileK;
    h->NGT = h->R * h->C;
    h->pad_elems = pad_elems;
    // the kernel packs a column-tile index and a 6-bit count into 32 bits
    if (h->NGT * kTileK >= (int64_t(1) << 26)) { delete h; return SPDP_ERR_UNSUPPORTED_SHAPE; }
    cudaError_t e = cudaGetDevice(&h->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) { note_cuda_error(e, "device query"); delete h; return SPDP_ERR_CUDA; }
    count_handle(h->device, 1);
    *out = h;
    return SPDP_OK;
}

// Allocates the arrays whose sizes follow from the shape (on `s`), as one piece.
spdp_status alloc_arrays(spdp_matrix* h, cudaStream_t s) {
    const int64_t cols = h->NGT * kTileK;
    size_t at = 0;
    auto place = [&](size_t bytes) {
        const size_t here = at;
        at += (bytes + 255) / 256 * 256;
        return here;
    };
    const size_t bitmap = place(cols * kWordsPerCol * sizeof(uint64_t)), colinfo = place(cols * sizeof(uint32_t)),
                 tileoffset = place((h->NGT + 1) * sizeof(uint32_t)), scales = place(h->q4 ? cols * sizeof(__half) : 0),
                 x = place(h->K * sizeof(__half)), mask = place((h->K + 31) / 32 * sizeof(uint32_t)), y = place(h->M * sizeof(float)),
                 status = place(2 * sizeof(int) + kPackTotals * sizeof(unsigned long long));
    spdp_status st = handle_alloc(h->device, at, &h->arrays);
    if (st != SPDP_OK) return st;
    char* base = static_cast<char*>(h->arrays.p);
    h->bitmap = reinterpret_cast<uint64_t*>(base + bitmap);
    h->colinfo = reinterpret_cast<uint32_t*>(base + colinfo);
    h->tileoffset = reinterpret_cast<uint32_t*>(base + tileoffset);
    if (h->q4) h->scales = reinterpret_cast<__half*>(base + scales);
    h->x_stage = reinterpret_cast<__half*>(base + x);
    h->mask_stage = reinterpret_cast<uint32_t*>(base + mask);
    h->y_stage = base + y;
    h->status_word = reinterpret_cast<int*>(base + status);
    h->pack_totals = reinterpret_cast<unsigned long long*>(h->status_word + 2);
    SPDP_CUDA_TRY(cudaMemsetAsync(h->status_word, 0, 2 * sizeof(int) + kPackTotals * sizeof(unsigned long long), s));
    return SPDP_OK;
}

// Chooses the number of CTAs (the kernel cuts the NGT GTiles into that many contiguous ranges) and (re)allocates what
// depends on it: the split-K workspaces (all zero = every tree node empty).  The caller synchronises `s`, so that the
// first call on any stream finds every tree node empty.
spdp_status build_partition(spdp_matrix* h, int num_ctas, cudaStream_t s) {
    const int64_t NGT = h->NGT;
    int P = num_ctas > 0 ? num_ctas : hostdev::default_ctas(h->R, h->C, h->sm_count * default_ctas_per_sm());
    if (P > 1024) P = 1024;          // the kernel's range arithmetic is 32-bit: NGT < 2^22 times P must fit
    if (P > NGT) P = static_cast<int>(NGT);
    if (P < 1) P = 1;
    const int64_t one = static_cast<int64_t>(P) * kTileM * sizeof(float);    // one row of split-K tree nodes per CTA
    const int64_t bytes = one + batch_workspace_bytes(P);
    // the new workspace first: where there is no memory for it the handle keeps the one it has
    DeviceBlock fresh = {};
    const spdp_status st = handle_alloc(h->device, bytes, &fresh);
    if (st != SPDP_OK) return st;
    const cudaError_t e = cudaMemsetAsync(fresh.p, 0, bytes, s);
    if (e != cudaSuccess) {
        handle_give(h->device, fresh, true);
        SPDP_CUDA_TRY(e);
    }
    handle_give(h->device, h->workspace_block, true);      // idle: a new handle has none, spdp_set_num_ctas has waited for the device
    h->workspace_block = fresh;
    h->workspace = static_cast<float*>(fresh.p);
    h->workspace_batch = h->workspace + P * kTileM;
    h->workspace_bytes = bytes;
    h->num_ctas = P;
    // a recorded host-vector call holds the old workspace and CTA count: it is recorded anew
    drop_host_graph(h);
    h->host_calls = 0;
    return SPDP_OK;
}

// The rest of a handle's set-up; synchronises `s`.
spdp_status finish_handle(spdp_matrix* h, cudaStream_t s) {
    spdp_status st = configure_spmspv_kernel();
    if (st != SPDP_OK) return st;
    st = configure_spmspv_batch_kernel();
    if (st != SPDP_OK) return st;
    st = configure_spmm_kernel();
    if (st != SPDP_OK) return st;
    st = configure_spmspv_q4_kernel();
    if (st != SPDP_OK) return st;
    SPDP_CUDA_TRY(cudaStreamSynchronize(s));
    handle_give(h->device, h->packing, true);
    return SPDP_OK;
}

constexpr int kBatchViaSingleCalls = 2;   // spdp_spmspv_batch: up to this many tokens go through the single-vector kernel

// The decode kernel of the handle's Values variant (fp16 values, or 4-bit codes with scales).
spdp_status launch_decode(const spdp_matrix* h, const __half* x, int rule, float thr, const uint32_t* mask, void* y,
                          int ydt, cudaStream_t s) {
    return h->q4 ? launch_spmspv_q4(h, x, rule, thr, mask, y, ydt, s) : launch_spmspv(h, x, rule, thr, mask, y, ydt, s);
}

bool rule_ok(int rule) { return rule == SPDP_DP_NONE || rule == SPDP_DP_ABS_GT || rule == SPDP_DP_MASK; }

// copy in -> kernel -> copy out, enqueued on s.
spdp_status enqueue_host_call(spdp_matrix* h, const void* x_host, int rule, float thr, const void* mask_host,
                              void* y_host, int ydt, cudaStream_t s) {
    SPDP_CUDA_TRY(cudaMemcpyAsync(h->x_stage, x_host, h->K * sizeof(__half), cudaMemcpyHostToDevice, s));
    if (rule == SPDP_DP_MASK)
        SPDP_CUDA_TRY(cudaMemcpyAsync(h->mask_stage, mask_host, ((h->K + 31) / 32) * sizeof(uint32_t),
                                      cudaMemcpyHostToDevice, s));
    spdp_status st = launch_decode(h, h->x_stage, rule, thr, rule == SPDP_DP_MASK ? h->mask_stage : nullptr,
                                   h->y_stage, ydt, s);
    if (st != SPDP_OK) return st;
    const size_t ybytes = static_cast<size_t>(h->M) * (ydt == SPDP_Y_F32 ? sizeof(float) : sizeof(__half));
    SPDP_CUDA_TRY(cudaMemcpyAsync(y_host, h->y_stage, ybytes, cudaMemcpyDeviceToHost, s));
    return SPDP_OK;
}

// The page-locked range that holds a host address, asked of the driver in one call (looked up through the runtime: the library
// does not link libcuda).
using PointerAttributesFn = CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
PointerAttributesFn pointer_attributes_fn() {
    static PointerAttributesFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
        return reinterpret_cast<PointerAttributesFn>(f);
    }();
    return fn;
}
hostdev::PinnedRange pinned_range(const void* p) {
    const PointerAttributesFn get = pointer_attributes_fn();
    unsigned type = 0, managed = 0;
    CUdeviceptr device = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* out[] = {&type, &managed, &device, &start, &size};
    // pageable memory is no error here: every attribute comes back zero
    if (get == nullptr || get(5, what, out, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed != 0 || device == 0)
        return {0, 0, 0};
    return {static_cast<uint64_t>(start), static_cast<uint64_t>(size), static_cast<uint64_t>(device)};
}
// The address through which the kernels may use a host buffer, or null (see hostdev::direct_address).
void* direct_address(const void* p, size_t bytes, size_t align) {
    return reinterpret_cast<void*>(static_cast<uintptr_t>(hostdev::direct_address(reinterpret_cast<uintptr_t>(p), bytes, align, pinned_range(p))));
}

// The host-vector call with pinned buffers, whose device addresses the kernels use: a small kernel fetches x (and the mask) once, the
// decode kernel stores y over the bus.  No copy engine between the steps, and programmatic launch between the two kernels.
// us per call, copy engine -> this: 1024x1024 31 -> 20, 11008x4096 31 -> 27, 28672x8192 68 -> 62.  (Letting every CTA of the
// decode kernel read its part of x over the bus: 48 and 140 us on the last two, because every row tile reads x again.)
int mask_words(const spdp_matrix* h, int rule) { return rule == SPDP_DP_MASK ? static_cast<int>((h->K + 31) / 32) : 0; }
spdp_status enqueue_pinned_call(spdp_matrix* h, const spdp_matrix::HostCall& c, cudaStream_t s) {
    const int words = mask_words(h, c.rule);
    spdp_status st = launch_fetch(c.x, h->K, h->x_stage, c.mask, words, h->mask_stage, s);
    if (st != SPDP_OK) return st;
    return launch_decode(h, h->x_stage, c.rule, c.thr, words ? h->mask_stage : nullptr, c.y, c.ydt, s);
}

// Records the two kernels once (on a private stream) and keeps the instantiated graph: one launch instead of two saves
// 4 to 6 us of a call.
spdp_status record_host_graph(spdp_matrix* h, const spdp_matrix::HostCall& c) {
    if (h->capture_stream == nullptr)
        SPDP_CUDA_TRY(cudaStreamCreateWithFlags(&h->capture_stream, cudaStreamNonBlocking));
    SPDP_CUDA_TRY(cudaStreamBeginCapture(h->capture_stream, cudaStreamCaptureModeThreadLocal));
    spdp_status st = enqueue_pinned_call(h, c, h->capture_stream);
    cudaError_t e = cudaStreamEndCapture(h->capture_stream, &h->host_graph);
    size_t roots = 1, nodes = 2;
    cudaGraphNode_t all[2] = {};
    if (st == SPDP_OK && e == cudaSuccess) e = cudaGraphGetRootNodes(h->host_graph, &h->host_nodes[0], &roots);
    if (st == SPDP_OK && e == cudaSuccess) e = cudaGraphGetNodes(h->host_graph, all, &nodes);
    if (st == SPDP_OK && e == cudaSuccess) e = (roots == 1 && nodes == 2) ? cudaGraphInstantiate(&h->host_exec, h->host_graph, 0) : cudaErrorUnknown;
    if (st != SPDP_OK || e != cudaSuccess) {
        if (e != cudaSuccess) note_cuda_error(e, "recording the host-vector call");
        h->host_exec = nullptr;
        drop_host_graph(h);
        return st != SPDP_OK ? st : SPDP_ERR_CUDA;
    }
    h->host_nodes[1] = all[0] == h->host_nodes[0] ? all[1] : all[0];
    h->host_args = c;
    return SPDP_OK;
}

// Launches the recorded graph with the arguments of this call.
spdp_status replay_pinned_call(spdp_matrix* h, const spdp_matrix::HostCall& c, cudaStream_t s) {
    const int words = mask_words(h, c.rule);
    const spdp_matrix::HostCall& had = h->host_args;
    if (c.x != had.x || c.mask != had.mask || c.rule != had.rule) {
        const spdp_status st = set_fetch_node(h->host_exec, h->host_nodes[0], c.x, h->K, h->x_stage, c.mask, words, h->mask_stage);
        if (st != SPDP_OK) { drop_host_graph(h); return st; }
    }
    if (c.y != had.y || c.rule != had.rule || c.ydt != had.ydt || std::memcmp(&c.thr, &had.thr, sizeof(float)) != 0) {
        const auto set = h->q4 ? set_spmspv_q4_node : set_spmspv_node;
        const spdp_status st = set(h, h->host_exec, h->host_nodes[1], h->x_stage, c.rule, c.thr, words ? h->mask_stage : nullptr, c.y, c.ydt);
        if (st != SPDP_OK) { drop_host_graph(h); return st; }
    }
    h->host_args = c;
    SPDP_CUDA_TRY(cudaGraphLaunch(h->host_exec, s));
    return SPDP_OK;
}

}  // namespace
}  // namespace spdp

using namespace spdp;

extern "C" {

spdp_status spdp_pack_tiled_cbc_ex(const void* W_dev, int64_t M, int64_t K, int64_t ldw, int tile_m,
                                   int tile_k, int pad_elems, void* stream, spdp_handle* out) {
    if (W_dev == nullptr || out == nullptr) return SPDP_ERR_INVALID_ARG;
    if (tile_m != kTileM || tile_k != kTileK) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (M < 1 || K < 1 || ldw < K) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (pad_elems != 8 && pad_elems != 1) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (reinterpret_cast<uintptr_t>(W_dev) & 1u) return SPDP_ERR_INVALID_ARG;
    spdp_matrix* h = nullptr;
    spdp_status st = new_handle(M, K, pad_elems, &h);
    if (st != SPDP_OK) return st;
    st = alloc_arrays(h, static_cast<cudaStream_t>(stream));
    if (st == SPDP_OK) st = build_partition(h, 0, static_cast<cudaStream_t>(stream));    // emptied before the kernels, not behind them
    if (st == SPDP_OK) st = pack_device(h, static_cast<const __half*>(W_dev), ldw, static_cast<cudaStream_t>(stream));
    if (st == SPDP_OK) st = finish_handle(h, static_cast<cudaStream_t>(stream));
    if (st != SPDP_OK) { release(h); return st; }
    *out = h;
    return SPDP_OK;
}

spdp_status spdp_pack_tiled_cbc(const void* W_dev, int64_t M, int64_t K, int64_t ldw, int tile_m,
                                int tile_k, void* stream, spdp_handle* out) {
    return spdp_pack_tiled_cbc_ex(W_dev, M, K, ldw, tile_m, tile_k, 8, stream, out);
}

spdp_status spdp_pack_tiled_cbc_q4(const void* W_dev, int64_t M, int64_t K, int64_t ldw, int tile_m, int tile_k,
                                   void* stream, spdp_handle* out) {
    if (W_dev == nullptr || out == nullptr) return SPDP_ERR_INVALID_ARG;
    if (tile_m != kTileM || tile_k != kTileK) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (M < 1 || K < 1 || ldw < K) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (reinterpret_cast<uintptr_t>(W_dev) & 1u) return SPDP_ERR_INVALID_ARG;
    spdp_matrix* h = nullptr;
    spdp_status st = new_handle(M, K, 32, &h);
    if (st != SPDP_OK) return st;
    h->q4 = 1;
    st = alloc_arrays(h, static_cast<cudaStream_t>(stream));
    if (st == SPDP_OK) st = build_partition(h, 0, static_cast<cudaStream_t>(stream));    // emptied before the kernels, not behind them
    if (st == SPDP_OK) st = pack_device(h, static_cast<const __half*>(W_dev), ldw, static_cast<cudaStream_t>(stream));
    if (st == SPDP_OK) st = finish_handle(h, static_cast<cudaStream_t>(stream));
    if (st != SPDP_OK) { release(h); return st; }
    *out = h;
    return SPDP_OK;
}

spdp_status spdp_export_q4(spdp_handle h, void* tileoffset_host, void* colinfo_host, void* bitmap_host, void* codes_host,
                           void* scales_host) {
    if (!valid(h) || !h->q4) return SPDP_ERR_INVALID_ARG;
    SPDP_CUDA_TRY(cudaDeviceSynchronize());
    if (tileoffset_host)
        SPDP_CUDA_TRY(cudaMemcpy(tileoffset_host, h->tileoffset, (h->NGT + 1) * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    if (colinfo_host)
        SPDP_CUDA_TRY(cudaMemcpy(colinfo_host, h->colinfo, h->NGT * kTileK * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    if (bitmap_host)
        SPDP_CUDA_TRY(cudaMemcpy(bitmap_host, h->bitmap, h->NGT * kTileK * kWordsPerCol * sizeof(uint64_t),
                                 cudaMemcpyDeviceToHost));
    if (codes_host && h->values_len > 0)
        SPDP_CUDA_TRY(cudaMemcpy(codes_host, h->values, h->values_len / 2, cudaMemcpyDeviceToHost));
    if (scales_host)
        SPDP_CUDA_TRY(cudaMemcpy(scales_host, h->scales, h->NGT * kTileK * sizeof(__half), cudaMemcpyDeviceToHost));
    return SPDP_OK;
}

spdp_status spdp_import_tiled_cbc(int64_t M, int64_t K, int pad_elems, const void* tileoffset_host,
                                  const void* colinfo_host, const void* bitmap_host,
                                  const void* values_host, int64_t values_len, spdp_handle* out) {
    if (tileoffset_host == nullptr || colinfo_host == nullptr || bitmap_host == nullptr || out == nullptr)
        return SPDP_ERR_INVALID_ARG;
    if (values_len < 0 || (values_len > 0 && values_host == nullptr)) return SPDP_ERR_INVALID_ARG;
    if (values_len >= (int64_t(1) << 32)) return SPDP_ERR_OVERFLOW;
    spdp_matrix* h = nullptr;
    spdp_status st = new_handle(M, K, pad_elems, &h);
    if (st != SPDP_OK) return st;
    const uint32_t* to = static_cast<const uint32_t*>(tileoffset_host);
    const uint32_t* ci = static_cast<const uint32_t*>(colinfo_host);
    const uint64_t* bm = static_cast<const uint64_t*>(bitmap_host);
    // Structural validation of the arrays (Sec. 4.1): offsets are prefix sums of the padded counts.
    int64_t nnz = 0, uneven = 0;
    bool ok = (to[0] == 0) && (static_cast<int64_t>(to[h->NGT]) == values_len);
    for (int64_t g = 0; ok && g < h->NGT; ++g) {
        int64_t off = 0;
        for (int cc = 0; cc < kTileK; ++cc) {
            const int64_t slot = g * kTileK + cc;
            const int64_t n = ci[slot] & 0xFFFFu;
            int64_t pc = 0;
            for (int w = 0; w < kWordsPerCol; ++w) pc += __builtin_popcountll(bm[slot * kWordsPerCol + w]);
            if (static_cast<int64_t>(ci[slot] >> 16) != off || pc != n) { ok = false; break; }
            off += (n + pad_elems - 1) / pad_elems * pad_elems;
            nnz += n;
            const int64_t column = g % h->C * kTileK + cc, diff = n - static_cast<int64_t>(ci[slot ^ 1] & 0xFFFFu);
            if ((column | 1) < K) uneven += diff * diff;
        }
        if (ok && static_cast<int64_t>(to[g + 1]) - static_cast<int64_t>(to[g]) != off) ok = false;
    }
    if (!ok) { release(h); return SPDP_ERR_INVALID_ARG; }
    h->nnz = nnz;
    h->uneven = uneven;
    h->values_len = values_len;
    const size_t vbytes = static_cast<size_t>(values_len) * sizeof(__half);
    auto body = [&]() -> spdp_status {
        cudaStream_t s = nullptr;
        spdp_status a = alloc_arrays(h, s);
        if (a == SPDP_OK) a = build_partition(h, 0, s);
        if (a == SPDP_OK) a = handle_alloc(h->device, vbytes < 16 ? 16 : vbytes, &h->values_block);
        if (a != SPDP_OK) return a;
        h->values = static_cast<__half*>(h->values_block.p);
        SPDP_CUDA_TRY(cudaStreamSynchronize(s));
        SPDP_CUDA_TRY(cudaMemcpy(h->tileoffset, to, (h->NGT + 1) * sizeof(uint32_t), cudaMemcpyHostToDevice));
        SPDP_CUDA_TRY(cudaMemcpy(h->colinfo, ci, h->NGT * kTileK * sizeof(uint32_t), cudaMemcpyHostToDevice));
        SPDP_CUDA_TRY(cudaMemcpy(h->bitmap, bm, h->NGT * kTileK * kWordsPerCol * sizeof(uint64_t),
                                 cudaMemcpyHostToDevice));
        if (vbytes) SPDP_CUDA_TRY(cudaMemcpy(h->values, values_host, vbytes, cudaMemcpyHostToDevice));
        return finish_handle(h, s);
    };
    st = body();
    if (st != SPDP_OK) { release(h); return st; }
    *out = h;
    return SPDP_OK;
}

spdp_status spdp_spmspv(spdp_handle h, const void* x_dev, spdp_dp_rule rule, float thr,
                        const void* mask_dev, void* y_dev, spdp_ydtype ydt, void* stream) {
    if (!valid(h) || x_dev == nullptr || y_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if (!rule_ok(rule) || (ydt != SPDP_Y_F16 && ydt != SPDP_Y_F32)) return SPDP_ERR_INVALID_ARG;
    if (rule == SPDP_DP_MASK && mask_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x_dev) & 1u) ||
        (reinterpret_cast<uintptr_t>(y_dev) & (ydt == SPDP_Y_F32 ? 3u : 1u)) ||
        (reinterpret_cast<uintptr_t>(mask_dev) & 3u))
        return SPDP_ERR_INVALID_ARG;
    if (h->pad_elems != 8 && !h->q4) return SPDP_ERR_UNSUPPORTED_SHAPE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device) return SPDP_ERR_INVALID_ARG;   // wrong current device
    return launch_decode(h, static_cast<const __half*>(x_dev), rule, thr,
                         static_cast<const uint32_t*>(mask_dev), y_dev, ydt, static_cast<cudaStream_t>(stream));
}

spdp_status spdp_spmspv_batch(spdp_handle h, const void* x_dev, int64_t ldx, int batch, spdp_dp_rule rule, float thr,
                              const void* mask_dev, int64_t mask_stride, void* y_dev, int64_t ldy,
                              spdp_ydtype ydt, void* stream) {
    if (!valid(h) || x_dev == nullptr || y_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if (batch < 1 || batch > SPDP_MAX_BATCH || ldx < h->K || ldy < h->M) return SPDP_ERR_INVALID_ARG;
    if (!rule_ok(rule) || (ydt != SPDP_Y_F16 && ydt != SPDP_Y_F32)) return SPDP_ERR_INVALID_ARG;
    if (rule == SPDP_DP_MASK && (mask_dev == nullptr || mask_stride < (h->K + 31) / 32)) return SPDP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x_dev) & 1u) ||
        (reinterpret_cast<uintptr_t>(y_dev) & (ydt == SPDP_Y_F32 ? 3u : 1u)) ||
        (reinterpret_cast<uintptr_t>(mask_dev) & 3u))
        return SPDP_ERR_INVALID_ARG;
    if (h->pad_elems != 8) return SPDP_ERR_UNSUPPORTED_SHAPE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device) return SPDP_ERR_INVALID_ARG;   // wrong current device
    const __half* x = static_cast<const __half*>(x_dev);
    const uint32_t* mask = static_cast<const uint32_t*>(mask_dev);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (batch <= kBatchViaSingleCalls) {
        // The batch kernel's cost per fetched column tile does not depend on the number of tokens; below
        // three tokens one single-vector launch per token is faster (measured: 91 against 102 us for two
        // tokens on the 28672 x 8192 layer).  Same stream, same handle: the launches run in order.
        const size_t ybytes = ydt == SPDP_Y_F32 ? sizeof(float) : sizeof(__half);
        for (int b = 0; b < batch; ++b) {
            spdp_status st = launch_spmspv(h, x + b * ldx, rule, thr, mask ? mask + b * mask_stride : nullptr,
                                           static_cast<unsigned char*>(y_dev) + b * ldy * ybytes, ydt, s);
            if (st != SPDP_OK) return st;
        }
        return SPDP_OK;
    }
    return launch_spmspv_batch(h, x, ldx, batch, rule, thr, mask, mask_stride, y_dev, ldy, ydt, s);
}

spdp_status spdp_spmm(spdp_handle h, const void* X_dev, int64_t N, int64_t ldx, void* Y_dev, int64_t ldy,
                      spdp_ydtype ydt, void* stream) {
    if (!valid(h) || X_dev == nullptr || Y_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if (N < 1 || N > (int64_t(1) << 24) || ldx < h->K || ldy < h->M) return SPDP_ERR_INVALID_ARG;
    if (ydt != SPDP_Y_F16 && ydt != SPDP_Y_F32) return SPDP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(X_dev) & 15u) || (ldx & 7) ||
        (reinterpret_cast<uintptr_t>(Y_dev) & (ydt == SPDP_Y_F32 ? 3u : 1u)))
        return SPDP_ERR_INVALID_ARG;
    if (h->pad_elems != 8) return SPDP_ERR_UNSUPPORTED_SHAPE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device) return SPDP_ERR_INVALID_ARG;   // wrong current device
    return launch_spmm(h, static_cast<const __half*>(X_dev), N, ldx, Y_dev, ldy, ydt, static_cast<cudaStream_t>(stream));
}

spdp_status spdp_spmspv_noalloc(const void* tileoffset_dev, const void* colinfo_dev, const void* bitmap_dev,
                                const void* values_dev, int64_t M, int64_t K, const void* x_dev,
                                spdp_dp_rule rule, float thr, const void* mask_dev, void* y_dev,
                                spdp_ydtype ydt, void* stream) {
    if (tileoffset_dev == nullptr || colinfo_dev == nullptr || bitmap_dev == nullptr || values_dev == nullptr ||
        x_dev == nullptr || y_dev == nullptr)
        return SPDP_ERR_INVALID_ARG;
    if (M < 1 || K < 1) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if (!rule_ok(rule) || (ydt != SPDP_Y_F16 && ydt != SPDP_Y_F32)) return SPDP_ERR_INVALID_ARG;
    if (rule == SPDP_DP_MASK && mask_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(values_dev) & 15u) || (reinterpret_cast<uintptr_t>(bitmap_dev) & 7u) ||
        (reinterpret_cast<uintptr_t>(tileoffset_dev) & 3u) || (reinterpret_cast<uintptr_t>(colinfo_dev) & 15u) ||
        (reinterpret_cast<uintptr_t>(x_dev) & 1u) || (reinterpret_cast<uintptr_t>(mask_dev) & 3u) ||
        (reinterpret_cast<uintptr_t>(y_dev) & (ydt == SPDP_Y_F32 ? 3u : 1u)))
        return SPDP_ERR_INVALID_ARG;
    return launch_spmspv_noalloc(static_cast<const uint32_t*>(tileoffset_dev), static_cast<const uint32_t*>(colinfo_dev),
                                 static_cast<const uint64_t*>(bitmap_dev), static_cast<const __half*>(values_dev), M, K,
                                 static_cast<const __half*>(x_dev), rule, thr, static_cast<const uint32_t*>(mask_dev),
                                 y_dev, ydt, static_cast<cudaStream_t>(stream));
}

spdp_status spdp_spmspv_host(spdp_handle h, const void* x_host, spdp_dp_rule rule, float thr,
                             const void* mask_host, void* y_host, spdp_ydtype ydt, void* stream) {
    if (!valid(h) || x_host == nullptr || y_host == nullptr) return SPDP_ERR_INVALID_ARG;
    if (!rule_ok(rule) || (ydt != SPDP_Y_F16 && ydt != SPDP_Y_F32)) return SPDP_ERR_INVALID_ARG;
    if (rule == SPDP_DP_MASK && mask_host == nullptr) return SPDP_ERR_INVALID_ARG;
    if (h->pad_elems != 8 && !h->q4) return SPDP_ERR_UNSUPPORTED_SHAPE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device) return SPDP_ERR_INVALID_ARG;   // wrong current device
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // What is pinned is looked up on every call, and every call's arguments go into the recorded graph: nothing is assumed
    // about a buffer because an earlier one had its address.  A buffer that a kernel may not touch takes the copies.
    spdp_matrix::HostCall c = {};
    c.rule = rule;
    c.thr = thr;
    c.ydt = ydt;
    const size_t ysize = ydt == SPDP_Y_F32 ? sizeof(float) : sizeof(__half);
    c.x = static_cast<const __half*>(direct_address(x_host, h->K * sizeof(__half), sizeof(__half)));
    c.y = c.x != nullptr ? direct_address(y_host, h->M * ysize, ysize) : nullptr;
    if (rule == SPDP_DP_MASK && c.y != nullptr)
        c.mask = static_cast<const uint32_t*>(direct_address(mask_host, mask_words(h, rule) * sizeof(uint32_t), sizeof(uint32_t)));
    spdp_status st;
    if (c.y == nullptr || (rule == SPDP_DP_MASK && c.mask == nullptr)) {
        st = enqueue_host_call(h, x_host, rule, thr, mask_host, y_host, ydt, s);
    } else {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        const bool capturing = cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
        // a handle that is called again gets its graph (recording takes longer than one call saves)
        if (!capturing && h->host_exec == nullptr && ++h->host_calls == 2 && record_host_graph(h, c) != SPDP_OK) cudaGetLastError();
        st = (!capturing && h->host_exec != nullptr) ? replay_pinned_call(h, c, s) : enqueue_pinned_call(h, c, s);
    }
    if (st != SPDP_OK) return st;
    SPDP_CUDA_TRY(cudaStreamSynchronize(s));
    return SPDP_OK;
}

spdp_status spdp_swiglu_dp(const void* gate_dev, const void* up_dev, int64_t K, float thr, void* x_dev_out,
                           void* mask_dev_out, void* count_dev_out, void* stream) {
    if (gate_dev == nullptr || up_dev == nullptr || x_dev_out == nullptr || mask_dev_out == nullptr) return SPDP_ERR_INVALID_ARG;
    if (K < 1 || K > (int64_t(1) << 30)) return SPDP_ERR_UNSUPPORTED_SHAPE;
    if ((reinterpret_cast<uintptr_t>(gate_dev) & 1u) || (reinterpret_cast<uintptr_t>(up_dev) & 1u) ||
        (reinterpret_cast<uintptr_t>(x_dev_out) & 1u) || (reinterpret_cast<uintptr_t>(mask_dev_out) & 3u) ||
        (reinterpret_cast<uintptr_t>(count_dev_out) & 3u))
        return SPDP_ERR_INVALID_ARG;
    return launch_swiglu_dp(static_cast<const __half*>(gate_dev), static_cast<const __half*>(up_dev), K, thr,
                            static_cast<__half*>(x_dev_out), static_cast<uint32_t*>(mask_dev_out),
                            static_cast<int*>(count_dev_out), static_cast<cudaStream_t>(stream));
}

spdp_status spdp_row_shard(int64_t M, int world, int rank, int64_t* first_row_out, int64_t* rows_out) {
    if (M < 1 || world < 1 || rank < 0 || rank >= world || first_row_out == nullptr || rows_out == nullptr)
        return SPDP_ERR_INVALID_ARG;
    const int64_t tiles = (M + kTileM - 1) / kTileM;
    const int64_t base = tiles / world, extra = tiles % world;
    const int64_t first_tile = rank * base + (rank < extra ? rank : extra);
    const int64_t my_tiles = base + (rank < extra ? 1 : 0);
    const int64_t first = first_tile * kTileM;
    int64_t last = (first_tile + my_tiles) * kTileM;
    if (last > M) last = M;
    *first_row_out = first < M ? first : M;
    *rows_out = last > first ? last - first : 0;
    return SPDP_OK;
}

spdp_status spdp_free(spdp_handle h) {
    if (h == nullptr) {                     // no handle: give back the memory that freed handles left
        give_back_all();
        give_back_pack_totals();
        return SPDP_OK;
    }
    if (!valid(h)) return SPDP_ERR_INVALID_ARG;
    release(h);
    return SPDP_OK;
}

spdp_status spdp_get_info(spdp_handle h, spdp_info* out) {
    if (!valid(h) || out == nullptr) return SPDP_ERR_INVALID_ARG;
    spdp_info i;
    std::memset(&i, 0, sizeof(i));
    i.M = h->M; i.K = h->K; i.R = h->R; i.C = h->C; i.NGT = h->NGT;
    i.pad_elems = h->pad_elems;
    i.nnz = h->nnz;
    i.values_len = h->values_len;
    i.packed_bytes = (h->NGT + 1) * 4 + h->NGT * kTileK * 4 + h->NGT * kTileK * kWordsPerCol * 8 +
                     (h->q4 ? h->values_len / 2 + h->NGT * kTileK * 2 : h->values_len * 2);
    i.workspace_bytes = h->workspace_bytes;
    i.tileoffset_dev = h->tileoffset;
    i.colinfo_dev = h->colinfo;
    i.bitmap_dev = h->bitmap;
    i.values_dev = h->values;
    i.num_ctas = h->num_ctas;
    i.device = h->device;
    *out = i;
    return SPDP_OK;
}

spdp_status spdp_export(spdp_handle h, void* tileoffset_host, void* colinfo_host, void* bitmap_host,
                        void* values_host) {
    if (!valid(h)) return SPDP_ERR_INVALID_ARG;
    if (h->q4) return SPDP_ERR_UNSUPPORTED_SHAPE;           // 4-bit handles: spdp_export_q4
    SPDP_CUDA_TRY(cudaDeviceSynchronize());
    if (tileoffset_host)
        SPDP_CUDA_TRY(cudaMemcpy(tileoffset_host, h->tileoffset, (h->NGT + 1) * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    if (colinfo_host)
        SPDP_CUDA_TRY(cudaMemcpy(colinfo_host, h->colinfo, h->NGT * kTileK * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    if (bitmap_host)
        SPDP_CUDA_TRY(cudaMemcpy(bitmap_host, h->bitmap, h->NGT * kTileK * kWordsPerCol * sizeof(uint64_t),
                                 cudaMemcpyDeviceToHost));
    if (values_host && h->values_len > 0)
        SPDP_CUDA_TRY(cudaMemcpy(values_host, h->values, h->values_len * sizeof(__half), cudaMemcpyDeviceToHost));
    return SPDP_OK;
}

spdp_status spdp_unpack(spdp_handle h, void* W_dev_out, int64_t ldw, void* stream) {
    if (!valid(h) || W_dev_out == nullptr) return SPDP_ERR_INVALID_ARG;
    if (ldw < h->K || h->q4) return SPDP_ERR_UNSUPPORTED_SHAPE;
    return unpack_device(h, static_cast<__half*>(W_dev_out), ldw, static_cast<cudaStream_t>(stream));
}

spdp_status spdp_active_columns(spdp_handle h, const void* x_dev, spdp_dp_rule rule, float thr,
                                const void* mask_dev, void* bitmask_dev_out, void* count_dev_out,
                                void* stream) {
    if (!valid(h) || x_dev == nullptr || bitmask_dev_out == nullptr) return SPDP_ERR_INVALID_ARG;
    if (!rule_ok(rule) || (rule == SPDP_DP_MASK && mask_dev == nullptr)) return SPDP_ERR_INVALID_ARG;
    return launch_active_columns(h, static_cast<const __half*>(x_dev), rule, thr,
                                 static_cast<const uint32_t*>(mask_dev), static_cast<uint32_t*>(bitmask_dev_out),
                                 static_cast<int*>(count_dev_out), static_cast<cudaStream_t>(stream));
}

spdp_status spdp_probe_stream_read(spdp_handle h, void* stream) {
    if (!valid(h)) return SPDP_ERR_INVALID_ARG;
    return launch_probe_stream_read(h, static_cast<cudaStream_t>(stream));
}

spdp_status spdp_probe_gather(spdp_handle h, const void* x_dev, spdp_dp_rule rule, float thr, const void* mask_dev,
                              void* stream) {
    if (!valid(h) || x_dev == nullptr) return SPDP_ERR_INVALID_ARG;
    if (!rule_ok(rule) || (rule == SPDP_DP_MASK && mask_dev == nullptr)) return SPDP_ERR_INVALID_ARG;
    if (h->pad_elems != 8) return SPDP_ERR_UNSUPPORTED_SHAPE;
    return launch_probe_gather(h, static_cast<const __half*>(x_dev), rule, thr, static_cast<const uint32_t*>(mask_dev),
                               static_cast<cudaStream_t>(stream));
}

spdp_status spdp_last_device_status(spdp_handle h, int* out) {
    if (!valid(h) || out == nullptr) return SPDP_ERR_INVALID_ARG;
    int v = 0;
    SPDP_CUDA_TRY(cudaDeviceSynchronize());
    SPDP_CUDA_TRY(cudaMemcpy(&v, h->status_word, sizeof(int), cudaMemcpyDeviceToHost));
    SPDP_CUDA_TRY(cudaMemset(h->status_word, 0, sizeof(int)));
    *out = v;
    return SPDP_OK;
}

spdp_status spdp_set_num_ctas(spdp_handle h, int num_ctas) {
    if (!valid(h) || num_ctas < 0) return SPDP_ERR_INVALID_ARG;
    DeviceScope on(h->device);
    SPDP_CUDA_TRY(cudaDeviceSynchronize());
    const spdp_status st = build_partition(h, num_ctas, nullptr);
    if (st != SPDP_OK) return st;
    SPDP_CUDA_TRY(cudaStreamSynchronize(nullptr));
    return SPDP_OK;
}

const char* spdp_last_cuda_error(void) { return g_cuda_error; }

const char* spdp_status_string(spdp_status s) {
    switch (s) {
        case SPDP_OK: return "SPDP_OK";
        case SPDP_ERR_INVALID_ARG: return "SPDP_ERR_INVALID_ARG";
        case SPDP_ERR_UNSUPPORTED_SHAPE: return "SPDP_ERR_UNSUPPORTED_SHAPE";
        case SPDP_ERR_ALLOC: return "SPDP_ERR_ALLOC";
        case SPDP_ERR_CUDA: return "SPDP_ERR_CUDA";
        case SPDP_ERR_OVERFLOW: return "SPDP_ERR_OVERFLOW";
        case SPDP_ERR_TIMEOUT: return "SPDP_ERR_TIMEOUT";
    }
    return "SPDP_ERR_UNKNOWN";
}

}  // extern "C"
