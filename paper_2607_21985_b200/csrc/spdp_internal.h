// Internal declarations shared by the translation units of libspdp (not part of the ABI).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "spdp.h"

namespace spdp {

constexpr int kTileM = 256;        // rows per column tile (Sec. 4.1)
constexpr int kTileK = 16;         // column tiles per GTile (Sec. 4.2.3)
constexpr int kWordsPerCol = 4;    // 64-bit bitmap words per column tile (Sec. 4.1)
constexpr int kPackTotals = 3;     // sums over a layer that packing hands to the host
constexpr uint64_t kMagic = 0x5350445042323030ull;   // "SPDPB200"

// A piece of device memory that a handle owns (memory.cu).
struct Slab;
struct DeviceBlock {
    void* p;
    size_t bytes;
    Slab* slab;     // the slab it is part of, or null: an allocation of its own
};

}  // namespace spdp

// Host-side state behind an spdp_handle.
struct spdp_matrix {
    uint64_t magic;
    int device;
    int sm_count;
    int64_t M, K, R, C, NGT;
    int pad_elems;
    int64_t nnz;
    int64_t uneven;         // see plan::batch_loads_one_by_one
    int64_t values_len;

    // Tiled-CBC arrays (device).  `arrays` is the allocation that holds every array whose size follows from the shape:
    // tileoffset, colinfo, bitmap, scales, the status word and the staging buffers; values has its own.
    spdp::DeviceBlock arrays, values_block;
    uint32_t* tileoffset;   // [NGT+1]
    uint32_t* colinfo;      // [NGT*16]
    uint64_t* bitmap;       // [NGT*16*4]
    __half* values;         // [values_len] (at least 16 bytes are allocated); 4-bit variant: values_len codes, two per byte
    int q4;                 // 1: the 4-bit variant (codes + scales), pad_elems = 32
    __half* scales;         // 4-bit variant: [NGT*16] one scale per column tile; else null

    // Work partition of one spmspv launch: the kernel cuts the NGT GTiles into num_ctas equal
    // contiguous ranges, one per CTA.
    int num_ctas;           // P
    float* workspace;       // device [P*256] split-K tree nodes, one row per CTA (all zero between calls)
    float* workspace_batch; // device [P*8*256] tree nodes of the small-batch call (all zero between calls)
    spdp::DeviceBlock workspace_block;  // both
    spdp::DeviceBlock packing;          // lengths of the GTiles while packing
    int* status_word;       // device [2]: the status word, and a sink word the benchmark probes may write
    unsigned long long* pack_totals;    // device [kPackTotals]: length of Values, nonzeros and unevenness, counted while packing
    int64_t workspace_bytes;

    // Staging for the host-vector entry point
    __half* x_stage;        // device [K]
    uint32_t* mask_stage;   // device [ceil(K/32)]
    void* y_stage;          // device [M] fp32-sized

    // spdp_spmspv_host with pinned buffers: its two kernels, recorded once as a graph whose nodes get each call's arguments.
    struct HostCall {
        const __half* x;                // device addresses of the pinned buffers
        const uint32_t* mask;
        void* y;
        int rule, ydt;
        float thr;
    };
    int64_t host_calls;             // pinned calls so far
    cudaGraph_t host_graph;         // null: not recorded yet
    cudaGraphExec_t host_exec;
    cudaGraphNode_t host_nodes[2];  // fetch, decode
    HostCall host_args;             // the arguments that host_exec holds
    cudaStream_t capture_stream;    // private stream used only to record that graph

    // Benchmark probe (spdp_probe_gather): the list of active column tiles it reads, built on first use.
    struct ProbeKey {
        const void* x;
        const void* mask;
        int rule;
        float thr;
    };
    void* probe_items;              // device uint2[R*K], null until the probe is first called
    void* probe_count;              // device uint64[1]
    ProbeKey probe_key;
};

namespace spdp {

// Records the message of a failed CUDA call for spdp_last_cuda_error().
void note_cuda_error(cudaError_t e, const char* what);

#define SPDP_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t e__ = (expr);                             \
        if (e__ != cudaSuccess) {                             \
            ::spdp::note_cuda_error(e__, #expr);              \
            return (e__ == cudaErrorMemoryAllocation) ? SPDP_ERR_ALLOC : SPDP_ERR_CUDA; \
        }                                                     \
    } while (0)

inline bool valid(const spdp_matrix* h) { return h != nullptr && h->magic == kMagic; }

// memory.cu
// Memory that a handle owns, usable on any stream, on the current device (`device`).
spdp_status handle_alloc(int device, size_t bytes, DeviceBlock* out);
// Takes it back for the next handle and empties `block`.  `idle`: nothing on the device uses it any more; else it is not used again.
void handle_give(int device, DeviceBlock& block, bool idle);
// A handle came (+1) or went (-1).
void count_handle(int device, int by);
// Everything that is kept and not in use goes back to the driver, on every device.
void give_back_all();
// Stream-ordered scratch memory for one call (given back with cudaFreeAsync on the same stream).
spdp_status scratch_alloc(int device, size_t bytes, cudaStream_t s, void** out);

// pack.cu
spdp_status pack_device(spdp_matrix* h, const __half* W, int64_t ldw, cudaStream_t s);     // either variant
spdp_status unpack_device(const spdp_matrix* h, __half* W, int64_t ldw, cudaStream_t s);
void give_back_pack_totals();                  // page-locked words of the pack calls, if none is on its way

// spmspv.cu
int default_ctas_per_sm();   // CTAs of the spMspV kernel that share one SM
spdp_status configure_spmspv_kernel();   // per-device kernel attributes; idempotent
spdp_status launch_spmspv(const spdp_matrix* h, const __half* x, int rule, float thr,
                          const uint32_t* mask, void* y, int ydt, cudaStream_t s);
spdp_status launch_spmspv_noalloc(const uint32_t* tileoffset, const uint32_t* colinfo, const uint64_t* bitmap,
                                  const __half* values, int64_t M, int64_t K, const __half* x, int rule,
                                  float thr, const uint32_t* mask, void* y, int ydt, cudaStream_t s);
// spmspv_batch.cu
int64_t batch_workspace_bytes(int num_ctas);
spdp_status configure_spmspv_batch_kernel();   // per-device kernel attributes; idempotent
spdp_status launch_spmspv_batch(const spdp_matrix* h, const __half* x, int64_t ldx, int batch, int rule, float thr,
                                const uint32_t* mask, int64_t mask_stride, void* y, int64_t ldy, int ydt,
                                cudaStream_t s);

// spmspv_q4.cu: the 4-bit variant
spdp_status configure_spmspv_q4_kernel();      // per-device kernel attributes; idempotent
spdp_status launch_spmspv_q4(const spdp_matrix* h, const __half* x, int rule, float thr, const uint32_t* mask, void* y,
                             int ydt, cudaStream_t s);

// The kernel of a node of an instantiated graph gets the arguments of another call on the same handle.
spdp_status set_spmspv_node(const spdp_matrix* h, cudaGraphExec_t exec, cudaGraphNode_t node, const __half* x, int rule, float thr,
                            const uint32_t* mask, void* y, int ydt);
spdp_status set_spmspv_q4_node(const spdp_matrix* h, cudaGraphExec_t exec, cudaGraphNode_t node, const __half* x, int rule, float thr,
                               const uint32_t* mask, void* y, int ydt);
spdp_status set_fetch_node(cudaGraphExec_t exec, cudaGraphNode_t node, const __half* x, int64_t K, __half* x_out, const uint32_t* mask,
                           int mask_words, uint32_t* mask_out);

// producer.cu
// x (and mask_words words of mask) from pinned host memory, by their device addresses, into device buffers.
spdp_status launch_fetch(const __half* x, int64_t K, __half* x_out, const uint32_t* mask, int mask_words, uint32_t* mask_out, cudaStream_t s);
spdp_status launch_swiglu_dp(const __half* gate, const __half* up, int64_t K, float thr, __half* x_out, uint32_t* mask_out,
                             int* count, cudaStream_t s);

// spmm.cu
spdp_status configure_spmm_kernel();            // per-device kernel attributes; idempotent
spdp_status launch_spmm(const spdp_matrix* h, const __half* X, int64_t N, int64_t ldx, void* Y, int64_t ldy, int ydt,
                        cudaStream_t s);

// probes.cu (context measurements for the benchmark)
spdp_status launch_probe_stream_read(const spdp_matrix* h, cudaStream_t s);
spdp_status launch_probe_gather(spdp_matrix* h, const __half* x, int rule, float thr, const uint32_t* mask,
                                cudaStream_t s);

spdp_status launch_active_columns(const spdp_matrix* h, const __half* x, int rule, float thr,
                                  const uint32_t* mask, uint32_t* bits, int* count, cudaStream_t s);

}  // namespace spdp
