// Device memory of the handles, and scratch memory of single calls.
//
// What a handle owns lies in cudaMalloc allocations, so that the arrays behind spdp_get_info can be reached by a peer and
// exported to another process like any other.  cudaMalloc and cudaFree are slow (about 0.3 ms a call; 3 ms per packed and freed
// layer with one for every array), so
//   up to kSmall bytes  are cut from slabs of kSlabBytes: a handle's metadata and workspace, and all of a small layer.  A hundred
//                       1024x1024 layers that are all kept are packed in 140 to 150 us each, 940 to 1440 with an allocation
//                       for every piece; four of 11008x4096 in 480, 1060;
//   more than that      is an allocation of its own, a whole number of the driver's 2 MB pages.  (Packed again in the memory of
//                       a freed handle, 1024x1024 takes 52 us, 11008x4096 119.)
// What freed handles leave (empty slabs and large blocks) is kept for the next ones up to kKeep bytes and kKeptBlocks large
// blocks per device.  An allocation that finds no memory gives it back first, and so does spdp_free(NULL).  Memory is taken
// back only when nothing on the device uses it any more, so the next owner may be any thread and any stream.
//
// The partial sums of one spdp_spmm call come from a stream-ordered pool (calls on several streams or threads get memory of
// their own), apart from the device's default pool, which gives its memory back at every synchronisation: 0.45 ms per call.
// It keeps up to kScratchKeep bytes over a synchronisation, all given back when the device's last handle goes and by
// spdp_free(NULL).
#include <algorithm>
#include <mutex>
#include <new>

#include "spdp_internal.h"

namespace spdp {

constexpr int kMaxDevices = 64;
constexpr size_t kUnit = size_t(16) << 10;              // what a slab is cut into
constexpr int kUnits = 2048;
constexpr size_t kSlabBytes = kUnit * kUnits;           // 32 MB
constexpr size_t kSmall = kSlabBytes / 4;
constexpr size_t kPage = size_t(2) << 20;
constexpr size_t kKeep = size_t(512) << 20;
constexpr int kKeptBlocks = 64;
constexpr uint64_t kScratchKeep = uint64_t(96) << 20;

struct Slab {
    unsigned char* base;
    int free_units;
    bool used[kUnits];
    Slab* next;
};

namespace {

struct DeviceMemory {
    Slab* slabs;
    DeviceBlock kept[kKeptBlocks];      // large blocks without an owner, oldest first
    int num_kept;
    size_t bytes_kept;                  // theirs and the empty slabs'
    cudaMemPool_t scratch_pool;
    int64_t handles;
};
std::mutex g_mu;
DeviceMemory g_memory[kMaxDevices];

// The functions below with a DeviceMemory are called with the lock held.

// `units` consecutive free units of a slab, or null.  Only slabs with that many free units are searched.
bool take_units(DeviceMemory& m, int units, DeviceBlock* out) {
    for (Slab* s = m.slabs; s != nullptr; s = s->next) {
        if (s->free_units < units) continue;
        for (int i = 0, run = 0; i < kUnits; ++i) {
            run = s->used[i] ? 0 : run + 1;
            if (run < units) continue;
            const int first = i + 1 - units;
            if (s->free_units == kUnits) m.bytes_kept -= kSlabBytes;
            s->free_units -= units;
            std::fill(s->used + first, s->used + first + units, true);
            *out = {s->base + first * kUnit, units * kUnit, s};
            return true;
        }
    }
    return false;
}

DeviceBlock take_kept(DeviceMemory& m, int i) {
    const DeviceBlock b = m.kept[i];
    for (int k = i + 1; k < m.num_kept; ++k) m.kept[k - 1] = m.kept[k];
    --m.num_kept;
    m.bytes_kept -= b.bytes;
    return b;
}

// Something that is kept and may go back to the driver: the oldest large block, else an empty slab; null if there is none.
void* take_any(DeviceMemory& m) {
    if (m.num_kept > 0) return take_kept(m, 0).p;
    for (Slab** at = &m.slabs; *at != nullptr; at = &(*at)->next) {
        Slab* s = *at;
        if (s->free_units < kUnits) continue;
        void* p = s->base;
        *at = s->next;
        m.bytes_kept -= kSlabBytes;
        delete s;
        return p;
    }
    return nullptr;
}

// Gives what is kept back to the driver until at most `most` bytes of it are left.  Answers whether there was any.
bool give_back(int device, size_t most) {
    bool any = false;
    for (;;) {
        void* p = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_mu);
            DeviceMemory& m = g_memory[device];
            if (m.bytes_kept > most || m.num_kept > kKeptBlocks - 1) p = take_any(m);
        }
        if (p == nullptr) return any;
        cudaFree(p);
        any = true;
    }
}

// cudaMalloc, again without what is kept where there is no memory.
spdp_status driver_alloc(int device, size_t bytes, void** p) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation && give_back(device, 0)) {
        cudaGetLastError();
        e = cudaMalloc(p, bytes);
    }
    SPDP_CUDA_TRY(e);
    return SPDP_OK;
}

void trim_scratch(int device) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_memory[device].scratch_pool != nullptr) cudaMemPoolTrimTo(g_memory[device].scratch_pool, 0);
}

}  // namespace

spdp_status handle_alloc(int device, size_t bytes, DeviceBlock* out) {
    if (device < 0 || device >= kMaxDevices) return SPDP_ERR_UNSUPPORTED_SHAPE;
    DeviceMemory& m = g_memory[device];
    void* p = nullptr;
    if (bytes <= kSmall) {
        const int units = static_cast<int>((std::max<size_t>(bytes, 1) + kUnit - 1) / kUnit);
        {
            std::lock_guard<std::mutex> lock(g_mu);
            if (take_units(m, units, out)) return SPDP_OK;
        }
        Slab* slab = new (std::nothrow) Slab();
        if (slab == nullptr) return SPDP_ERR_ALLOC;
        const spdp_status st = driver_alloc(device, kSlabBytes, &p);
        if (st == SPDP_OK) {
            slab->base = static_cast<unsigned char*>(p);
            slab->free_units = kUnits;
            std::lock_guard<std::mutex> lock(g_mu);
            slab->next = m.slabs;                       // in front: the newest has room
            m.slabs = slab;
            m.bytes_kept += kSlabBytes;
            take_units(m, units, out);
            return SPDP_OK;
        }
        delete slab;
        if (st != SPDP_ERR_ALLOC) return st;            // no room for a slab: a piece of its own
    }
    bytes = bytes <= kSmall ? (bytes + 511) / 512 * 512 : (bytes + kPage - 1) / kPage * kPage;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        int best = -1;                                  // a kept block serves where less than an eighth of it would lie idle
        for (int i = 0; i < m.num_kept; ++i)
            if (m.kept[i].bytes >= bytes && m.kept[i].bytes - bytes <= bytes / 8 && (best < 0 || m.kept[i].bytes < m.kept[best].bytes)) best = i;
        if (best >= 0) {
            *out = take_kept(m, best);
            return SPDP_OK;
        }
    }
    const spdp_status st = driver_alloc(device, bytes, &p);
    if (st == SPDP_OK) *out = {p, bytes, nullptr};
    return st;
}

void handle_give(int device, DeviceBlock& block, bool idle) {
    const DeviceBlock b = block;
    block = {};
    if (b.p == nullptr) return;
    if (b.slab == nullptr && (!idle || b.bytes > kKeep)) {
        cudaFree(b.p);                                  // which waits for the device
        return;
    }
    if (!idle) return;                                  // part of a slab that may be in use: never again
    if (b.slab == nullptr) give_back(device, kKeep - b.bytes);
    {
        std::lock_guard<std::mutex> lock(g_mu);
        DeviceMemory& m = g_memory[device];
        if (b.slab == nullptr) {
            if (m.num_kept < kKeptBlocks) {
                m.kept[m.num_kept++] = b;
                m.bytes_kept += b.bytes;
                return;
            }
        } else {
            const size_t first = (static_cast<unsigned char*>(b.p) - b.slab->base) / kUnit, units = b.bytes / kUnit;
            std::fill(b.slab->used + first, b.slab->used + first + units, false);
            b.slab->free_units += static_cast<int>(units);
            if (b.slab->free_units < kUnits) return;
            m.bytes_kept += kSlabBytes;
        }
    }
    if (b.slab == nullptr) cudaFree(b.p);               // another thread was faster with the last place
    else give_back(device, kKeep);
}

void count_handle(int device, int by) {
    if (device < 0 || device >= kMaxDevices) return;
    bool last;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        last = (g_memory[device].handles += by) == 0;
    }
    if (last) trim_scratch(device);
}

void give_back_all() {
    for (int d = 0; d < kMaxDevices; ++d) {
        while (give_back(d, 0)) {}
        trim_scratch(d);
    }
}

spdp_status scratch_alloc(int device, size_t bytes, cudaStream_t s, void** out) {
    if (device < 0 || device >= kMaxDevices) return SPDP_ERR_UNSUPPORTED_SHAPE;
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (g_memory[device].scratch_pool == nullptr) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = device;
            cudaMemPool_t made = nullptr;
            SPDP_CUDA_TRY(cudaMemPoolCreate(&made, &props));
            uint64_t keep = kScratchKeep;
            const cudaError_t e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) {
                cudaMemPoolDestroy(made);
                SPDP_CUDA_TRY(e);
            }
            g_memory[device].scratch_pool = made;
        }
        pool = g_memory[device].scratch_pool;
    }
    SPDP_CUDA_TRY(cudaMallocFromPoolAsync(out, bytes, pool, s));
    return SPDP_OK;
}

}  // namespace spdp
